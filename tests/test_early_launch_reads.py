"""Kernels that start while the kernel before them on the stream still runs (they call
after_previous() first) read what that kernel writes by plain loads.  __ldg and const __restrict__
parameters take the read-only path, defined only for memory that nobody writes during the kernel's life,
and __restrict__ lets the compiler move a load over the wait; both stay with the tables below, which
are complete (uploaded, stream synchronised) before any chain of launches begins.  A stale read has no
reliable symptom, so the source is what is checked."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2203_07820_gb300", "csrc")
TABLES = {"items", "work",                                                  # launch descriptors
          "group", "prow", "pnode", "pval", "hcoup", "snode", "srow", "sproj", "sval"}   # projectors


def _block(src, at, opening, closing):
    depth = 0
    for i in range(at, len(src)):
        depth += (src[i] == opening) - (src[i] == closing)
        if depth == 0:
            return src[at:i + 1], i + 1
    raise AssertionError("unbalanced source")


def early_kernels():
    """(file, name, parameters, body) of every kernel that waits in after_previous()"""
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh", ".h")):
            continue
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        for m in re.finditer(r"__global__\s+void\b", src):
            at = m.end()
            # attributes with parentheses, then the kernel's name and parameter list
            while True:
                k = re.compile(r"\s*(__launch_bounds__|__cluster_dims__)\s*(?=\()").match(src, at)
                if not k:
                    break
                at = _block(src, k.end(), "(", ")")[1]
            k = re.compile(r"\s*(\w+)\s*(?=\()").match(src, at)
            params, at = _block(src, k.end(), "(", ")")
            brace = re.compile(r"\s*(?=\{)").match(src, at)
            if not brace:
                continue
            body = _block(src, brace.end(), "{", "}")[0]
            if "after_previous()" in body:
                yield name, k.group(1), params, body


def test_fresh_data_is_read_by_plain_loads():
    found = list(early_kernels())
    assert {"k_sf_cell", "k_sf_faces", "k_nl_coef", "k_nl_add", "k_multidot_partial", "k_multidot_final",
            "k_lz_three_term", "k_lz_reorth", "k_lz_scale"} <= {k for _, k, _, _ in found}
    for name, kernel, params, body in found:
        restricted = set(re.findall(r"__restrict__\s+(\w+)", params))
        assert restricted <= TABLES, (name, kernel, restricted - TABLES)
        assert "__ldg" not in body, (name, kernel)


def test_helpers_of_those_kernels_do_not_use_the_read_only_path():
    # device functions shared by them
    for name in ("nonlocal.cuh", "sumfac.h"):
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        assert "__ldg" not in src, name
        for params in re.findall(r"__device__ __forceinline__ void sums\((.*?)\)\s*\{", src, flags=re.S):
            assert "__restrict__" not in params


def test_every_early_launch_is_of_such_a_kernel():
    waiting = {k for _, k, _, _ in early_kernels()}
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")):
            src = open(os.path.join(CSRC, name)).read()
            for kernel in re.findall(r"launch_after\(\(?(k_\w+)", src):
                assert kernel in waiting, (name, kernel)
