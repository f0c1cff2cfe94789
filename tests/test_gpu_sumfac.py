"""The tensor-product form of the local operator against the FP64 oracle's dense cell
matrices: every degree, both quadrature rules, anisotropic boxes with even, odd and
two-cell axes, column counts around the kernels' tiles (several cells per CTA below 8 columns,
ragged tiles, more than one face-buffer chunk); meshes whose quadrature rule has no such form
keep the dense products.  Tolerance: both sides are FP64 sums of the same products in another
order, so the parity tests' 1e-12 of the largest entry."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.fixture(scope="module")
def dg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2203_07820_gb300 as dg
    return dg


def _system(dg, L, n, p, vquad=0, nq1d=0, seed=1):
    s = synth.Stream(seed)
    cent = np.array([[Ld * s.uniform() for Ld in L] for _ in range(3)])
    om = oracle.PeriodicMesh(L, n, p, **({"nq1d": nq1d} if nq1d else {}))
    oh = oracle.Hamiltonian(om, vquad=vquad)
    mesh = dg.dftfe_mesh_create(L, n, p, vquad=vquad, nq1d=nq1d)
    ham = dg.dftfe_ham_create(mesh)
    v = synth.gaussian_wells(om.quad_xyz(vquad).reshape(-1, 3), cent, 2.0, 1.0, np.array(L))
    oh.set_potential(v)
    dg.dftfe_ham_set_potential(ham, torch.from_numpy(np.ascontiguousarray(v).reshape(-1)).cuda())
    return om, oh, mesh, ham


def _destroy(dg, mesh, ham):
    dg.dftfe_ham_destroy(ham)
    dg.dftfe_mesh_destroy(mesh)


@pytest.mark.parametrize("vquad", [0, 1])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6, 7, 8])
def test_apply_and_cell_matrices(dg, p, vquad):
    n = (3, 2, 4) if p <= 5 else (2, 3, 2)
    om, oh, mesh, ham = _system(dg, (5.0, 4.0, 6.5), n, p, vquad)
    try:
        out = torch.empty((om.ncells, om.nodes_per_cell, om.nodes_per_cell), dtype=torch.float64, device="cuda")
        dg.dftfe_ham_export(ham, c0=0, cell_mats=out)
        ref = np.asarray(oh.cell_matrices())
        assert np.abs(out.cpu().numpy() - ref).max() <= 1e-13 * np.abs(ref).max()
        for ncol in (1, 2, 3, 7, 9, 33, 130):
            X0 = synth.random_block(50 + ncol, om.ndofs, ncol)
            X = torch.from_numpy(X0).cuda()
            Y = torch.full_like(X, float("nan"))
            dg.dftfe_ham_apply(ham, X, Y)
            ref = oh.apply(X0)
            err = np.abs(Y.cpu().numpy() - ref).max()
            assert err <= TOL * np.abs(ref).max(), (ncol, err)
    finally:
        _destroy(dg, mesh, ham)


@pytest.mark.parametrize("p,nq1d", [(3, 6), (4, 3), (6, 9)])
def test_other_quadrature_rules_keep_the_dense_products(dg, p, nq1d):
    om, oh, mesh, ham = _system(dg, (5.0, 4.0, 6.5), (3, 2, 2), p, 0, nq1d)
    try:
        for ncol in (1, 4, 37):
            X0 = synth.random_block(60 + ncol, om.ndofs, ncol)
            X = torch.from_numpy(X0).cuda()
            Y = torch.full_like(X, float("nan"))
            dg.dftfe_ham_apply(ham, X, Y)
            ref = oh.apply(X0)
            assert np.abs(Y.cpu().numpy() - ref).max() <= TOL * np.abs(ref).max(), ncol
    finally:
        _destroy(dg, mesh, ham)


def test_batch_of_both_forms_is_bit_identical_to_single_passes(dg):
    """Tensor-product systems of two degrees, a dense one (other quadrature rule) and narrow
    blocks in one FP64 batch."""
    specs = [((5.0, 4.0, 6.5), (3, 2, 4), 4, 0, 0, 12, 5), ((4.0, 4.0, 4.0), (2, 2, 2), 6, 1, 0, 9, 9),
             ((5.0, 4.0, 5.0), (2, 3, 2), 3, 0, 5, 10, 4), ((4.0, 5.0, 4.0), (2, 2, 3), 4, 0, 0, 6, 2)]
    made = [_system(dg, *s[:5], seed=i) for i, s in enumerate(specs)]
    batch = dg.dftfe_batch_create([m[3] for m in made])
    try:
        X1, X2, bd1, bd2, ev, rs, deg = [], [], [], [], [], [], []
        for i, ((om, oh, mesh, ham), s) in enumerate(zip(made, specs)):
            N = s[5]
            x = torch.from_numpy(synth.random_block(80 + i, om.ndofs, N)).cuda()
            X1.append(x)
            X2.append(x.clone())
            b = dg.dftfe_spectrum_bounds(ham, 12, 3, N)
            bd1.append(b)
            bd2.append(dg.make_bounds(b.a, b.b, b.a0))
            ev.append(torch.empty(N, dtype=torch.float64, device="cuda"))
            rs.append(torch.empty_like(ev[-1]))
            deg.append(5 + i)
        blocks = [s[6] for s in specs]
        for _ in range(2):
            dg.dftfe_batch_chfsi_pass(batch, X1, blocks, deg, bd1, ev, rs)
            for i, m in enumerate(made):
                dg.dftfe_chfsi_pass(m[3], X2[i], blocks[i], deg[i], bd2[i], ev[i], rs[i])
        for a, b in zip(X1, X2):
            assert torch.equal(a, b)
    finally:
        dg.dftfe_batch_destroy(batch)
        for m in made:
            _destroy(dg, m[2], m[3])


def _projectors(M, order, seed=3):
    """Projectors of atoms with 1, 2, 3, 4, 5 and 9 channels on one support each: empty, one node,
    below and above the entries a CTA stages at a time, most of the mesh.  `order` "atom" keeps an
    atom's channels together, "channel" interleaves the atoms."""
    rng = np.random.default_rng(seed)
    atoms = [(1, 37), (2, 0), (3, 1), (4, 4600), (5, 530), (9, 260)]
    rows = []
    for a, (nch, n) in enumerate(atoms):
        nodes = np.sort(rng.choice(M, n, replace=False))
        rows += [(j, a, nodes, rng.standard_normal(n), 0.5 + rng.random(), rng.standard_normal((n, 3)))
                 for j in range(nch)]
    if order == "channel":
        rows.sort(key=lambda r: (r[0], r[1]))
    rowptr = np.cumsum([0] + [len(r[2]) for r in rows]).astype(np.int64)
    return (np.array([r[4] for r in rows]), rowptr, np.concatenate([r[2] for r in rows]).astype(np.int64),
            np.concatenate([r[3] for r in rows]), np.concatenate([r[5] for r in rows]))


@pytest.mark.parametrize("ncol", [1, 2, 5, 16, 33, 130])
def test_projectors_on_common_supports(dg, ncol):
    """The nonlocal term of grouped projectors against the dense products, in both precisions, and
    against the same projectors in an order that leaves them apart, real and complex.  Bounds: a
    coefficient's sum has chains of at most 40 + 16 + 16 + 8 additions, a node's at most 24 terms
    and the update, so 112 u |C| h |C|^T |X| + 2 u |Y| (u the unit roundoff of the form)."""
    om, oh, mesh, ham = _system(dg, (5.0, 4.0, 4.0), (5, 4, 4), 4)
    try:
        M = om.ndofs
        X0 = synth.random_block(70 + ncol, M, ncol)
        X = torch.from_numpy(X0).cuda()
        Z = torch.complex(X, X.flip(0)).contiguous()
        apply = {}
        for prec in (dg.DFTFE_FP64, dg.DFTFE_MIXED_TF32X3):
            apply[prec] = torch.empty_like(X)
            dg.dftfe_ham_apply(ham, X, apply[prec], prec)
        for order in ("atom", "channel"):
            hc, rp, nd, chi, disp = _projectors(M, order)
            C = np.zeros((M, len(hc)))
            for a in range(len(hc)):
                s = slice(rp[a], rp[a + 1])
                C[nd[s], a] = np.sqrt(om.mass[nd[s]]) * chi[s]
            bound = np.abs(C) @ (hc[:, None] * (np.abs(C).T @ np.abs(X0)))
            ref = C @ (hc[:, None] * (C.T @ X0))
            dg.dftfe_ham_set_nonlocal(ham, hc, rp, nd, chi)
            for prec, u in ((dg.DFTFE_FP64, 2.0 ** -53), (dg.DFTFE_MIXED_TF32X3, 2.0 ** -24)):
                Y = torch.full_like(X, float("nan"))
                dg.dftfe_ham_apply(ham, X, Y, prec)
                y = Y.cpu().numpy()
                err = np.abs(y - apply[prec].cpu().numpy() - ref)
                assert np.all(err <= 112 * u * bound + 2 * u * np.abs(y)), (order, prec)
        dg.dftfe_ham_set_kpoint(ham, (0.2, -0.1, 0.15), disp)
        zbound = np.abs(C) @ (hc[:, None] * (np.abs(C).T @ np.abs(Z.cpu().numpy())))
        for prec, u in ((dg.DFTFE_FP64, 2.0 ** -53), (dg.DFTFE_MIXED_TF32X3, 2.0 ** -24)):
            got = []
            for order in ("atom", "channel"):
                hc, rp, nd, chi, disp = _projectors(M, order)
                dg.dftfe_ham_set_nonlocal(ham, hc, rp, nd, chi)
                dg.dftfe_ham_set_kpoint(ham, (0.2, -0.1, 0.15), disp)
                Y = torch.full_like(Z, float("nan"))
                dg.dftfe_ham_apply_z(ham, Z, Y, prec)
                got.append(Y.cpu().numpy())
            # complex products: twice the terms of the real sums on each side
            assert np.all(np.abs(got[0] - got[1]) <= 448 * u * zbound + 4 * u * np.abs(got[0])), prec
    finally:
        _destroy(dg, mesh, ham)


@pytest.mark.parametrize("vquad", [0, 1])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
def test_pairs_keep_non_finite_entries(dg, bad, vquad):
    """A NaN or an infinity in the block or in the potential reaches every entry of the FP64-accurate
    products that it makes non-finite in FP64; the other columns, and without column scaling the
    other rows, stay right."""
    om, oh, mesh, ham = _system(dg, (5.0, 4.0, 6.5), (3, 2, 4), 4, vquad)
    try:
        X = torch.from_numpy(synth.random_block(7, om.ndofs, 5)).cuda()
        row = om.ndofs // 3
        Xbad = X.clone()
        Xbad[row, 2] = bad
        _, ncell, _, nq = dg.dftfe_mesh_info(mesh)
        v = torch.from_numpy(synth.random_block(9, ncell * nq, 1)).cuda().reshape(-1)
        vbad = v.clone()
        vbad[v.numel() // 2] = bad
        for pot, x in ((v, Xbad), (vbad, X)):
            dg.dftfe_ham_set_potential(ham, pot)
            ref = torch.empty_like(X)
            dg.dftfe_ham_apply(ham, x, ref)
            lost = ~torch.isfinite(ref)
            assert lost.any()
            for prec in (dg.DFTFE_FP64_FLOAT_PAIRS, dg.DFTFE_FP64_SLICES):
                Y = torch.zeros_like(X)
                dg.dftfe_ham_apply(ham, x, Y, prec)
                assert not torch.isfinite(Y[lost]).any(), prec
                keep = ~lost
                if prec == dg.DFTFE_FP64_SLICES and x is Xbad:
                    keep = keep & (torch.arange(5, device="cuda") != 2)
                assert (Y - ref)[keep].abs().max().item() <= 1e-12 * ref[keep].abs().max().item(), prec
    finally:
        _destroy(dg, mesh, ham)


def test_pairs_beyond_the_range_of_fp32(dg):
    """Entries above 2^128: the scaled form keeps them, the unscaled one has no representation for them and
    says so."""
    om, oh, mesh, ham = _system(dg, (5.0, 4.0, 6.5), (3, 2, 4), 4)
    try:
        X = torch.from_numpy(synth.random_block(7, om.ndofs, 5)).cuda()
        for scale in (2.0 ** 140, 2.0 ** 900):
            x = X * scale
            ref, Y = torch.empty_like(X), torch.empty_like(X)
            dg.dftfe_ham_apply(ham, x, ref)
            dg.dftfe_ham_apply(ham, x, Y, dg.DFTFE_FP64_SLICES)
            assert (Y - ref).abs().max().item() <= TOL * ref.abs().max().item()
            dg.dftfe_ham_apply(ham, x, Y, dg.DFTFE_FP64_FLOAT_PAIRS)
            assert not torch.isfinite(Y).any()
    finally:
        _destroy(dg, mesh, ham)


def test_projectors_with_empty_supports_add_nothing(dg):
    om, oh, mesh, ham = _system(dg, (5.0, 4.0, 4.0), (3, 2, 2), 4)
    try:
        X = torch.from_numpy(synth.random_block(5, om.ndofs, 6)).cuda()
        bounds = dg.dftfe_spectrum_bounds(ham, 10, 1, 6)

        def results():
            out = []
            for prec in (dg.DFTFE_FP64, dg.DFTFE_MIXED_TF32X3, dg.DFTFE_FP64_FLOAT_PAIRS):
                Y = torch.full_like(X, float("nan"))
                dg.dftfe_ham_apply(ham, X, Y, prec)
                out.append(Y)
            Y = X.clone()
            dg.dftfe_chebyshev_filter(ham, Y, 5, bounds, dg.DFTFE_MIXED_TF32X3)
            return out + [Y]

        without = results()
        dg.dftfe_ham_set_nonlocal(ham, np.array([0.5, 0.7]), np.zeros(3, dtype=np.int64), np.zeros(0, dtype=np.int64),
                                  np.zeros(0))
        for a, b in zip(without, results()):
            assert torch.equal(a, b)
    finally:
        _destroy(dg, mesh, ham)
