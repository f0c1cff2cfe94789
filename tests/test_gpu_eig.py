"""The dense eigensolver behind Rayleigh-Ritz (tridiagonalisation, divide and conquer, back
transformation) at the sizes where its code paths change: single rows, the edges of the
merges done in one CTA (16 rows) and of the register tiles (multiples of 32, groups of four
reflectors), one CTA against several, and sizes beyond the shared-memory rows (Jacobi).
Spectra: well separated (random block) and heavily degenerate (a rotated block of exact
eigenvectors of the empty cubic box, whose levels repeat up to 24 times).  Tolerances: the
solver is backward stable, so values and residuals are within a small multiple of eps |H|
(N-independent 1e-12 |H|), columns orthonormal to 1e-12 (the parity tests' bounds)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2203_07820_gb300 as dg
    return dg


@pytest.fixture(scope="module")
def box(dg):
    """An empty 5 bohr cube, 6^3 cells, p = 3 (5,832 DoFs): H~ is the Kronecker sum of three 1D
    operators, whose eigenvectors are formed here from the exported cell matrices."""
    n, p, L = 6, 3, 5.0
    mesh = dg.dftfe_mesh_create(L, n, p)
    ham = dg.dftfe_ham_create(mesh)
    M, ncell, _, nq = dg.dftfe_mesh_info(mesh)
    dg.dftfe_ham_set_potential(ham, torch.zeros(ncell * nq, dtype=torch.float64, device="cuda"))
    dg.dftfe_ham_set_kpoint(ham, (0.0, 0.0, 0.0))
    # 1D operator: H~ applied to a product vector that is constant (in psi) along y and z
    g = n * p
    mass = torch.empty(M, dtype=torch.float64, device="cuda")
    dg.dftfe_ham_export(ham, mass=mass)
    torch.cuda.synchronize()
    m1 = mass.reshape(g, g, g)[0, 0]
    s1 = torch.sqrt(m1 / m1.sum())
    X = torch.einsum("z,y,xn->zyxn", s1, s1, torch.eye(g, dtype=torch.float64, device="cuda")).reshape(M, g).contiguous()
    Y = torch.empty_like(X)
    dg.dftfe_ham_apply(ham, X, Y)
    K1 = X.t() @ Y
    lam, V1 = torch.linalg.eigh(0.5 * (K1 + K1.t()))
    yield ham, M, lam, V1
    dg.dftfe_ham_destroy(ham)
    dg.dftfe_mesh_destroy(mesh)


def _check(dg, ham, X, cplx, ref=None):
    N = X.shape[1]
    ap, rr = (dg.dftfe_ham_apply_z, dg.dftfe_rayleigh_ritz_z) if cplx else (dg.dftfe_ham_apply, dg.dftfe_rayleigh_ritz)
    W = torch.empty_like(X)
    ap(ham, X, W)
    H = X.mH @ W
    H = 0.5 * (H + H.mH)
    th = torch.linalg.eigvalsh(H)
    nrm = max(th.abs().max().item(), 1.0)
    Y, HY, ev = X.clone(), torch.empty_like(X), torch.empty(N, dtype=torch.float64, device="cuda")
    rr(ham, Y, ev, HY)
    torch.cuda.synchronize()
    assert bool((ev[1:] >= ev[:-1]).all())
    assert (ev - th).abs().max().item() <= 1e-12 * nrm
    if ref is not None:
        assert (ev - ref).abs().max().item() <= 1e-11 * nrm
    assert (Y.mH @ Y - torch.eye(N, dtype=Y.dtype, device="cuda")).abs().max().item() <= 1e-12
    off = Y.mH @ HY - torch.diag(ev).to(Y.dtype)
    assert off.abs().max().item() <= 1e-12 * nrm


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 15, 16, 17, 31, 32, 33, 40, 41, 63, 65, 97, 128, 129, 255, 257, 300])
def test_random_blocks(dg, box, N, cplx):
    ham, M, lam, V1 = box
    g = torch.Generator(device="cuda")
    g.manual_seed(N)
    if cplx:
        X = torch.view_as_complex(torch.rand((M, N, 2), generator=g, dtype=torch.float64, device="cuda") - 0.5)
    else:
        X = torch.rand((M, N), generator=g, dtype=torch.float64, device="cuda") - 0.5
    _check(dg, ham, torch.linalg.qr(X)[0].contiguous(), cplx)


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("N", [7, 19, 57, 81, 200, 360])
@pytest.mark.parametrize("rotated", [True, False])
def test_degenerate_spectra(dg, box, N, cplx, rotated):
    """The N lowest states of the box, as they are (H^ diagonal) or rotated at random."""
    ham, M, lam, V1 = box
    e = (lam[:, None, None] + lam[None, :, None] + lam[None, None, :]).reshape(-1)
    idx = torch.argsort(e, stable=True)[:N]
    q = V1.shape[0]
    X = torch.einsum("zn,yn,xn->zyxn", V1[:, idx // (q * q)], V1[:, idx // q % q], V1[:, idx % q]).reshape(M, N)
    if rotated:
        g = torch.Generator(device="cuda")
        g.manual_seed(N)
        R = torch.rand((N, N), generator=g, dtype=torch.float64, device="cuda") - 0.5
        if cplx:
            R = R + 1j * (torch.rand((N, N), generator=g, dtype=torch.float64, device="cuda") - 0.5)
        X = X.to(R.dtype) @ torch.linalg.qr(R)[0]
    elif cplx:
        X = X.to(torch.complex128)
    _check(dg, ham, X.contiguous(), cplx, e[idx])


def test_beyond_the_shared_memory_rows(dg, box):
    """1,900 columns: the rows no longer fit the shared memory of the GPU and Jacobi takes over."""
    ham, M, lam, V1 = box
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    X = torch.linalg.qr(torch.rand((M, 1900), generator=g, dtype=torch.float64, device="cuda") - 0.5)[0].contiguous()
    _check(dg, ham, X, False)


def _unitary(N, blocks, eps, seed):
    """R expm(i eps K), R real orthogonal and K real symmetric, both block diagonal in `blocks` (None:
    one block): H^ = U^H diag(theta) U is real up to an imaginary part of about eps."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    U = torch.zeros((N, N), dtype=torch.complex128, device="cuda")
    for s in range(0, N, blocks or N):
        n = min(blocks or N, N - s)
        R = torch.linalg.qr(torch.rand((n, n), generator=g, dtype=torch.float64, device="cuda") - 0.5)[0]
        K = torch.rand((n, n), generator=g, dtype=torch.float64, device="cuda") - 0.5
        U[s:s + n, s:s + n] = R.to(U.dtype) @ torch.linalg.matrix_exp(1j * eps * (K + K.t()))
    return U


@pytest.mark.parametrize("eps", [1e-8, 1e-9, 1e-10])
@pytest.mark.parametrize("N,blocks", [(2, None), (3, None), (16, 2), (33, 2), (40, None), (65, None)])
def test_weakly_complex_blocks(dg, box, N, blocks, eps):
    """H^ whose imaginary part is eps of its real part, down to the couplings of decoupled 2 x 2
    blocks, where nothing lies below the entry that a reflector makes real."""
    ham, M, lam, V1 = box
    e = (lam[:, None, None] + lam[None, :, None] + lam[None, None, :]).reshape(-1)
    # one state of each level, so that every pair of columns is coupled
    order = torch.argsort(e, stable=True)
    first = torch.cat([torch.ones(1, dtype=torch.bool, device="cuda"), e[order].diff() > 1e-3])
    idx = order[first][:N]
    assert idx.numel() == N
    q = V1.shape[0]
    X = torch.einsum("zn,yn,xn->zyxn", V1[:, idx // (q * q)], V1[:, idx // q % q], V1[:, idx % q]).reshape(M, N)
    _check(dg, ham, (X.to(torch.complex128) @ _unitary(N, blocks, eps, N)).contiguous(), True, e[idx])


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("power", [13, 25, 300, -20, -300])
def test_the_scale_of_the_operator_does_not_matter(dg, box, power, cplx):
    """An empty box 2^power times as long: H~ is 2^(-2 power) times that of the small box, to the last
    bit, and so are the Ritz values; the vectors are the same."""
    ham, M, lam, V1 = box
    N = 72
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    X = torch.rand((M, N, 2), generator=g, dtype=torch.float64, device="cuda") - 0.5
    X = torch.linalg.qr(torch.view_as_complex(X) if cplx else X[:, :, 0])[0].contiguous()
    mesh2 = dg.dftfe_mesh_create(5.0 * 2.0 ** power, 6, 3)
    ham2 = dg.dftfe_ham_create(mesh2)
    try:
        _, ncell, _, nq = dg.dftfe_mesh_info(mesh2)
        dg.dftfe_ham_set_potential(ham2, torch.zeros(ncell * nq, dtype=torch.float64, device="cuda"))
        dg.dftfe_ham_set_kpoint(ham2, (0.0, 0.0, 0.0))
        out = []
        for h in (ham, ham2):
            Y, HY, ev = X.clone(), torch.empty_like(X), torch.empty(N, dtype=torch.float64, device="cuda")
            (dg.dftfe_rayleigh_ritz_z if cplx else dg.dftfe_rayleigh_ritz)(h, Y, ev, HY)
            out.append((Y, HY, ev))
        torch.cuda.synchronize()
        (Y, HY, ev), (Y2, HY2, ev2) = out
        assert torch.equal(ev2 * 4.0 ** power, ev)
        assert torch.equal(Y2, Y) and torch.equal(HY2 * 4.0 ** power, HY)
    finally:
        dg.dftfe_ham_destroy(ham2)
        dg.dftfe_mesh_destroy(mesh2)
