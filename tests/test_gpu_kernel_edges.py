"""Kernels at the edges of their tiles, blocks and dispatch ranges, against the oracle or a
numpy product in extended precision.  Tolerances are the a-priori rounding bounds."""
import numpy as np
import pytest
import torch

from oracle import chebyshev as ch
from oracle.planewave import PWOperator
from synth import make_cell

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1406_4350_gb300 import build
    build.build()


def _F(x):
    from paper_1406_4350_gb300.chebfi import fortran
    return fortran(x)


def _np(t):
    torch.cuda.synchronize()
    return t.cpu().numpy()


def _ctx(cell=None):
    from paper_1406_4350_gb300.chebfi import ChebFI
    return ChebFI.from_cell(cell) if cell is not None else ChebFI(0)


def _rand(rng, m, n):
    return rng.standard_normal((m, n)) + 1j * rng.standard_normal((m, n))


# one entry; one short of, at and past the 8 x 32, 16 x 16 and 32 x 8 tiles; K below one k
# tile, at it, past it, and long enough to be split to the last tile
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (8, 32, 1021), (9, 33, 16), (7, 31, 17), (32, 8, 300), (33, 7, 15),
                                   (15, 17, 2049), (16, 16, 64), (1021, 32, 8), (300, 3, 40)])
@pytest.mark.parametrize("conjA,conjB", [(False, False), (True, False), (False, True), (True, True)])
def test_cuda_core_fp64_gemm(m, n, k, conjA, conjB):
    from paper_1406_4350_gb300._lib import GEMM_CUDA_CORES
    rng = np.random.default_rng(100 * m + 10 * n + k)
    A = _rand(rng, k, m) if conjA else _rand(rng, m, k)
    B = _rand(rng, n, k) if conjB else _rand(rng, k, n)
    C0 = _rand(rng, m, n)
    a = A.conj().T if conjA else A
    b = B.conj().T if conjB else B
    ref = 0.5 * (a.astype(np.clongdouble) @ b.astype(np.clongdouble)) + 2.0 * C0
    g = _ctx()
    g.set_fp64_gemm(GEMM_CUDA_CORES)
    C = _np(g.gemm_fp64(_F(A), _F(B), conjA, conjB, alpha=0.5, beta=2.0, C=_F(C0)))
    bound = (2 * k + 8) * U * (np.abs(a) @ np.abs(b) + 2.0 * np.abs(C0))
    assert np.all(np.abs((C - ref).astype(complex)) <= 2.0 * bound)


# one 32 x 32 diagonal block, its edges, two blocks, and the recursive factor's 256-leaf edge
@pytest.mark.parametrize("nb", [1, 2, 31, 32, 33, 64, 95, 257])
def test_cholesky_qr_block_edges(nb):
    cell = make_cell(8.0, 20, 6.0, 2, 8, nb, True, 31)
    op = PWOperator.from_cell(cell)
    g = _ctx(cell)
    Y = _F(cell.Y0)
    g.orthonormalise(Y)
    Yg = _np(Y)
    # Y = Y0 L^-H with S-Gram L L^H: S-orthonormal, and Y^H S Y0 = L^H is upper triangular
    # with a positive real diagonal
    SY0 = op.apply_S(cell.Y0)
    gram = cell.Y0.conj().T @ SY0
    tol = 50.0 * nb * U * np.linalg.cond(gram)
    np.testing.assert_allclose(Yg.conj().T @ op.apply_S(Yg), np.eye(nb), atol=tol)
    LH = Yg.conj().T @ SY0
    scale = np.sqrt(np.abs(np.diag(gram)).max())
    assert np.abs(np.tril(LH, -1)).max(initial=0.0) <= tol * scale
    assert np.all(np.diag(LH).real > 0) and np.abs(np.diag(LH).imag).max() <= tol * scale


# the modular GEMM: one entry; one short of, at and past its 256-row tile, the 128-row halves
# of a CTA pair, the 128- and 256-column forms; K below and past a k-tile and a 512-product
# chunk, and long with few tiles (split over K); rows past M inside a group of four
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (127, 128, 63), (129, 129, 65), (256, 256, 512), (255, 257, 513),
                                   (258, 300, 1030), (30, 7, 20001), (511, 127, 9000)])
def test_modular_gemm_is_exact_on_integers(m, n, k):
    from paper_1406_4350_gb300._lib import GEMM_TENSOR
    rng = np.random.default_rng(m + n + k)
    A = rng.integers(-1000, 1001, (k, m)) + 1j * rng.integers(-1000, 1001, (k, m))
    B = rng.integers(-1000, 1001, (k, n)) + 1j * rng.integers(-1000, 1001, (k, n))
    ar, ai = A.real.astype(np.int64).T, -A.imag.astype(np.int64).T
    br, bi = B.real.astype(np.int64), B.imag.astype(np.int64)
    g = _ctx()
    g.set_fp64_gemm(GEMM_TENSOR, 14)
    C = _np(g.gemm_fp64(_F(A), _F(B), conjA=True))
    assert np.array_equal(C.real, (ar @ br - ai @ bi).astype(np.float64))
    assert np.array_equal(C.imag, (ar @ bi + ai @ br).astype(np.float64))


# the eigensolver's routes: FP64 Jacobi below 8 bands, one block up to 32 and 64, the block
# tournament from 65 (an even and an odd number of 64-column tiles), general and clustered
# spectra (S = I, V = 0: the free-electron shells, exactly degenerate)
@pytest.mark.parametrize("nb", [2, 7, 8, 31, 33, 64, 65, 129, 192])
@pytest.mark.parametrize("shells", [False, True])
def test_rayleigh_ritz_route_edges(nb, shells):
    cell = make_cell(8.0, 20, 6.0, 2, 8, nb, not shells, 33)
    if shells:
        cell.vloc = np.zeros_like(cell.vloc)
        cell.D = np.zeros_like(cell.D)
    op = PWOperator.from_cell(cell)
    g = _ctx(cell)
    Y = _F(cell.Y0)
    ev, rs = g.rayleigh_ritz(Y)
    w, Yg = _np(ev), _np(Y)
    w_ref, _ = ch.rayleigh_ritz(op, cell.Y0)
    scale = np.abs(w_ref).max()
    # the Gram matrix's condition number multiplies the rounding of every entry
    cond = np.linalg.cond(cell.Y0.conj().T @ op.apply_S(cell.Y0))
    tol = 200.0 * nb * U * cond
    np.testing.assert_allclose(w, w_ref, atol=tol * scale)
    np.testing.assert_allclose(Yg.conj().T @ op.apply_S(Yg), np.eye(nb), atol=tol)
    np.testing.assert_allclose(Yg.conj().T @ op.apply_H(Yg), np.diag(w), atol=tol * scale)
    np.testing.assert_allclose(_np(rs), ch.residuals(op, Yg, w), atol=tol * scale)


# every grid length with compiled FFT passes (and two without: 18 and 50), a sphere that is
# not centred (general k), band counts that leave the last block ragged
@pytest.mark.parametrize("n", [16, 18, 20, 24, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 80, 90, 96, 100, 108])
def test_apply_h_on_every_grid_length(n):
    L = 0.42 * n
    ecut = 0.5 * (2.0 * np.pi / L * 0.24 * n) ** 2
    cell = make_cell(L, n, ecut, 1, 8, 3, True, 35, kpt=(0.02, -0.05, 0.03))
    ref = PWOperator.from_cell(cell).apply_H(cell.Y0)
    g = _ctx(cell)
    scale = np.abs(ref).max()
    # the parity tolerances of the FP64 and FP32 forms
    assert np.abs(_np(g.apply_H(_F(cell.Y0), prec=0)) - ref).max() <= 1e-11 * scale
    assert np.abs(_np(g.apply_H(_F(cell.Y0), prec=1)) - ref).max() <= 2e-5 * scale


# the fixed-point plane pass of the FP64 form: potentials and blocks at the ends of its scales
# (a band's planes are scaled by their own sums, the product with V_loc by its own maximum)
@pytest.mark.parametrize("n", [24, 32, 48, 64, 72, 96])
@pytest.mark.parametrize("kind", ["plain", "tiny", "huge", "spike", "zero", "core"])
def test_fixed_point_planes_at_every_scale(n, kind):
    L = 0.42 * n
    ecut = 0.5 * (2.0 * np.pi / L * 0.23 * n) ** 2
    cell = make_cell(L, n, ecut, 1, 8, 6, False, 36, kpt=(0.02, -0.05, 0.03))
    cell.D = np.zeros_like(cell.D)
    V = cell.vloc
    if kind == "tiny":
        V = V * 1e-12
    elif kind == "huge":
        V = V * 1e9
    elif kind == "zero":
        V = np.zeros_like(V)
    elif kind == "spike":
        V = np.zeros_like(V)
        V[n // 3, n // 5, n // 2] = -7.0
    elif kind == "core":  # a hard core beside an ordinary potential
        V = V.copy()
        V[1, 2, 3] = 1e6
    cell.vloc = V
    Y = cell.Y0.copy()
    Y[:, 1] *= 1e18
    Y[:, 2] *= 1e-18
    Y[:, 3] = 0.0
    Y[:, 4] = 0.0
    Y[cell.npw // 2, 4] = 1.0  # one plane wave: every plane's sum is its one column's value
    Y[:, 5] = 1.0              # all in phase: the sum is attained at the origin
    op = PWOperator.from_cell(cell)
    ref = op.apply_H(Y)
    got = _np(_ctx(cell).apply_H(_F(Y)))
    # H y = K y + V y: the double-float z passes round 2^-44 of a line's norm, the planes less
    norm = np.linalg.norm(Y, axis=0)
    tol = 2.0 ** -43 * (np.abs(V).max() + ecut) * norm
    assert np.all(np.linalg.norm(got - ref, axis=0) <= tol)
    assert np.all(got[:, 3] == 0.0)


def test_fixed_point_planes_keep_non_finite_bands_apart():
    cell = make_cell(10.0, 24, 6.0, 1, 8, 4, False, 37)
    Y = cell.Y0.copy()
    Y[5, 1] = np.nan
    Y[7, 2] = np.inf
    g = _ctx(cell)
    got = _np(g.apply_H(_F(Y)))
    good = _np(g.apply_H(_F(cell.Y0)))
    assert np.isnan(got[:, 1]).all() and np.isnan(got[:, 2]).all()
    assert np.array_equal(got[:, [0, 3]], good[:, [0, 3]])


# the FP32 CUDA-core GEMM through the FP32 filter: projector and band counts at the edges of
# its 64 x 64 and 64 x 32 tiles and of its K splits, with and without S
@pytest.mark.parametrize("nb", [1, 31, 33, 64, 65, 130])
@pytest.mark.parametrize("natoms,nlmn,paw", [(1, 1, False), (8, 8, True), (9, 8, True)])
def test_fp32_filter_tile_edges(nb, natoms, nlmn, paw):
    cell = make_cell(12.0, 30, 5.0, natoms, nlmn, nb, paw, 38)
    op = PWOperator.from_cell(cell)
    lo, hi, _, _ = ch.bounds(op, cell.Y0, mode="rigorous")
    ref = ch.filter_plain(op, cell.Y0, 3, lo, hi)
    g = _ctx(cell)
    Y = _F(cell.Y0)
    g.cheb_filter(Y, 3, lo, hi, prec=1)
    assert np.abs(_np(Y) - ref).max() <= 2e-5 * 3 * np.abs(ref).max()  # the FP32 tolerance per step


# the derivative with respect to V_loc on grids with fixed-point planes, compiled FP64 planes
# and the general passes; bands of very different sizes share no scale
@pytest.mark.parametrize("n", [16, 18, 24, 30, 32, 45, 48, 60, 64])
def test_vloc_gradient_on_every_kind_of_grid(n):
    L = 0.42 * n
    ecut = 0.5 * (2.0 * np.pi / L * 0.24 * n) ** 2
    cell = make_cell(L, n, ecut, 1, 8, 5, True, 39, kpt=(0.02, -0.05, 0.03))
    rng = np.random.default_rng(n)
    Y, G = cell.Y0.copy(), _rand(rng, cell.npw, 5)
    Y[:, 1] *= 1e9
    G[:, 1] *= 1e-9
    Y[:, 2] = 0.0
    m = np.asarray(cell.miller)

    def box(c):
        b = np.zeros((n, n, n), dtype=complex)
        b[m[:, 0] % n, m[:, 1] % n, m[:, 2] % n] = c
        return np.fft.ifftn(b) * n ** 3
    ref = sum((box(G[:, j]).conj() * box(Y[:, j])).real for j in range(5)) / n ** 3
    g = _ctx(cell)
    _, gV, _ = g.apply_H_backward(_F(Y), _F(G), (n, n, n), len(cell.D))
    # two transforms of log2(n^3) levels and the product, each about 2^-52 of its norm
    bound = 64.0 * 2.0 ** -52 * sum(np.linalg.norm(G[:, j]) * np.linalg.norm(Y[:, j]) for j in range(5)) / n ** 1.5
    assert np.linalg.norm(_np(gV) - ref) <= bound


# fixed-point planes between FP64 z passes (the compiled lengths without double-float passes)
# against the oracle and against the FP64 units, over FP64's range of scales
@pytest.mark.parametrize("n", [16, 20, 30, 36, 40, 45, 54, 60, 80, 90, 100, 108])
@pytest.mark.parametrize("kind", ["plain", "tiny", "huge", "spike"])
def test_fixed_point_planes_between_fp64_passes(n, kind):
    L = 0.42 * n
    ecut = 0.5 * (2.0 * np.pi / L * 0.23 * n) ** 2
    cell = make_cell(L, n, ecut, 1, 8, 6, False, 40, kpt=(0.02, -0.05, 0.03))
    cell.D = np.zeros_like(cell.D)
    V = cell.vloc * {"plain": 1.0, "tiny": 1e-12, "huge": 1e9, "spike": 0.0}[kind]
    if kind == "spike":
        V[n // 3, n // 5, n // 2] = -7.0
    cell.vloc = V
    Y = cell.Y0.copy()
    Y[:, 1] *= 1e150
    Y[:, 2] *= 1e-150
    Y[:, 3] = 0.0
    Y[:, 4] = 0.0
    Y[cell.npw // 2, 4] = 1.0
    Y[:, 5] = 1.0
    ref = PWOperator.from_cell(cell).apply_H(Y)
    g = _ctx(cell)
    got = _np(g.apply_H(_F(Y)))
    g.set_fft64(0)
    native = _np(g.apply_H(_F(Y)))
    # two transforms of log2(n^3) <= 21 levels and the product, each about 2^-52 of its norm;
    # norms by the largest component first, as 1e-150 squared is zero
    size = np.abs(Y).max(axis=0)
    size[3] = 1.0
    norm = np.linalg.norm(Y / size, axis=0)
    tol = 64.0 * 2.0 ** -52 * (np.abs(V).max() + ecut) * norm
    assert np.all(np.linalg.norm((got - ref) / size, axis=0) <= tol)
    assert np.all(np.linalg.norm((got - native) / size, axis=0) <= tol)
    assert np.all(got[:, 3] == 0.0)


def test_non_finite_bands_stay_apart_between_fp64_passes():
    cell = make_cell(10.0, 30, 6.0, 1, 8, 4, False, 37)
    Y = cell.Y0.copy()
    Y[5, 1] = np.nan
    Y[7, 2] = np.inf
    g = _ctx(cell)
    got = _np(g.apply_H(_F(Y)))
    good = _np(g.apply_H(_F(cell.Y0)))
    assert np.isnan(got[:, 1]).all() and np.isnan(got[:, 2]).all()
    assert np.array_equal(got[:, [0, 3]], good[:, [0, 3]])
