"""Results over the range of scales that FP64 has.  Tolerances are the a-priori rounding bounds."""
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

def _scaled(cell, e):
    """The cell with its potentials and, for e < 0, its kinetic energies 2^e times as large (e
    even; for e > 0 a lattice that small is refused, and H is V and D alone)."""
    f = 2.0 ** (-min(e, 0) // 2)
    cell.lattice = cell.lattice * f
    cell.kpt = cell.kpt / f
    cell.vloc = cell.vloc * 2.0 ** e
    cell.D = cell.D * 2.0 ** e
    return cell


# one block and the block tournament of the FP32 stage; scales whose squares, and that
# themselves, pass float's range.  The refinement must converge from that stage.
@pytest.mark.parametrize("nb", [40, 100])
@pytest.mark.parametrize("e", [-200, -70, 0, 70, 200])
def test_rayleigh_ritz_at_every_scale(nb, e):
    cell = _scaled(make_cell(8.0, 20, 6.0, 2, 8, nb, True, 42), e)
    op = PWOperator.from_cell(cell)
    g = _ctx(cell)
    Y = _F(cell.Y0)
    ev, rs = g.rayleigh_ritz(Y)
    w, Yg = _np(ev), _np(Y)
    assert g.eigensolver_steps >= 1
    w_ref, _ = ch.rayleigh_ritz(op, cell.Y0)
    scale = np.abs(w_ref).max()
    # the Gram matrix's condition number multiplies the rounding of every entry
    tol = 200.0 * nb * U * np.linalg.cond(cell.Y0.conj().T @ op.apply_S(cell.Y0))
    np.testing.assert_allclose(w / scale, w_ref / scale, atol=tol)
    np.testing.assert_allclose(Yg.conj().T @ op.apply_S(Yg), np.eye(nb), atol=tol)
    np.testing.assert_allclose(Yg.conj().T @ op.apply_H(Yg) / scale, np.diag(w) / scale, atol=tol)
    np.testing.assert_allclose(_np(rs) / scale, ch.residuals(op, Yg, w) / scale, atol=tol)


# products that take the modular engine by their size: rows and columns of any scale whose
# products are representable come out exact (integers times powers of two); every way the
# operands are read (columns up to 1024 and 2048, longer columns, rows)
@pytest.mark.parametrize("m,n,k", [(192, 200, 300), (96, 97, 1500), (97, 96, 2100)])
@pytest.mark.parametrize("conjA,conjB", [(False, False), (True, False), (False, True), (True, True)])
def test_modular_gemm_at_every_scale(m, n, k, conjA, conjB):
    rng = np.random.default_rng(m + k)
    a = rng.integers(-1000, 1001, (2, m, k))
    b = rng.integers(-1000, 1001, (2, k, n))
    re, im = a[0] @ b[0] - a[1] @ b[1], a[0] @ b[1] + a[1] @ b[0]
    ei = rng.integers(-900, 901, m)[:, None]
    ei[:4, 0] = [-1010, 1000, 505, -505]
    # columns of the opposite scale, so that products of both signs of exponent are in range
    fj = rng.integers(-60, 61, n)[None, :]
    A = (np.ldexp(1.0, ei) * a[0]) + 1j * (np.ldexp(1.0, ei) * a[1])
    B = (np.ldexp(1.0, fj) * b[0]) + 1j * (np.ldexp(1.0, fj) * b[1])
    with np.errstate(over="ignore", under="ignore"):
        ref_re, ref_im = np.ldexp(re.astype(float), ei + fj), np.ldexp(im.astype(float), ei + fj)
    for flip in (False, True):  # the wide scales on op(A)'s rows, then on op(B)'s columns
        g = _ctx()
        if not flip:
            X, Z, cx, cz = A, B, conjA, conjB
        else:
            X, Z, cx, cz = B.T, A.T, conjA, conjB
        g.profile(True)
        C = _np(g.gemm_fp64(_F(X.conj().T if cx else X), _F(Z.conj().T if cz else Z), cx, cz))
        assert "k_oz_gemm" in g.profile_totals()
        C = C.T if flip else C
        inside = (ei + fj > -1000) & (ei + fj < 950)  # in FP64's normal range
        assert np.array_equal(np.where(inside, C.real, 0), np.where(inside, ref_re, 0))
        assert np.array_equal(np.where(inside, C.imag, 0), np.where(inside, ref_im, 0))


def _vpart(cell, Y):
    """The sphere's coefficients of V psi in extended precision, and ||V psi|| + ||V|| rms(psi), what
    an FP64 transform's rounding is relative to."""
    n = int(cell.grid[0])
    m = np.asarray(cell.miller) % n
    out, size = np.empty(Y.shape, np.clongdouble), np.empty(Y.shape[1])
    V = cell.vloc.astype(np.longdouble)
    for j in range(Y.shape[1]):
        box = np.zeros((n, n, n), np.clongdouble)
        box[m[:, 0], m[:, 1], m[:, 2]] = Y[:, j]
        psi = np.fft.ifftn(box) * np.longdouble(n) ** 3
        f = V * psi
        out[:, j] = (np.fft.fftn(f) / np.longdouble(n) ** 3)[m[:, 0], m[:, 1], m[:, 2]]
        size[j] = (np.linalg.norm(f.astype(complex)) +
                   np.linalg.norm(cell.vloc) * np.linalg.norm(Y[:, j])) / n ** 1.5
    return out, size


def _without_kinetic(n, core=0.0, scale=1.0):
    """A cell so large that its kinetic energies are 2^-120 of their size, and no projectors' part."""
    L = 0.42 * n
    cell = make_cell(L, n, 0.5 * (2.0 * np.pi / L * 0.23 * n) ** 2, 1, 8, 3, False, 43, kpt=(0.02, -0.05, 0.03))
    cell.D = np.zeros_like(cell.D)
    cell.vloc = cell.vloc * scale
    if core:
        cell.vloc[n // 3, n // 5, n // 2] = core
    cell.lattice = cell.lattice * 2.0 ** 60
    cell.kpt = cell.kpt * 2.0 ** -60
    return cell


def _vpart_error(cell):
    """Errors of V psi, relative to what an FP64 transform's rounding is relative to."""
    ref, size = _vpart(cell, cell.Y0)
    got = _np(_ctx(cell).apply_H(_F(cell.Y0)))
    return np.linalg.norm((got - ref).astype(complex), axis=0) / size


# V psi alone, for an ordinary potential, and one with a core at one point.  3 log2 n levels
# each way that round half a unit each, adding up as their root; on the lengths with
# double-float z passes, twice what those round without the core
@pytest.mark.parametrize("n", [36, 60, 64, 80])
def test_a_core_takes_no_bits_from_the_other_planes(n):
    plain = _vpart_error(_without_kinetic(n))
    cored = _vpart_error(_without_kinetic(n, 64.0))
    if n == 64:
        assert cored.max() <= 2.0 * plain.max()
    else:
        assert max(plain.max(), cored.max()) <= 0.5 * np.sqrt(6.0 * np.log2(n)) * U, (plain / U, cored / U)


# Potentials far from one, whose planes' exponents are far from zero.  A power of two changes no
# digit of V psi: the results differ by it and no more than the rounding of the kinetic part's
# 2^-80 beside it (on the double-float lengths a unit of the pairs)
@pytest.mark.parametrize("n", [16, 24, 48, 60, 90, 96])
@pytest.mark.parametrize("e", [-40, -3, 3, 30])
def test_local_potential_of_any_size(n, e):
    cell = _without_kinetic(n)
    one = _np(_ctx(cell).apply_H(_F(cell.Y0)))
    ref = PWOperator.from_cell(cell).apply_H(cell.Y0)
    assert np.abs(one - ref).max() <= 1e-11 * np.abs(ref).max()  # the FP64 form's parity tolerance
    got = _np(_ctx(_without_kinetic(n, scale=2.0 ** e)).apply_H(_F(cell.Y0))) * 2.0 ** -e
    assert np.abs(got - one).max() <= 2.0 ** -46 * np.abs(one).max()


# products that the FP64 units would take longer for, and that no caller has asked to round
# differently: no less exact than on those units, entry by entry and on operands of this library
@pytest.mark.parametrize("what", ["square", "deep", "PhY", "Gp", "gram"])
def test_products_of_middle_size_are_as_exact_as_fp64(what):
    from paper_1406_4350_gb300._lib import GEMM_CUDA_CORES
    rng = np.random.default_rng(44)

    def rand(*s):
        return rng.standard_normal(s) + 1j * rng.standard_normal(s)
    if what == "square":
        A, B = rand(256, 256), rand(256, 256)
    elif what == "deep":
        A, B = rand(6000, 200), rand(6000, 30)
    else:
        cell = make_cell(12.0, 30, 8.0, 32, 8, 128, True, 45)
        p = cell.P.conj().T @ cell.Y0
        A, B = {"PhY": (cell.P, cell.Y0), "Gp": (cell.P.conj().T @ cell.P, p), "gram": (cell.Y0, cell.Y0)}[what]
    m, n = A.shape[1], B.shape[1]
    assert 6e7 <= 8.0 * m * n * A.shape[0] < 1e9
    i, j = rng.integers(0, m, 200), rng.integers(0, n, 200)
    ref = np.array([(A[:, a].conj().astype(np.clongdouble) * B[:, b].astype(np.clongdouble)).sum()
                    for a, b in zip(i, j)])
    size = np.array([(np.abs(A[:, a]) * np.abs(B[:, b])).sum() for a, b in zip(i, j)])
    err = []
    for engine in (None, GEMM_CUDA_CORES):
        g = _ctx()
        if engine is not None:
            g.set_fp64_gemm(engine)
        g.profile(True)
        C = _np(g.gemm_fp64(_F(A), _F(B), conjA=True))
        assert ("k_oz_gemm" in g.profile_totals()) == (engine is None)
        err.append(np.sqrt(np.mean((np.abs((C[i, j] - ref).astype(complex)) / size) ** 2)))
    assert err[0] <= err[1], (err[0] / U, err[1] / U)
