"""The certificate of the filtered iteration on matrices it has to refuse.

Each matrix is block diagonal: 160 rows with the eigenvalues 1, 2, 3, ... (rotated
a little, so that there is something to iterate on) and a dense block of
large diagonal D whose eigenvalues are D and above, but for one that may lie
among the wanted ones.  The starting vectors, sums of unit vectors of the 128
smallest diagonal entries, have no part in the dense block and the products keep
exact zeros there, so an eigenvalue in it is always skipped by the iteration;
only the factorisation can show it.  From D = 1e7 on its mark in the scaled
matrix is below the rounding errors of an FP32 factorisation.

Tolerance on lambda: a Householder reduction and its bisection err by less
than (n + 4) eps64 ||C||, the certificate allows 64 eps64 max C_rr; ||C|| <= 2 D
here and max C_rr >= D, so 2 (n + 128) eps64 max C_rr.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1310_6380_gb300 import binding as bs  # noqa: E402
from paper_1310_6380_gb300 import cells  # noqa: E402

EPS = np.finfo(float).eps
NV = 160


def matrices(n, D, hidden, count, seed):
    """(count, n, n) and their eigenvalues; hidden: the dense block's low eigenvalue or None."""
    rng = np.random.default_rng(seed)
    C, lam = np.zeros((count, n, n), complex), np.empty((count, n))
    for i in range(count):
        q = n - NV
        low = np.arange(1.0, NV + 1) + 0.1 * rng.random(NV)
        K = rng.standard_normal((NV, NV)) + 1j * rng.standard_normal((NV, NV))
        V = np.linalg.qr(np.eye(NV) + 0.02 * (K - K.conj().T))[0]
        C[i, :NV, :NV] = (V * low) @ V.conj().T
        high = D * (1.0 + rng.random(q))
        if hidden is not None:
            high[0] = hidden
        V = np.linalg.qr(rng.standard_normal((q, q)) + 1j * rng.standard_normal((q, q)))[0]
        C[i, NV:, NV:] = (V * high) @ V.conj().T
        C[i] = 0.5 * (C[i] + C[i].conj().T)
        lam[i] = np.sort(np.concatenate([low, high]))
    return C, lam


def solve(C, nb):
    w, red = np.empty((len(C), nb)), np.full(len(C), 7, np.int32)
    bs.bs_lowest_eigenvalues(np.ascontiguousarray(C), nb, w, red)
    return w ** 2, red


@pytest.mark.parametrize("n, D", [(288, 1e3), (288, 1e4), (290, 1e6), (300, 1e7), (352, 1e8),
                                  (352, 1e9)])
def test_a_skipped_eigenvalue_is_found(n, D):
    nb = 6
    C, lam = matrices(n, D, 2.5, 24, int(np.log10(D)))
    got, red = solve(C, nb)
    assert np.abs(got - lam[:, :nb]).max() <= 2 * (n + 128) * EPS * np.abs(C).max()
    assert red.all()


@pytest.mark.parametrize("n, D, nb", [(192, 1e3, 1), (288, 1e3, 6), (300, 1e3, 22)])
def test_nothing_skipped_is_certified(n, D, nb):
    C, lam = matrices(n, D, None, 24, n)
    got, red = solve(C, nb)
    assert np.abs(got - lam[:, :nb]).max() <= 2 * (n + 128) * EPS * np.abs(C).max()
    assert not red.any()


def spectrum_matrices(n, low, high, angle, count, seed):
    """Hermitian matrices with the given eigenvalues `low`, the others evenly in `high`,
    whose eigenvectors are unit vectors turned into each other by about `angle`."""
    rng = np.random.default_rng(seed)
    C, lam = np.empty((count, n, n), complex), np.empty((count, n))
    for i in range(count):
        lam[i] = np.sort(np.concatenate([low, np.linspace(*high, n - len(low))]))
        K = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
        V = np.linalg.qr(np.eye(n) + angle / np.sqrt(n) * (K - K.conj().T))[0]
        C[i] = (V * lam[i]) @ V.conj().T
        C[i] = 0.5 * (C[i] + C[i].conj().T)
        # positive semidefinite to rounding, with a diagonal that is not negative
    return C, lam


@pytest.mark.parametrize("n", [98, 200])
@pytest.mark.parametrize("low", [[1e-6], [1e-4, 1e-4], [0.01, 0.02, 20.0]], ids=["one", "two", "three"])
@pytest.mark.parametrize("top", [1e3, 1e5])
@pytest.mark.parametrize("angle", [0.1, 0.5])
def test_lone_low_eigenvalues(n, low, top, angle):
    """A few eigenvalues far below the others, as at wavevectors near Gamma: the
    filters grow them in every column, the Gram matrices become
    ill-conditioned, and the small eigenproblem begins far from diagonal."""
    C, lam = spectrum_matrices(n, low, (50.0, top), angle, 16, n)
    got, red = solve(C, len(low))
    assert np.abs(got - lam[:, :len(low)]).max() <= (n + 128) * EPS * top


@pytest.mark.parametrize("kind, n, nb, angle", [
    ("even", 97, 22, 1.0), ("even", 98, 22, 0.3), ("even", 128, 15, 0.3), ("levels", 98, 7, 0.3),
    ("levels", 129, 11, 0.1), ("lone", 98, 13, 0.3)])
def test_ritz_values_keep_48_bits(kind, n, nb, angle):
    """Many random spectra (even, on 41 levels, a low group far below the others): the
    vectors of the small eigenproblem enter the Ritz values in 48 bits however
    many rotations they went through.  Tolerance: (n + 4) eps64 ||C|| for the reference's
    reduction, the certificate's 64 eps64 max C_rr."""
    rng = np.random.default_rng(n)
    count, top = 384, 1e4
    C = np.empty((count, n, n), complex)
    for i in range(count):
        lam = top * rng.random(n)
        if kind == "levels":
            lam = np.round(lam / top * 40) * (top / 40)
        elif kind == "lone":
            lam = np.concatenate([10.0 ** rng.uniform(-6, 1, nb), rng.uniform(20, 40, n - nb)])
        K = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
        V = np.linalg.qr(np.eye(n) + angle / np.sqrt(n) * (K - K.conj().T))[0]
        C[i] = (V * np.sort(lam)) @ V.conj().T
        C[i] = 0.5 * (C[i] + C[i].conj().T)
    lam = np.linalg.eigvalsh(C)
    got, _ = solve(C, nb)
    err = np.abs(got - np.maximum(lam[:, :nb], 0.0)).max(1)
    tol = EPS * ((n + 4) * lam[:, -1] + 64 * np.einsum("kii->ki", C).real.max(1))
    assert (err / tol).max() <= 1.0


@pytest.mark.parametrize("e", [-400, -120, -40, 40, 62, 124, 400])
def test_any_unit(e):
    """A power of two as the unit changes no bit of any step: the same matrices
    are certified and omega is 2^(e/2) times as large.  (The Ritz values of an
    epoxy/steel cell of 10 um in SI units, near 2^62, have squares beyond FP32.)"""
    C, _ = matrices(230, 1e3, None, 4, 3)
    C = np.ascontiguousarray(C)
    w, red = np.empty((4, 8)), np.full(4, 7, np.int32)
    bs.bs_lowest_eigenvalues(C, 8, w, red)
    we, rede = np.empty((4, 8)), np.full(4, 7, np.int32)
    bs.bs_lowest_eigenvalues(C * 2.0 ** e, 8, we, rede)
    assert not red.any() and not rede.any()
    assert np.array_equal(we, w * 2.0 ** (e // 2))


def reduced_matrices(cell, M, Q, nb, f=1.0):
    """C(k) of a cell whose lattice is scaled by f, and bs_solve_k's omega of it."""
    h = bs.bs_create_cell(np.asarray(cell.h1) * f, np.asarray(cell.h2) * f,
                          np.ascontiguousarray(cell.phase, np.uint16), cell.lam.copy(),
                          cell.mu.copy(), cell.rho.copy(), M, bs.BS_PREC_FP64)
    try:
        bs.bs_assemble(h)
        n = bs.bs_cell_dims(h)[1]
        C = np.empty((len(Q), n, n), np.complex128)
        for k in range(len(Q)):
            bs.bs_reduced_matrix(h, Q[k].copy(), C[k].view(np.float64))
        st, w = np.full(len(Q), 7, np.int32), np.empty((len(Q), nb))
        bs.bs_solve_k(h, Q, nb, w, st)
    finally:
        bs.bs_destroy_cell(h)
    assert not st.any()
    low = np.tril(C.transpose(0, 2, 1), -1)
    d = np.einsum("kii->ki", C).real
    return low + low.conj().transpose(0, 2, 1) + d[:, :, None] * np.eye(n), w


@pytest.mark.parametrize("a", [1e-6, 1e-5, 6.023e-3, 1e3])
def test_cells_of_any_size_are_certified(a):
    """The steel/epoxy cell in SI units at lattice constants from 1 um to 1 km:
    omega a does not depend on a."""
    cell = cells.steel_epoxy_hex_cell(48)
    scale = a / np.linalg.norm(cell.h1)
    Q = np.array([[0.13, 0.21], [0.5, 0.0], [0.3, 0.3]])
    ref = None
    for f in (1.0, scale):
        C, ws = reduced_matrices(cell, 4, Q, 12, f)
        w, red = np.empty((3, 12)), np.full(3, 7, np.int32)
        bs.bs_lowest_eigenvalues(np.ascontiguousarray(C), 12, w, red)
        assert not red.any()
        tol = 2 * (C.shape[1] + 128) * EPS * np.abs(C).max()
        assert np.abs(w ** 2 - ws ** 2).max() <= tol
        if ref is None:
            ref = w
        else:
            assert np.abs((w * f) ** 2 - ref ** 2).max() <= 2 * tol * f * f


def supercell(cell, t):
    cell.phase = np.tile(cell.phase[::t, ::t], (t, t))
    return cell


@pytest.mark.parametrize("make, M, nb", [
    (lambda: cells.bilayer_cell(48), 3, 8), (lambda: cells.bilayer_cell(48), 5, 18),
    (lambda: cells.bilayer_cell(48, layer1=(4, 1.5, 1.2), layer2=(8, 4, 2)), 5, 22),
    (lambda: cells.bilayer_cell(48), 7, 18),
    (lambda: supercell(cells.circle_cell(48, 0.3), 2), 5, 18),
    (lambda: supercell(cells.circle_cell(48, 0.3), 3), 5, 18)])
def test_cells_whose_matrices_fall_apart(make, M, nb):
    """C(k) of layered cells and of supercells is block diagonal: every block is
    reached, so all are certified."""
    cell = make()
    Q = np.ascontiguousarray(cells.ibz_path("square", 41, cell.h1, cell.h2)[1::2])
    C, ws = reduced_matrices(cell, M, Q, nb)
    w, red = np.empty((len(Q), nb)), np.full(len(Q), 7, np.int32)
    bs.bs_lowest_eigenvalues(np.ascontiguousarray(C), nb, w, red)
    assert np.abs(w ** 2 - ws ** 2).max() <= 2 * (C.shape[1] + 128) * EPS * np.abs(C).max()
    assert not red.any()
