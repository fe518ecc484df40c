"""The rounding errors that the filtered iteration's certificate allows for,
restated in numpy: a blocked FP32 factorisation of the scaled, lifted matrix
(filt_lift_kernel, ldl64_*_kernel) against the matrix it factors, for cells up to
a contrast that the iteration would not take.  The certificate takes the norm of
the error as (128 + 4 sqrt(n)) u; the spectral norm has to stay below half of
that, and the pivots positive when sigma lies below the next eigenvalue."""
import numpy as np
import pytest
import scipy.linalg as sla

from oracle import mixed_variational as mv
from paper_1310_6380_gb300 import cells

U = 2.0 ** -24
f4, c8 = np.float32, np.complex64


def factor(A):
    """Right-looking LDL^dagger in complex64, panels of 64."""
    A, n = A.astype(c8).copy(), len(A)
    L, d = np.eye(n, dtype=c8), np.zeros(n, f4)
    for j0 in range(0, n, 64):
        j1 = min(n, j0 + 64)
        for c in range(j0, j1):
            d[c] = A[c, c].real
            L[c + 1:, c] = A[c + 1:, c] / d[c]
            A[c + 1:, c + 1:j1] -= np.outer(A[c + 1:, c], L[c + 1:j1, c].conj())
        A[j1:, j1:] -= (L[j1:, j0:j1] * d[j0:j1]) @ L[j1:, j0:j1].conj().T
    return L, d


def scaled(C, s, shift, w32):
    """W (C / s + shift) W with the roundings of the kernel."""
    off = (C.real.astype(f4) + 1j * C.imag.astype(f4)).astype(c8) * f4(1.0 / s)
    np.fill_diagonal(off, (C.diagonal().real / s + shift).astype(f4))
    return off * (w32[:, None] * w32)


def circle(contrast, M):
    m = np.array([4.0, 1.5, 1.2])
    return cells.circle_cell(48, 0.3, tuple(m), tuple(m * [contrast, contrast, 2.0])), M


@pytest.mark.parametrize("cell, M", [circle(1e-3, 4), circle(0.02, 5), circle(1.0, 5),
                                     circle(30.0, 6), circle(1e4, 4),
                                     (cells.voronoi_cell(32, 20, seed=3), 3),
                                     (cells.voronoi_cell(48, 60, seed=4), 7),
                                     (cells.steel_epoxy_hex_cell(32), 5)])
def test_error_of_the_factorisation(cell, M):
    nb = 10
    oc = mv.OracleCell(cell, M)
    A, Om = oc.pencil(np.array([0.21, 0.13]))
    Lr = np.linalg.cholesky(Om)
    C = sla.solve_triangular(Lr, sla.solve_triangular(Lr, A, lower=True).conj().T, lower=True)
    C = 0.5 * (C + C.conj().T)
    n = len(C)
    th, V = np.linalg.eigh(C)
    dg = C.diagonal().real
    s = 0.2 * np.sort(dg)[nb - 1]
    w32 = np.sqrt(s / (dg + s)).astype(f4)
    w = w32.astype(float)
    i = nb - 1 + int(np.argmax(np.diff(th[nb - 1:32])))      # the widest gap
    sigma, lift = 0.5 * (th[i] + th[i + 1]), th[i + 1] - th[:i + 1]
    z = V[:, :i + 1].astype(c8) * w32[:, None] * np.sqrt((lift / s).astype(f4))
    exact = (w[:, None] * w) * (C / s - sigma / s * np.eye(n)) + z.astype(complex) @ z.conj().T.astype(complex)
    L, d = factor(scaled(C, s, -sigma / s, w32) + z @ z.conj().T)
    E = L.astype(complex) @ (d[:, None] * L.conj().T.astype(complex)) - exact
    assert np.linalg.norm(E, 2) <= (64 + 2 * np.sqrt(n)) * U
    assert exact.diagonal().real.max() <= 2
    assert (d > 0).all()
    # and one vector short it is not positive
    _, d = factor(scaled(C, s, -sigma / s, w32) + z[:, 1:] @ z[:, 1:].conj().T)
    assert (d < 0).sum() == 1
