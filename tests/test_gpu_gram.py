"""The Gram factors of FP64 cells (16 x 16 output tiles, inverse by doubling)
against those of mixed cells (32-wide panels) through the reduced matrix C(k),
at orders that are ragged against the tiles (N = 9 ... 361).

Both factorisations are backward stable: C = L^-1 H T^-1 H^* L^-* differs by a
modest multiple of N eps64 times the condition numbers of the two Gram matrices,
taken from the oracle.
"""
import numpy as np
import pytest

from oracle import mixed_variational as mv
from paper_1310_6380_gb300 import cells

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1310_6380_gb300 import binding as bs  # noqa: E402

EPS = np.finfo(float).eps


@pytest.mark.parametrize("M", [1, 2, 3, 4, 5, 7, 9])
def test_factors_agree(M):
    cell = cells.voronoi_cell(48, 9, seed=M, lattice="hex" if M % 2 else "square")
    C = []
    for prec in (bs.BS_PREC_FP64, bs.BS_PREC_MIXED):
        h = bs.bs_create_cell(cell.h1, cell.h2, np.ascontiguousarray(cell.phase, np.uint16),
                              cell.lam.copy(), cell.mu.copy(), cell.rho.copy(), M, prec)
        try:
            bs.bs_assemble(h)
            n = bs.bs_cell_dims(h)[1]
            c = np.empty((n, n), np.complex128)
            bs.bs_reduced_matrix(h, np.array([0.21, -0.34]), c.view(np.float64))
        finally:
            bs.bs_destroy_cell(h)
        C.append(c.T[np.tril_indices(n)])   # column-major, the lower triangle is defined
    oc = mv.OracleCell(cell, M)
    kappa = np.linalg.cond(oc.Omega) * np.linalg.cond(oc.Phi)
    scale = np.abs(C[0]).max()
    d = np.abs(C[0] - C[1]).max()
    assert d <= 4 * n * EPS * kappa * scale, (d / scale, kappa)
