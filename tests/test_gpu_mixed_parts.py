"""The FP32 reduction of the mixed path in parts on side streams: a matrix sees
the same operations in the same order whatever runs beside it.  Fifteen
wavevectors are reduced in one part, more of them in two (of unequal size), so
the first fifteen of a longer list, some of them in the second part, keep their
bits.  n = 1058 takes both forms of the step's last part."""
import numpy as np
import pytest

from paper_1310_6380_gb300 import cells

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1310_6380_gb300 import binding as bs  # noqa: E402


@pytest.mark.parametrize("M, nk", [(1, 40), (4, 17), (11, 19)])
def test_parts_do_not_change_a_matrix(M, nk):
    cell = cells.voronoi_cell(48, 9, seed=2)
    Q = cells.ibz_path(cell.lattice, nk, cell.h1, cell.h2)[:nk].copy()
    h = bs.bs_create_cell(cell.h1, cell.h2, np.ascontiguousarray(cell.phase, np.uint16),
                          cell.lam.copy(), cell.mu.copy(), cell.rho.copy(), M, bs.BS_PREC_MIXED)
    try:
        bs.bs_assemble(h)
        w, st = np.empty((nk, 4)), np.empty(nk, np.int32)
        bs.bs_solve_k(h, Q, 4, w, st)
        few, sf = np.empty((15, 4)), np.empty(15, np.int32)
        bs.bs_solve_k(h, Q[:15].copy(), 4, few, sf)
    finally:
        bs.bs_destroy_cell(h)
    assert np.array_equal(sf, st[:15]) and np.array_equal(few, w[:15])
