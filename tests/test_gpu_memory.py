"""The filtered iteration's workspace when the device is nearly full: smaller chunks
while one fits, the reductions when none does, and the same results."""
import numpy as np
import pytest

from paper_1310_6380_gb300 import cells

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1310_6380_gb300 import binding as bs  # noqa: E402


@pytest.mark.parametrize("left_mb, taken", [(600, 60), (24, 0)])
def test_little_memory(left_mb, taken):
    cell = cells.voronoi_cell(48, 12, seed=3)
    Q = np.ascontiguousarray(cells.ibz_path("square", 121, cell.h1, cell.h2)[1::2])
    h = bs.bs_create_cell(cell.h1, cell.h2, np.ascontiguousarray(cell.phase, np.uint16),
                          cell.lam.copy(), cell.mu.copy(), cell.rho.copy(), 7, bs.BS_PREC_FP64)
    hog = None
    try:
        bs.bs_assemble(h)
        ref, w, st = np.empty((60, 18)), np.empty((60, 18)), np.full(60, 7, np.int32)
        bs.bs_set_reduction(bs.BS_REDUCE_TWOSTAGE)      # n = 450: what AUTO falls back to
        bs.bs_solve_k(h, Q, 18, ref, st)                # allocates the cell's other workspace
        bs.bs_set_reduction(bs.BS_REDUCE_AUTO)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info()[0]
        hog = torch.empty(free - (left_mb << 20), dtype=torch.uint8, device="cuda")
        for _ in range(2):
            bs.bs_solve_k(h, Q, 18, w, st)
            assert not st.any()
            assert bs.bs_filter_counts(h) == (taken, 0)
            assert np.abs(w - ref).max() <= 1e-10 * ref.max()
    finally:
        bs.bs_set_reduction(bs.BS_REDUCE_AUTO)
        bs.bs_destroy_cell(h)
        del hog
        torch.cuda.empty_cache()
