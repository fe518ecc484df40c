"""A tensor-core wait that reaches its limit inside bs_stress_coefficients: the call
reports it or, on device arrays, bs_sync does; the result is NaN, and the next
call does not know of it.  The flag is set from the host (bs_set_late_wait)."""
import numpy as np
import pytest

from paper_1310_6380_gb300 import cells

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1310_6380_gb300 import binding as bs  # noqa: E402


@pytest.mark.parametrize("on_device", [False, True])
def test_late_wait(on_device):
    cell = cells.voronoi_cell(32, 6, seed=4)
    h = bs.bs_create_cell(cell.h1, cell.h2, np.ascontiguousarray(cell.phase, np.uint16),
                          cell.lam.copy(), cell.mu.copy(), cell.rho.copy(), 3, bs.BS_PREC_FP64)
    try:
        bs.bs_assemble(h)
        N, n = bs.bs_cell_dims(h)
        rng = np.random.default_rng(0)
        Q = rng.uniform(-0.5, 0.5, (4, 2))
        U = rng.standard_normal((4, 3, n)) + 1j * rng.standard_normal((4, 3, n))
        if on_device:
            Qd, Ud = torch.from_numpy(Q).cuda(), torch.from_numpy(U).cuda()
            S = torch.empty((4, 3, 3 * N), dtype=torch.complex128, device="cuda")
            call = lambda: bs.bs_stress_coefficients(h, Qd, Ud, S)
            result = lambda: S.cpu().numpy().copy()
        else:
            S = np.empty((4, 3, 3 * N), np.complex128)
            call = lambda: bs.bs_stress_coefficients(h, Q, U, S)
            result = lambda: S.copy()
        call()
        good = result()
        assert np.isfinite(good).all()
        bs.bs_set_late_wait(h, True)
        if on_device:
            call()
            assert np.isnan(result()).all()
            with pytest.raises(bs.BSError) as ei:
                bs.bs_sync(h)
        else:
            with pytest.raises(bs.BSError) as ei:
                call()
            assert np.isnan(result()).all()
        assert ei.value.code == bs.BS_ECUDA
        bs.bs_set_late_wait(h, False)
        call()
        assert np.array_equal(result(), good)
        bs.bs_sync(h)
    finally:
        bs.bs_destroy_cell(h)
