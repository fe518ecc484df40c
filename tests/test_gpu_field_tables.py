"""The two kernels that fill the phase table of bs_mode_field: many wavevectors take
the table of roots, one alone the direct evaluation.  Both are held to the
documented bound of the field, so they agree within twice that."""
import numpy as np
import pytest

from paper_1310_6380_gb300 import cells

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1310_6380_gb300 import binding as bs  # noqa: E402


@pytest.mark.parametrize("M, G, nk", [(0, 5, 1400), (2, 5, 700), (2, 64, 90), (7, 33, 80), (3, 256, 50),
                                      (15, 48, 40), (5, 1024, 30)])
def test_many_wavevectors_and_one(M, G, nk):
    cell = cells.voronoi_cell(48, 6, seed=4, lattice="hex")
    h = bs.bs_create_cell(cell.h1, cell.h2, np.ascontiguousarray(cell.phase, np.uint16),
                          cell.lam.copy(), cell.mu.copy(), cell.rho.copy(), M, bs.BS_PREC_FP64)
    N, W = (2 * M + 1) ** 2, (2 * M + 1 + 3) // 4 * 4
    assert nk * 2 * W * G >= 49152 + 512 * G
    rng = np.random.default_rng(G)
    Q = rng.uniform(-3.0, 3.0, (nk, 2))
    coef = rng.standard_normal((nk, 1, N)) + 1j * rng.standard_normal((nk, 1, N))
    out, one = np.empty((nk, 1, G, G), np.complex64), np.empty((1, 1, G, G), np.complex64)
    try:
        bs.bs_mode_field(h, Q, coef, G, out)
        for k in (0, nk // 2, nk - 1):
            bs.bs_mode_field(h, Q[k:k + 1].copy(), coef[k:k + 1].copy(), G, one)
            bound = (2 * (2 * M + 1) + 4) * 2.0 ** -24 * np.abs(coef[k]).sum()
            assert np.abs(out[k] - one[0]).max() <= 2 * bound
    finally:
        bs.bs_destroy_cell(h)
