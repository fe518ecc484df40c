"""Stress coefficients on exact-slice products and fields summed in conjugate row
pairs, at the sizes where the new paths change over.

A column of a product does not depend on the columns beside it: its digit sums
are exact integers and its scale is its own, so a wavevector alone and the same
one among enough of them to fill several column chunks give the same bits.
"""
import numpy as np
import pytest

from oracle import mode_shapes as ms
from paper_1310_6380_gb300 import cells

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1310_6380_gb300 import binding as bs  # noqa: E402

U32 = 2.0 ** -24


def make(cell, M):
    return bs.bs_create_cell(cell.h1, cell.h2, np.ascontiguousarray(cell.phase, np.uint16),
                             cell.lam.copy(), cell.mu.copy(), cell.rho.copy(), M, bs.BS_PREC_FP64)


# 2 x 180 x 12 = 4320 columns (three chunks, the last ragged) and one column
@pytest.mark.parametrize("M, nk, nvec", [(3, 180, 12), (2, 9, 5), (4, 3, 1)])
def test_stress_columns_are_independent(M, nk, nvec):
    h = make(cells.voronoi_cell(32, 6, seed=4), M)
    try:
        bs.bs_assemble(h)
        N, n = bs.bs_cell_dims(h)
        rng = np.random.default_rng(M)
        Q = rng.uniform(-0.5, 0.5, (nk, 2))
        U = rng.standard_normal((nk, nvec, n)) + 1j * rng.standard_normal((nk, nvec, n))
        S = np.empty((nk, nvec, 3 * N), np.complex128)
        bs.bs_stress_coefficients(h, Q, U, S)
        one = np.empty((1, 1, 3 * N), np.complex128)
        for k, j in ((0, 0), (nk // 2, nvec // 2), (nk - 1, nvec - 1)):
            bs.bs_stress_coefficients(h, Q[k:k + 1].copy(), U[k:k + 1, j:j + 1].copy(), one)
            assert np.array_equal(one[0, 0], S[k, j]), (k, j)
        # a mode that is not a number stays one, and the others do not change
        U[nk // 2, nvec // 2, n // 3] = np.nan
        U[0, 0, 0] = np.inf
        T = np.empty_like(S)
        bs.bs_stress_coefficients(h, Q, U, T)
    finally:
        bs.bs_destroy_cell(h)
    gone = ~np.isfinite(T).all(axis=2)
    assert gone[nk // 2, nvec // 2] and gone[0, 0] and gone.sum() == len({(nk // 2, nvec // 2),
                                                                          (0, 0)})
    assert np.array_equal(T[~gone], S[~gone])


# one row, one pair, an odd middle row, the last grid of the table of roots and
# the first beyond it; wavevectors outside the first zone
@pytest.mark.parametrize("G", [1, 2, 5, 1024, 1025])
def test_field_pairs_match_oracle(G):
    M = 2
    cell = cells.voronoi_cell(32, 6, seed=4, lattice="hex")
    h = make(cell, M)
    N = (2 * M + 1) ** 2
    rng = np.random.default_rng(G)
    Q = np.array([[0.0, 0.0], [0.31, -0.44], [-3.7, 12.2]])
    coef = rng.standard_normal((3, 1, N)) + 1j * rng.standard_normal((3, 1, N))
    out = np.empty((3, 1, G, G), np.complex64)
    try:
        bs.bs_mode_field(h, Q, coef, G, out)
    finally:
        bs.bs_destroy_cell(h)
    bound = (2 * (2 * M + 1) + 4) * U32 * np.abs(coef).sum(axis=-1)
    for i in range(3):
        ref = ms.field_on_grid(cell, M, Q[i], coef[i], G)
        assert (np.abs(out[i] - ref).max(axis=(1, 2)) <= bound[i]).all()
