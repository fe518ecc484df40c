"""Cells whose materials lie far apart, on the route that BS_REDUCE_AUTO gives them:
the filtered iteration certifies what it takes, and what it would not certify
goes to the reductions at once.

Tolerance on lambda: the certificate allows 64 eps64 max C_rr, a reduction and its
bisection err by less than (n + 4) eps64 ||C||, as in test_gpu_filter.py.
"""
import numpy as np
import pytest

from paper_1310_6380_gb300 import cells

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1310_6380_gb300 import binding as bs  # noqa: E402

EPS = np.finfo(float).eps
MATRIX = np.array([4.0, 1.5, 1.2])


def circle(contrast, density=1.0, r=0.3, P=48):
    """A circular inclusion of `contrast` times the matrix's moduli."""
    return cells.circle_cell(P, r, tuple(MATRIX), tuple(MATRIX * [contrast, contrast, density]))


def path(cell, nk):
    return np.ascontiguousarray(cells.ibz_path(cell.lattice, 2 * nk + 1, cell.h1, cell.h2)[1::2])


def args(cell, M, precision=bs.BS_PREC_FP64):
    return (cell.h1, cell.h2, np.ascontiguousarray(cell.phase, np.uint16), cell.lam.copy(),
            cell.mu.copy(), cell.rho.copy(), M, precision)


def solve(cell, M, Q, nb):
    """omega under BS_REDUCE_AUTO and one-stage, the counts of the first, n, max C_rr."""
    h = bs.bs_create_cell(*args(cell, M))
    try:
        bs.bs_assemble(h)
        n = bs.bs_cell_dims(h)[1]
        out, counts = [], []
        for mode in (bs.BS_REDUCE_AUTO, bs.BS_REDUCE_ONESTAGE):
            bs.bs_set_reduction(mode)
            w, st = np.empty((len(Q), nb)), np.full(len(Q), 7, np.int32)
            bs.bs_solve_k(h, Q, nb, w, st)
            assert not st.any()
            out.append(w)
            counts.append(bs.bs_filter_counts(h))
        C = np.empty((n, n), np.complex128)
        bs.bs_reduced_matrix(h, Q[0].copy(), C.view(np.float64))
    finally:
        bs.bs_set_reduction(bs.BS_REDUCE_AUTO)
        bs.bs_destroy_cell(h)
    assert counts[1] == (0, 0)
    return out[0], out[1], counts[0], n, np.abs(C.diagonal()).max()


# soft and stiff, light and heavy inclusions; n = 98, 242, 338 and 450
@pytest.mark.parametrize("M", [3, 5, 6, 7])
@pytest.mark.parametrize("contrast, density", [(0.02, 1.0), (0.01, 1.0), (0.1, 5.0), (30.0, 1.0),
                                               (100.0, 1.0), (50.0, 7.0), (1.0, 30.0), (1.0, 0.05)])
def test_moderate_contrast_is_certified(contrast, density, M):
    cell = circle(contrast, density)
    Q = path(cell, 12)
    a, b, counts, n, cmax = solve(cell, M, Q, 12)
    assert np.abs(a ** 2 - b ** 2).max() <= (n + 128) * EPS * cmax
    assert counts == (12, 0)


@pytest.mark.parametrize("M, nb", [(5, 18), (7, 8)])
@pytest.mark.parametrize("contrast, density", [(1e-4, 1.0), (1e-3, 1.0), (3e3, 1.0), (1e4, 1.0),
                                               (1.0, 3e3)])
def test_extreme_contrast_takes_the_reductions(contrast, density, M, nb):
    cell = circle(contrast, density)
    Q = path(cell, 6)
    a, b, counts, n, cmax = solve(cell, M, Q, nb)
    assert np.abs(a ** 2 - b ** 2).max() <= (n + 128) * EPS * cmax
    assert counts == (0, 0)


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("solver", [bs.BS_SOLVER_FP64, bs.BS_SOLVER_DENSE])
def test_batch_groups(solver, graph):
    """A group with few extreme cells takes the iteration, the reduction behind it
    solves theirs (also in a replayed graph); one with many takes the reductions."""
    few = [circle(c, P=32) for c in (20, 1e4, 0.1, 30, 5, 10, 0.05, 15)]
    many = [circle(c, P=32) for c in (20, 1e4, 1e-3, 30, 3e-4, 10, 0.05, 15)]
    for group, want in ((few, 8 * 6), (many, 0)):
        Q = np.stack([path(c, 6) for c in group])
        b = bs.bs_batch_create([args(c, 5, bs.BS_PREC_MIXED) for c in group], 6, 18)
        try:
            bs.bs_batch_set_solver(b, solver)
            bs.bs_batch_set_graph(b, graph)
            for _ in range(3 if graph else 1):
                w, st = np.empty((8, 6, 18)), np.full((8, 6), 7, np.int32)
                bs.bs_batch_solve(b, Q, w, st)
                taken, reduced = bs.bs_batch_filter_counts(b)
                assert taken == want and reduced <= want // 8 and not st.any()
        finally:
            bs.bs_batch_destroy(b)
        if solver == bs.BS_SOLVER_FP64 or want:
            for i, c in enumerate(group):
                _, ref, _, n, cmax = solve(c, 5, Q[i], 18)
                assert np.abs(w[i] ** 2 - ref ** 2).max() <= (n + 128) * EPS * cmax


def test_three_dimensions():
    cell = cells.sphere_cell3(16, 0.3, tuple(MATRIX), tuple(MATRIX * [1e4, 1e4, 1.0]))
    soft = cells.sphere_cell3(16, 0.3, tuple(MATRIX), tuple(MATRIX * [0.05, 0.05, 1.0]))
    Q = np.ascontiguousarray(cells.ibz_path_cubic(13)[1::2])
    for c, want in ((cell, (0, 0)), (soft, (6, 0))):
        h = bs.bs_create_cell3(c.h1, c.h2, c.h3, np.ascontiguousarray(c.phase, np.uint16), c.lam.copy(),
                               c.mu.copy(), c.rho.copy(), 2)
        try:
            bs.bs_assemble3(h)
            st = np.full(6, 7, np.int32)
            bs.bs_solve_k3(h, Q, 12, np.empty((6, 12)), st)
            assert not st.any()
            assert bs.bs_filter_counts3(h) == want
        finally:
            bs.bs_destroy_cell3(h)


def test_anisotropic_phases_count_as_their_tensors():
    """The spread of a cell given as stiffness tensors is that of the same cell
    given as moduli."""
    for contrast, want in ((100.0, (6, 0)), (1e4, (0, 0))):
        cell = circle(contrast)
        Q = path(cell, 6)
        h = bs.bs_create_cell(*args(cell, 5))
        try:
            C = cells.isotropic_stiffness(cell.lam, cell.mu)
            bs.bs_set_stiffness(h, np.ascontiguousarray(np.stack(
                [C[:, 0, 0], C[:, 1, 1], C[:, 0, 1], C[:, 0, 2], C[:, 1, 2], C[:, 2, 2]], axis=1)))
            bs.bs_assemble(h)
            st = np.full(6, 7, np.int32)
            bs.bs_solve_k(h, Q, 10, np.empty((6, 10)), st)
            assert not st.any()
            assert bs.bs_filter_counts(h) == want
        finally:
            bs.bs_destroy_cell(h)
