"""bs_set_reduction takes effect at the next bs_batch_solve, and a solve keeps to
one mode whatever another thread sets meanwhile.

Tolerance on lambda as in test_gpu_filter.py: (n + 128) eps64 max C_rr between two
FP64 routes; the dense solver's FP32 reduction with its refinement is held to its
documented residual bound, 1e-6 of omega.
"""
import threading

import numpy as np
import pytest

from paper_1310_6380_gb300 import cells

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1310_6380_gb300 import binding as bs  # noqa: E402

EPS = np.finfo(float).eps
NK, NB = 6, 10


@pytest.fixture(autouse=True)
def restore_reduction():
    yield
    bs.bs_set_reduction(bs.BS_REDUCE_AUTO)


def batch(solver):
    cl = [cells.config3_cell(i) for i in (0, 3, 5, 8)]
    args = [(c["cell"].h1, c["cell"].h2, np.ascontiguousarray(c["cell"].phase, np.uint16),
             c["cell"].lam, c["cell"].mu, c["cell"].rho, c["M"], bs.BS_PREC_MIXED) for c in cl]
    # (generic wavevectors: at Gamma omega is the root of a rounding error)
    Q = np.random.default_rng(1).uniform(0.05, 0.45, (4, NK, 2))
    b = bs.bs_batch_create(args, NK, NB)
    bs.bs_batch_set_solver(b, solver)
    return b, Q


def run(b, Q):
    w, st = np.empty((4, NK, NB)), np.full((4, NK), 7, np.int32)
    bs.bs_batch_solve(b, Q, w, st)
    assert not st.any()
    return w


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("mode", [bs.BS_REDUCE_ONESTAGE, bs.BS_REDUCE_TWOSTAGE])
@pytest.mark.parametrize("solver", [bs.BS_SOLVER_FP64, bs.BS_SOLVER_DENSE])
def test_mode_takes_effect_at_the_next_solve(solver, mode, graph):
    b, Q = batch(solver)
    try:
        bs.bs_batch_set_graph(b, graph)
        auto = run(b, Q)
        assert bs.bs_batch_filter_counts(b) == (4 * NK, 0)
        run(b, Q)
        bs.bs_set_reduction(mode)
        forced = run(b, Q)
        assert bs.bs_batch_filter_counts(b) == (0, 0)
        again = run(b, Q)
        bs.bs_set_reduction(bs.BS_REDUCE_AUTO)
        back = run(b, Q)
        assert bs.bs_batch_filter_counts(b) == (4 * NK, 0)
    finally:
        bs.bs_batch_destroy(b)
    assert np.array_equal(auto, back)
    assert np.array_equal(forced, again)
    # a batch that never knew another mode
    bs.bs_set_reduction(mode)
    b, Q = batch(solver)
    try:
        bs.bs_batch_set_graph(b, graph)
        fresh = run(b, Q)
    finally:
        bs.bs_batch_destroy(b)
    tol = 1e-6 if solver == bs.BS_SOLVER_DENSE else 1e-11
    assert np.abs(forced - fresh).max() <= tol * fresh.max()
    assert np.abs(forced - auto).max() <= tol * auto.max()


@pytest.mark.parametrize("solver", [bs.BS_SOLVER_FP64, bs.BS_SOLVER_DENSE])
def test_mode_changed_by_another_thread(solver):
    b, Q = batch(solver)
    stop = threading.Event()

    def toggle():
        modes = [bs.BS_REDUCE_ONESTAGE, bs.BS_REDUCE_AUTO]
        i = 0
        while not stop.is_set():
            bs.bs_set_reduction(modes[i & 1])
            i += 1

    t = threading.Thread(target=toggle)
    try:
        ref = run(b, Q)
        t.start()
        for _ in range(40):
            w = run(b, Q)
            # each group went one way as a whole: none of its matrices was reduced
            # because it had been built for the other
            taken, reduced = bs.bs_batch_filter_counts(b)
            assert reduced == 0
            assert np.abs(w - ref).max() <= 1e-6 * ref.max()
    finally:
        stop.set()
        t.join()
        bs.bs_batch_destroy(b)
