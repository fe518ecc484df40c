"""The filtered subspace iteration behind BS_REDUCE_AUTO, against the
reductions to tridiagonal form of the same C(k) (themselves checked against
the oracle).

Tolerance on lambda = omega^2: the certificate allows 64 eps64 ||C||, a
Householder reduction and its bisection err by less than (n + 4) eps64 ||C||;
||C|| is at most the trace norm bound n max_r C_rr but is of the size of
max_r C_rr for these matrices, so (n + 128) eps64 max_r C_rr.
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


@pytest.fixture(autouse=True)
def restore_reduction():
    yield
    bs.bs_set_reduction(bs.BS_REDUCE_AUTO)


def solve2(cell, M, Q, nb):
    """omega of the filtered iteration and of the one-stage reduction, max C_rr."""
    h = bs.bs_create_cell(cell.h1, cell.h2, np.ascontiguousarray(cell.phase, np.uint16),
                          cell.lam.copy(), cell.mu.copy(), cell.rho.copy(), M, bs.BS_PREC_FP64)
    try:
        bs.bs_assemble(h)
        n = bs.bs_cell_dims(h)[1]
        out = []
        for mode in (bs.BS_REDUCE_AUTO, bs.BS_REDUCE_ONESTAGE):
            bs.bs_set_reduction(mode)
            w = np.empty((len(Q), nb))
            st = np.full(len(Q), 7, np.int32)
            bs.bs_solve_k(h, Q, nb, w, st)
            assert not st.any()
            out.append(w)
        C = np.empty((n, n), np.complex128)
        bs.bs_reduced_matrix(h, Q[-1].copy(), C.view(np.float64))
    finally:
        bs.bs_destroy_cell(h)
    return out[0], out[1], n, np.abs(C.diagonal()).max()


CASES = [
    # name, cell, M, nbands, wavevectors: n = 242, 338, 450, 578, 722, 882 are
    # ragged against the 64-wide tiles; 1 and 22 branches (the most guard
    # vectors, and the fewest); Gamma and the corners; exact degeneracies
    ("one_branch", lambda: cells.voronoi_cell(32, 5, seed=1), 5, 1, 3),
    ("most_branches", lambda: cells.voronoi_cell(32, 9, seed=2, lattice="hex"), 5, 22, 9),
    ("one_k", lambda: cells.circle_cell(32, 0.3), 6, 8, 1),
    ("circle_symmetric", lambda: cells.circle_cell(32, 0.3), 7, 18, 13),
    ("homogeneous", lambda: cells.homogeneous_cell(32), 5, 18, 13),
    ("si_units", lambda: cells.steel_epoxy_hex_cell(48), 6, 12, 10),
    ("m8", lambda: cells.ellipse_cell(64, 7, seed=3), 8, 10, 5),
    ("m9", lambda: cells.voronoi_cell(64, 40, seed=4), 9, 17, 4),
    ("m10", lambda: cells.voronoi_cell(64, 200, seed=5), 10, 18, 7),
]


@pytest.mark.parametrize("name,make,M,nb,nk", CASES, ids=[c[0] for c in CASES])
def test_matches_the_one_stage_reduction(name, make, M, nb, nk):
    cell = make()
    Q = cells.ibz_path(cell.lattice, max(nk, 2), cell.h1, cell.h2)[:nk].copy()
    a, b, n, cmax = solve2(cell, M, Q, nb)
    assert np.abs(a ** 2 - b ** 2).max() <= (n + 128) * EPS * cmax


def test_uncertified_matrices_are_reduced():
    """A homogeneous 3-D cell at Gamma has 24 equal eigenvalues from the 22nd
    on: no cut above the 22nd branch lies in the block, so that matrix takes
    the reduction behind the iteration; the generic wavevectors beside it do
    not have to."""
    P = 6
    h = np.eye(3)
    mu, lam, rho = 1.0, -0.6, 1.0
    Q = np.array([[0.0, 0.0, 0.0], [0.13, 0.29, 0.41], [0.0, 0.0, 0.0], [0.31, 0.07, 0.22]])
    hd = bs.bs_create_cell3(h[0], h[1], h[2], np.zeros((P, P, P), np.uint16), np.array([lam]),
                            np.array([mu]), np.array([rho]), 2)
    try:
        bs.bs_assemble3(hd)
        w = np.empty((4, 22))
        st = np.full(4, 7, np.int32)
        bs.bs_solve_k3(hd, Q, 22, w, st)
    finally:
        bs.bs_destroy_cell3(hd)
    assert not st.any()
    r = np.arange(-2, 3)
    g = np.stack(np.meshgrid(r, r, r, indexing="ij"), -1).reshape(-1, 3)
    for q, got in zip(Q, w):
        k2 = (2 * np.pi) ** 2 * np.sum((g + q) ** 2, 1)
        lam_exact = np.sort(np.concatenate([k2 * (lam + 2 * mu), k2 * mu, k2 * mu]) / rho)
        # formation of C(k) from its monomials adds a few eps of max |K|^2 per entry
        assert np.abs(got ** 2 - lam_exact[:22]).max() <= (375 + 128) * EPS * lam_exact[-1]


def test_batch_fp64_solver():
    cl = [cells.config3_cell(i) for i in (0, 3, 5, 8)]
    args = [(c["cell"].h1, c["cell"].h2, np.ascontiguousarray(c["cell"].phase, np.uint16),
             c["cell"].lam, c["cell"].mu, c["cell"].rho, c["M"], bs.BS_PREC_MIXED) for c in cl]
    Q = np.stack([c["Q"][:6] for c in cl])
    b = bs.bs_batch_create(args, 6, 10)
    try:
        bs.bs_batch_set_solver(b, bs.BS_SOLVER_FP64)
        w = np.empty((4, 6, 10))
        st = np.full((4, 6), 7, np.int32)
        bs.bs_batch_solve(b, Q, w, st)
    finally:
        bs.bs_batch_destroy(b)
    assert not st.any()
    for i, c in enumerate(cl):
        _, ref, n, cmax = solve2(c["cell"], c["M"], np.ascontiguousarray(Q[i]), 10)
        assert np.abs(w[i] ** 2 - ref ** 2).max() <= (n + 128) * EPS * cmax


@pytest.mark.parametrize("M,nb,nk", [(3, 1, 1), (3, 22, 40), (3, 9, 13), (4, 22, 1), (4, 10, 25)])
def test_smallest_matrices(M, nb, nk):
    """n = 98 and 162, the smallest that take the iteration (two and three tiles)."""
    for cell in (cells.circle_cell(32, 0.3), cells.voronoi_cell(32, 9, seed=2, lattice="hex")):
        Q = cells.ibz_path(cell.lattice, max(nk, 2), cell.h1, cell.h2)[:nk].copy()
        a, b, n, cmax = solve2(cell, M, Q, nb)
        assert np.abs(a ** 2 - b ** 2).max() <= (n + 128) * EPS * cmax


def test_many_matrices():
    """2160 matrices of 24 cells: among so many the FP32 count of one or two is
    spoilt by a pivot near zero and taken again at the second shift."""
    for seed in range(24):
        cell = cells.voronoi_cell(32, 12, seed=seed, lattice="hex" if seed % 2 else "square")
        Q = cells.ibz_path(cell.lattice, 90, cell.h1, cell.h2)[:90].copy()
        a, b, n, cmax = solve2(cell, 5, Q, 18)
        assert np.abs(a ** 2 - b ** 2).max() <= (n + 128) * EPS * cmax, seed


def test_batch_dense_solver():
    """The dense batch solver's groups take the iteration on their FP64 C(k)."""
    cl = [cells.config3_cell(i) for i in (0, 3, 5, 8)]
    args = [(c["cell"].h1, c["cell"].h2, np.ascontiguousarray(c["cell"].phase, np.uint16),
             c["cell"].lam, c["cell"].mu, c["cell"].rho, c["M"], bs.BS_PREC_MIXED) for c in cl]
    Q = np.stack([c["Q"][:6] for c in cl])
    b = bs.bs_batch_create(args, 6, 10)
    try:
        w, st = np.empty((4, 6, 10)), np.full((4, 6), 7, np.int32)
        bs.bs_batch_solve(b, Q, w, st)
    finally:
        bs.bs_batch_destroy(b)
    assert not st.any()
    for i, c in enumerate(cl):
        _, ref, n, cmax = solve2(c["cell"], c["M"], np.ascontiguousarray(Q[i]), 10)
        assert np.abs(w[i] ** 2 - ref ** 2).max() <= (n + 128) * EPS * cmax
