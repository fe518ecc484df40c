"""What a user of the library has it do, as a list of cases.

Each case is one call sequence through the public entry points
(paper_1310_6380_gb300.binding) at sizes taken from the repository's own
configurations: the band structure of one cell on the FP64 path (isotropic
pixel cell, triangle mesh, anisotropic phases, 3-D voxels), on the mixed
path, ragged batches of cells on the three batch solvers, mode shapes, and
the warm-start network's training step.  listed() holds the configurations
themselves, draw() more of the same ranges.

The wavevectors are the midpoints of equal arcs of the closed IBZ boundary
(a path sampled without its ends): exactly at Gamma the two or three
acoustic frequencies are the square roots of rounding errors, which no
comparison can use.
"""
from __future__ import annotations

import math
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

from paper_1310_6380_gb300 import binding as bs
from paper_1310_6380_gb300 import cells, warmstart

NET_MP, NET_NVEC = 3, 12     # the shipped network: 12 vectors of the waves |alpha|, |beta| <= 3


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # one wavevector of an assembled small cell: the inner call of a root
        # search or an optimiser that walks k; only latency counts
        dict(name="one_k", kind="solve", cell="circle", P=32, nphase=2, lattice="square", M=3, nk=1,
             nbands=8, assemble=False),
        # the small band structure (32 x 32 circle, 30 k, 8 branches)
        dict(name="circle_m3", kind="solve", cell="circle", P=32, nphase=2, lattice="square", M=3,
             nk=30, nbands=8, assemble=True),
        # the benchmark's configuration: 1132-phase Voronoi cell, M = 10, 90 k
        # on the square path, 18 branches, FP64
        dict(name="voronoi_m10", kind="solve", cell="voronoi", P=256, nphase=1132, lattice="square",
             M=10, nk=90, nbands=18, assemble=True),
        # the same on the mixed path
        dict(name="voronoi_m10_mixed", kind="mixed", cell="voronoi", P=256, nphase=1132,
             lattice="square", M=10, nk=90, nbands=18, assemble=True),
        # the paper's workload shape: hexagonal steel/epoxy cell on a
        # 968-element mesh, M = 5, 70 k, 18 branches, FP64
        dict(name="mesh_hex_m5", kind="mesh", n=22, lattice="hex", M=5, nk=70, nbands=18),
        # rotated orthotropic phases (the full compliance Gram matrix)
        dict(name="aniso_m10", kind="aniso", cell="voronoi", P=256, nphase=1132, lattice="square",
             M=10, nk=90, nbands=18),
        # 3-D: spherical inclusion, 32^3 voxels, M = 3, 30 k, 12 branches
        dict(name="sphere3d_m3", kind="cell3", P=32, M=3, nk=30, nbands=12),
        # ragged batches of 64 x 64 cells (M = 5..8, 30 k, 10 branches): dense
        # mixed, plain FP64, and LOBPCG started from the network
        dict(name="batch_dense", kind="batch", solver="dense", ncells=48, nk=30, nbands=10),
        dict(name="batch_fp64", kind="batch", solver="fp64", ncells=24, nk=30, nbands=10),
        dict(name="batch_lobpcg", kind="batch", solver="lobpcg", ncells=48, nk=30, nbands=10),
        # stress coefficients and both fields of 12 modes at 90 k on the
        # 256 x 256 pixel centres of the M = 10 cell
        dict(name="modes_m10", kind="modes", cell="voronoi", P=256, nphase=1132, lattice="square",
             M=10, nk=90, nvec=12, G=256),
        # forward, loss and backward of the warm-start network (the training
        # minibatch: 64 cells x 4 k)
        dict(name="net_train", kind="net", ncells=64, kper=4, nb=10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "mixed", "mesh", "aniso", "cell3", "batch", "modes",
                       "net"])
    lattice = rng.choice(["square", "hex"])
    if kind in ("solve", "mixed", "aniso"):
        M = rng.randint(2, 10)
        c = rng.choice(["circle", "ellipse", "voronoi"])
        P = rng.randint(max(24, 2 * M + 1), 256)
        nph = 2 if c == "circle" else _log(rng, 2, 16 if c == "ellipse" else 1132)
        nk, nb = _log(rng, 1, 90), rng.randint(4, 18)
        case = dict(kind=kind, cell=c, P=P, nphase=nph, lattice=lattice, M=M, nk=nk, nbands=nb)
        if kind != "aniso":
            case["assemble"] = True
        return case
    if kind == "mesh":
        return dict(kind=kind, n=rng.randint(18, 30), lattice=lattice, M=rng.randint(2, 6),
                    nk=_log(rng, 2, 70), nbands=rng.randint(4, 18))
    if kind == "cell3":
        return dict(kind=kind, P=rng.randint(8, 32), M=rng.randint(1, 3), nk=_log(rng, 1, 30),
                    nbands=rng.randint(4, 12))
    if kind == "batch":
        solver = rng.choice(["dense", "fp64", "lobpcg"])
        return dict(kind=kind, solver=solver, ncells=_log(rng, 2, 20 if solver == "fp64" else 40),
                    nk=rng.randint(5, 30), nbands=rng.randint(4, 10))
    if kind == "modes":
        return dict(kind=kind, cell="voronoi", P=rng.randint(64, 256), nphase=_log(rng, 2, 1132),
                    lattice=lattice, M=rng.randint(3, 10), nk=_log(rng, 1, 90),
                    nvec=rng.randint(1, 12), G=rng.randint(17, 256))
    return dict(kind="net", ncells=_log(rng, 2, 64), kper=rng.randint(1, 4), nb=rng.randint(4, 10))


# ------------------------------------------------------------------ inputs
def _path(lattice, nk, h1, h2):
    """nk wavevectors at the midpoints of nk equal arcs of the IBZ boundary."""
    q = cells.ibz_path(lattice, 2 * nk + 1, h1, h2)
    return np.ascontiguousarray(q[1::2])


def _cell(case, seed):
    rng = np.random.default_rng(seed)
    kind, P, lattice, nph = case["cell"], case["P"], case["lattice"], case["nphase"]
    if kind == "circle":
        # a soft matrix with a stiff heavy inclusion, within 20 % of (4, 1.5, 1.2) / (110, 80, 7.8)
        f = rng.uniform(0.8, 1.2, 6)
        c = cells.circle_cell(P, rng.uniform(0.2, 0.4),
                              tuple(np.array([4.0, 1.5, 1.2]) * f[:3]),
                              tuple(np.array([110.0, 80.0, 7.8]) * f[3:]), lattice)
    elif kind == "ellipse":
        c = cells.ellipse_cell(P, nph - 1, int(rng.integers(1 << 30)), lattice)
    else:
        c = cells.voronoi_cell(P, nph, int(rng.integers(1 << 30)), lattice)
    if case["kind"] == "aniso":
        c = cells.anisotropic_cell(c, int(rng.integers(1 << 30)))
    return c


def _mesh(case, seed):
    rng = np.random.default_rng(seed)
    a = 6.023e-3             # steel cylinders in epoxy, SI units
    f = rng.uniform(0.9, 1.1, 6)
    steel = np.array([264e9 - 2 * 81e9, 81e9, 7780.0]) * f[:3]
    epoxy = np.array([7.54e9 - 2 * 1.48e9, 1.48e9, 1142.0]) * f[3:]
    return cells.mesh_circle_cell(case["n"], rng.uniform(0.25, 0.4), tuple(epoxy), tuple(steel),
                                  case["lattice"], a, seed=int(rng.integers(1 << 30)))


def _cell3(case, seed):
    rng = np.random.default_rng(seed)
    f = rng.uniform(0.8, 1.2, 6)
    return cells.sphere_cell3(case["P"], rng.uniform(0.2, 0.4),
                              tuple(np.array([4.0, 1.5, 1.2]) * f[:3]),
                              tuple(np.array([110.0, 80.0, 7.8]) * f[3:]))


def _path3(nk):
    return np.ascontiguousarray(cells.ibz_path_cubic(2 * nk + 1)[1::2])


def _batch(case, seed):
    """Cells of the ragged batch's generator, and their wavevectors."""
    cs = [cells.c3_style_cell(3_000_000 + 1000 * (seed % 100_000) + i) for i in range(case["ncells"])]
    Q = np.stack([_path(c["cell"].lattice, case["nk"], c["cell"].h1, c["cell"].h2) for c in cs])
    return [c["cell"] for c in cs], [c["M"] for c in cs], Q


def _waves(M):
    r = np.arange(-M, M + 1)
    return np.repeat(r, 2 * M + 1), np.tile(r, 2 * M + 1)


def _modes(case, seed):
    """Displacement coefficients that fall off with the wave number, as those
    of the lowest branches do: (nk, nvec, 2N) complex128."""
    rng = np.random.default_rng(seed + 1)
    al, be = _waves(case["M"])
    N = len(al)
    fall = 1.0 / (1.0 + np.tile(al ** 2 + be ** 2, 2)) ** 1.5
    shape = (case["nk"], case["nvec"], 2 * N)
    u = (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) * fall
    return np.ascontiguousarray(u / np.linalg.norm(u, axis=-1, keepdims=True))


def _net(case, seed):
    """A minibatch of training cells, the initial parameters and targets."""
    rng = np.random.default_rng(seed + 2)
    cl = [cells.c3_style_cell(4_000_000 + 1000 * (seed % 100_000) + i) for i in range(case["ncells"])]
    pack = warmstart.CellPack([c["cell"] for c in cl])
    Q = np.stack([c["Q"][rng.choice(30, case["kper"], replace=False)] for c in cl])
    p = warmstart.init_params(NET_NVEC, NET_MP, int(rng.integers(1 << 30)))
    L = 2 * (2 * NET_MP + 1) ** 2
    al, be = _waves(NET_MP)
    shape = (case["ncells"] * case["kper"], case["nb"], L)
    v = (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) / (1.0 + np.tile(al ** 2 + be ** 2, 2))
    v /= np.linalg.norm(v, axis=-1, keepdims=True)
    return pack, np.ascontiguousarray(Q.reshape(-1, 2)), p, np.ascontiguousarray(v, np.complex64)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


class State:
    """What a program keeps between calls: handles, device inputs, output buffers."""

    def __init__(self):
        self.free = []

    def __del__(self):
        for f, h in self.free:
            f(h)


def _params_of_shipped_net():
    import os
    path = os.path.join(os.path.dirname(os.path.abspath(warmstart.__file__)), "data", "warmstart.npz")
    with np.load(path) as z:
        return np.ascontiguousarray(z["params"], np.float32)


def prepare(case, seed):
    s = State()
    kind = s.kind = case["kind"]
    if kind in ("solve", "mixed", "aniso", "modes"):
        c = _cell(case, seed)
        s.h = bs.bs_create_cell(c.h1, c.h2, _dev(c.phase.astype(np.uint16)), _dev(c.lam), _dev(c.mu),
                                _dev(c.rho), case["M"],
                                bs.BS_PREC_MIXED if kind == "mixed" else bs.BS_PREC_FP64)
        s.free.append((bs.bs_destroy_cell, s.h))
        if kind == "aniso":
            C = c.stiffness
            bs.bs_set_stiffness(s.h, _dev(np.stack([C[:, 0, 0], C[:, 1, 1], C[:, 0, 1], C[:, 0, 2],
                                                    C[:, 1, 2], C[:, 2, 2]], axis=1)))
        s.Q = _dev(_path(case["lattice"], case["nk"], c.h1, c.h2))
    if kind == "mesh":
        c = _mesh(case, seed)
        s.h = bs.bs_create_cell_mesh(c.h1, c.h2, _dev(c.centroid), _dev(c.area),
                                     _dev(c.phase.astype(np.uint16)), _dev(c.lam), _dev(c.mu),
                                     _dev(c.rho), case["M"])
        s.free.append((bs.bs_destroy_cell, s.h))
        s.Q = _dev(_path(case["lattice"], case["nk"], c.h1, c.h2))
    if kind == "cell3":
        c = _cell3(case, seed)
        s.h = bs.bs_create_cell3(c.h1, c.h2, c.h3, _dev(c.phase), _dev(c.lam), _dev(c.mu), _dev(c.rho),
                                 case["M"])
        s.free.append((bs.bs_destroy_cell3, s.h))
        s.Q = _dev(_path3(case["nk"]))
    if kind in ("solve", "mixed", "aniso", "mesh", "cell3"):
        s.nbands = case["nbands"]
        s.w = torch.empty((case["nk"], case["nbands"]), dtype=torch.float64, device="cuda")
        s.st = torch.empty(case["nk"], dtype=torch.int32, device="cuda")
        s.assemble = case.get("assemble", True)
        if not s.assemble:
            bs.bs_assemble(s.h, torch.cuda.current_stream())
    if kind == "batch":
        cl, Ms, Q = _batch(case, seed)
        s.h = bs.bs_batch_create([(c.h1, c.h2, np.ascontiguousarray(c.phase, np.uint16), c.lam, c.mu,
                                   c.rho, M, bs.BS_PREC_MIXED) for c, M in zip(cl, Ms)],
                                 case["nk"], case["nbands"])
        s.free.append((bs.bs_batch_destroy, s.h))
        s.lob = case["solver"] == "lobpcg"
        bs.bs_batch_set_solver(s.h, {"dense": bs.BS_SOLVER_DENSE, "fp64": bs.BS_SOLVER_FP64,
                                     "lobpcg": bs.BS_SOLVER_LOBPCG}[case["solver"]])
        s.Q = _dev(Q)
        s.w = torch.empty((case["ncells"], case["nk"], case["nbands"]), dtype=torch.float64,
                          device="cuda")
        s.st = torch.empty((case["ncells"], case["nk"]), dtype=torch.int32, device="cuda")
        if s.lob:
            s.net = bs.bs_cnn_create(NET_NVEC, NET_MP, case["ncells"], case["ncells"] * case["nk"])
            s.free.append((bs.bs_cnn_destroy, s.net))
            bs.bs_cnn_set_params(s.net, _params_of_shipped_net())
            p = warmstart.CellPack(cl)
            s.inputs = [_dev(a) for a in (p.phase, p.table, p.toff, p.nph, p.hexflag)]
            s.kper = case["nk"]
            s.U = torch.empty((case["ncells"], case["nk"], NET_NVEC, 2 * (2 * NET_MP + 1) ** 2),
                              dtype=torch.complex64, device="cuda")
    if kind == "modes":
        bs.bs_assemble(s.h, torch.cuda.current_stream())
        U, G, N = _modes(case, seed), case["G"], (2 * case["M"] + 1) ** 2
        s.U, s.G, s.N = _dev(U), G, N
        s.S = torch.empty((case["nk"], case["nvec"], 3 * N), dtype=torch.complex128, device="cuda")
        s.fu = torch.empty((case["nk"], 2 * case["nvec"], G, G), dtype=torch.complex64, device="cuda")
        s.fs = torch.empty((case["nk"], 3 * case["nvec"], G, G), dtype=torch.complex64, device="cuda")
    if kind == "net":
        pack, Q, p, V = _net(case, seed)
        s.net = bs.bs_cnn_create(NET_NVEC, NET_MP, case["ncells"], len(Q))
        s.free.append((bs.bs_cnn_destroy, s.net))
        bs.bs_cnn_set_params(s.net, p)
        s.inputs = [_dev(a) for a in (pack.phase, pack.table, pack.toff, pack.nph, pack.hexflag)]
        s.Q, s.V, s.kper = _dev(Q), _dev(V), case["kper"]
        s.loss = torch.empty(len(Q), dtype=torch.float32, device="cuda")
        s.grad = torch.empty(len(p), dtype=torch.float32, device="cuda")
    return s


def run(s):
    stream = torch.cuda.current_stream()
    if s.kind in ("solve", "mixed", "aniso", "mesh"):
        if s.assemble:
            bs.bs_assemble(s.h, stream)
        bs.bs_solve_k(s.h, s.Q, s.nbands, s.w, s.st, stream)
        return {"omega": s.w, "status": s.st}
    if s.kind == "cell3":
        bs.bs_assemble3(s.h, stream)
        bs.bs_solve_k3(s.h, s.Q, s.nbands, s.w, s.st, stream)
        return {"omega": s.w, "status": s.st}
    if s.kind == "batch":
        if s.lob:
            bs.bs_cnn_forward(s.net, *s.inputs, s.Q.view(-1, 2), s.kper,
                              torch.view_as_real(s.U), stream)
            bs.bs_batch_set_start(s.h, s.U, NET_MP)
        bs.bs_batch_solve(s.h, s.Q, s.w, s.st, stream)
        out = {"omega": s.w, "status": s.st}
        if s.lob:
            out["start"] = s.U
        return out
    if s.kind == "modes":
        bs.bs_stress_coefficients(s.h, s.Q, s.U, s.S, stream)
        nk, nv = s.U.shape[0], s.U.shape[1]
        bs.bs_mode_field(s.h, s.Q, s.U.view(nk, 2 * nv, s.N), s.G, s.fu, stream)
        bs.bs_mode_field(s.h, s.Q, s.S.view(nk, 3 * nv, s.N), s.G, s.fs, stream)
        return {"stress": s.S, "field_u": s.fu, "field_s": s.fs}
    # lr = 0: the gradients alone, so that a repeated pass sees the same weights
    bs.bs_cnn_train_step(s.net, *s.inputs, s.Q, s.kper, s.V, 0.0, s.loss, stream)
    bs.bs_cnn_get_params(s.net, None, s.grad)
    return {"loss": s.loss, "grad": s.grad}


# ------------------------------------------------------------------ work
def _work_cell(N, gram, P, nf, nphase, nk, nbands, dim=2):
    """Set-up of one cell and its k: separable form factors, Cholesky factors
    of the Gram blocks (gram: their sizes), the matrix-vector products of
    the wanted branches; inputs and outputs moved once."""
    n, D = dim * N, 2 * round(N ** (1 / dim)) - 1
    f = 8.0 * nf * sum(P ** (dim - i) * D ** (i + 1) for i in range(dim))
    f += sum(4.0 / 3.0 * g ** 3 for g in gram)
    f += nk * 8.0 * n * n * nbands
    b = P ** dim * 2 + nphase * 24 + nk * (8 * dim + 8 * nbands + 4)
    return b, f


def work(case):
    k = case["kind"]
    if k in ("solve", "mixed", "aniso"):
        N = (2 * case["M"] + 1) ** 2
        gram = [N, 3 * N] if k == "aniso" else [N, N, N]
        if case.get("assemble", True):
            b, f = _work_cell(N, gram, case["P"], 7 if k == "aniso" else 3, case["nphase"], case["nk"],
                              case["nbands"])
        else:
            b = 6 * 16.0 * 4 * N * N / 2 + case["nk"] * (20 + 8 * case["nbands"])
            f = case["nk"] * (8.0 * 4 * N * N * case["nbands"])
    elif k == "mesh":
        N, nel = (2 * case["M"] + 1) ** 2, 2 * case["n"] ** 2
        b, f = _work_cell(N, [N, N, N], 1, 0, 2, case["nk"], case["nbands"])
        f += 8.0 * 4 * nel * (4 * case["M"] + 1) ** 2 / 2
        b += nel * 26
    elif k == "cell3":
        N = (2 * case["M"] + 1) ** 3
        b, f = _work_cell(N, [N, N, N], case["P"], 3, 2, case["nk"], case["nbands"], dim=3)
    elif k == "batch":
        b = f = 0.0
        for M in (5, 6, 7, 8):      # a quarter of the cells each, on average
            N = (2 * M + 1) ** 2
            b1, f1 = _work_cell(N, [N, N, N], 64, 3, 9, case["nk"], case["nbands"])
            b, f = b + b1 * case["ncells"] / 4, f + f1 * case["ncells"] / 4
        if case["solver"] == "lobpcg":
            b += case["ncells"] * case["nk"] * NET_NVEC * 98 * 8
            f += 2.0 * case["ncells"] * (10e6 + 1.5e6 * case["nk"])
    elif k == "modes":
        N, nm, G, W = (2 * case["M"] + 1) ** 2, case["nk"] * case["nvec"], case["G"], 2 * case["M"] + 1
        b = nm * (5 * 16.0 * N + 5 * 8.0 * G * G) + 3 * 8.0 * N * N
        f = nm * (24.0 * N * N + 5 * (8.0 * W * G * G + 8.0 * W * W * G))
    else:
        ns = case["ncells"] * case["kper"]
        npar = 1_759_056
        b = case["ncells"] * 64 * 64 * 2 + ns * (16 + case["nb"] * 98 * 8 + 4) + 2 * 4.0 * npar
        f = 6.0 * (10e6 * case["ncells"] + 1.73e6 * ns)
    return {"bytes": float(b), "flops": float(f)}


# ------------------------------------------------------------------ 64-bit values
# The mixed variational pencil written out with dense numpy / torch calls:
# A = H Phi^-1 H^dagger, Omega, and the eigenvalues of A u = omega^2 Omega u.
def _recip(h):
    return 2.0 * np.pi * np.linalg.inv(np.asarray(h, float))      # column i is q^i


def _toeplitz(g, idx):
    """g: (..., 4M+1 per axis); idx: the wave indices per axis; T[a, b] = g[a - b]."""
    off = (g.shape[-1] - 1) // 2
    return g[(Ellipsis,) + tuple(i[:, None] - i[None, :] + off for i in idx)]


def _ff_pixels(f, M, V):
    """f: (nf, P, ..., P) fields at pixel centres -> (nf, 4M+1, ...) centroid sums."""
    P, d = f.shape[-1], f.ndim - 1
    E = np.exp(-2j * np.pi * np.outer(np.arange(-2 * M, 2 * M + 1), (np.arange(P) + 0.5) / P))
    g = f.astype(complex)
    for ax in range(d):
        g = np.moveaxis(np.tensordot(E, g, axes=(1, ax + 1)), 0, ax + 1)
    return g * (V / P ** d)


def _ff_points(f, cen, area, M):
    """The same over mesh elements: f (nf, nel)."""
    d = np.arange(-2 * M, 2 * M + 1)
    Ea = np.exp(-2j * np.pi * np.outer(d, cen[:, 0]))
    Eb = np.exp(-2j * np.pi * np.outer(d, cen[:, 1]))
    return np.stack([(Ea * (g * area)) @ Eb.T for g in f])


def _voigt_compliance(c):
    """(nphase, 3, 3) compliance of (s11, s22, s12) against (e11, e22, 2 e12)."""
    st = getattr(c, "stiffness", None)
    if st is None:
        st = np.zeros((len(c.lam), 3, 3))
        st[:, 0, 0] = st[:, 1, 1] = c.lam + 2 * c.mu
        st[:, 0, 1] = st[:, 1, 0] = c.lam
        st[:, 2, 2] = c.mu
    return np.linalg.inv(st)


def _compliance3(c):
    """(nphase, 6, 6), stress order 11, 22, 33, 23, 13, 12."""
    C = np.zeros((len(c.lam), 6, 6))
    C[:, :3, :3] += c.lam[:, None, None]
    for i in range(3):
        C[:, i, i] += 2 * c.mu
        C[:, 3 + i, 3 + i] = c.mu
    return np.linalg.inv(C)


# strain component -> (row of u, derivative axis) pairs
_PAIRS2 = [[(0, 0)], [(1, 1)], [(0, 1), (1, 0)]]
_PAIRS3 = [[(0, 0)], [(1, 1)], [(2, 2)], [(1, 2), (2, 1)], [(0, 2), (2, 0)], [(0, 1), (1, 0)]]


class _Pencil:
    def __init__(self, c, M):
        self.dim = dim = 3 if hasattr(c, "h3") else 2
        h = np.array([c.h1, c.h2, c.h3] if dim == 3 else [c.h1, c.h2], float)
        self.q = _recip(h)
        V = abs(np.linalg.det(h))
        r = np.arange(-M, M + 1)
        self.idx = [g.ravel() for g in np.meshgrid(*([r] * dim), indexing="ij")]
        self.pairs = _PAIRS3 if dim == 3 else _PAIRS2
        S = _compliance3(c) if dim == 3 else _voigt_compliance(c)
        ns = len(self.pairs)
        tab = np.concatenate([S.reshape(len(c.rho), -1), c.rho[:, None], np.ones((len(c.rho), 1))], 1)
        f = np.moveaxis(tab[np.asarray(c.phase, np.int64)], -1, 0)
        g = (_ff_points(f, c.centroid, c.area, M) if hasattr(c, "centroid") else _ff_pixels(f, M, V))
        T = _toeplitz(g, self.idx)
        self.N = N = len(self.idx[0])
        dev = self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.I1 = torch.from_numpy(T[-1]).to(dev)
        Phi = T[:-2].reshape(ns, ns, N, N).transpose(0, 2, 1, 3).reshape(ns * N, ns * N)
        Lp = torch.linalg.cholesky(torch.from_numpy(np.ascontiguousarray(Phi)).to(dev))
        self.Zp = torch.linalg.solve_triangular(
            Lp, torch.eye(ns * N, dtype=Lp.dtype, device=dev), upper=False)
        Lr = torch.linalg.cholesky(torch.from_numpy(T[-2]).to(dev))
        self.Zr = torch.linalg.solve_triangular(
            Lr, torch.eye(N, dtype=Lr.dtype, device=dev), upper=False)

    def H(self, Q):
        K = np.stack([np.asarray(Q[i], float) + self.idx[i] for i in range(self.dim)], 1) @ self.q.T
        Kt = torch.from_numpy(K).to(self.dev)
        N = self.N
        H = torch.zeros((self.dim * N, len(self.pairs) * N), dtype=torch.complex128, device=self.dev)
        for c, prs in enumerate(self.pairs):
            for row, ax in prs:
                H[row * N:(row + 1) * N, c * N:(c + 1) * N] = 1j * self.I1 * Kt[:, ax][None, :]
        return H

    def reduced(self, Q):
        N = self.N
        B = self.Zp @ self.H(Q).conj().T
        B = torch.cat([B[:, i * N:(i + 1) * N] @ self.Zr.conj().T for i in range(self.dim)], 1)
        return (B.conj().T @ B).cpu().numpy()

    def omega(self, Qs, nbands):
        def one(C):
            return np.sqrt(np.maximum(np.linalg.eigvalsh(C)[:nbands], 0.0))
        with ThreadPoolExecutor(8) as ex:
            return np.array(list(ex.map(one, [self.reduced(Q) for Q in Qs])))

    def stress(self, Qs, U):
        out = []
        for Q, u in zip(Qs, U):
            r = self.H(Q).conj().T @ torch.from_numpy(u.T.copy()).to(self.dev)
            out.append(-(self.Zp.conj().T @ (self.Zp @ r)).T)
        return torch.stack(out)


def _fields(coef, Qs, M, G):
    """coef (nk, nf, N) complex128 -> (nk, nf, G, G) complex64 rounded from 64 bits' sums."""
    W, out = 2 * M + 1, []
    x = (torch.arange(G, dtype=torch.float64, device=coef.device) + 0.5) / G
    m = torch.arange(-M, M + 1, dtype=torch.float64, device=coef.device)
    for q, c in zip(Qs, coef):
        ph = [torch.exp(2j * math.pi * (m + float(q[i]))[:, None] * x[None, :]) for i in range(2)]
        f = torch.einsum("fab,ap->fpb", c.view(-1, W, W), ph[0])
        out.append(torch.einsum("fpb,bq->fpq", f, ph[1]))
    return torch.stack(out)


def _net_inputs(pack, i):
    ph = pack.phase[i].astype(np.int64)
    t = pack.table[pack.toff[i]:pack.toff[i] + 3 * pack.nph[i]].reshape(3, -1)
    lam, mu, rho = (v[ph] for v in t)
    return np.stack([np.log(lam + 2 * mu) - 3.5, (np.log(mu) - 2.2) / 1.2, (np.log(rho) - 1.0) / 0.6])


def _net_forward(p, pack, Q, kper):
    """The network in 64 bits: parameters p (flat float64 tensor), Q (samples, 2)."""
    x = torch.from_numpy(np.stack([_net_inputs(pack, i) for i in range(pack.n)])).to(p.device)
    o = 0

    def take(*shape):
        nonlocal o
        n = math.prod(shape)
        o += n
        return p[o - n:o].view(*shape)

    F = torch.nn.functional
    for ci, co in ((3, 16), (16, 32), (32, 32), (32, 32)):
        w, b = take(co, ci, 3, 3), take(co)
        x = F.avg_pool2d(F.relu(F.conv2d(F.pad(x, (1, 1, 1, 1), mode="circular"), w, b)), 2)
    q = torch.from_numpy(np.asarray(Q, float)).to(p.device)
    hexf = torch.from_numpy(pack.hexflag.astype(float)).to(p.device).repeat_interleave(kper)
    t = 2 * math.pi * q
    kf = torch.stack([q[:, 0], q[:, 1], t[:, 0].cos(), t[:, 0].sin(), t[:, 1].cos(), t[:, 1].sin(),
                      hexf], 1)
    y = torch.cat([x.flatten(1).repeat_interleave(kper, 0), kf], 1)
    L = 2 * (2 * NET_MP + 1) ** 2
    for l, (di, do) in enumerate(((519, 512), (512, 512), (512, NET_NVEC * L * 2))):
        w, b = take(do, di), take(do)
        y = F.linear(y, w, b)
        if l < 2:
            y = F.relu(y)
    return torch.view_as_complex(y.view(len(q), NET_NVEC, L, 2))


def exact(case, seed):
    k = case["kind"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if k in ("solve", "mixed", "aniso", "mesh", "cell3"):
        c = _cell3(case, seed) if k == "cell3" else _mesh(case, seed) if k == "mesh" else _cell(case, seed)
        Q = _path3(case["nk"]) if k == "cell3" else _path(case["lattice"], case["nk"], c.h1, c.h2)
        return {"omega": _Pencil(c, case["M"]).omega(Q, case["nbands"]),
                "status": np.zeros(case["nk"], np.int32)}
    if k == "batch":
        if case["ncells"] * case["nk"] > 800 and case["solver"] != "lobpcg":
            return None      # some 20 seconds and more of dense eigenvalues
        cl, Ms, Q = _batch(case, seed)
        out = {"omega": None, "status": np.zeros(Q.shape[:2], np.int32)}
        if case["ncells"] * case["nk"] <= 800:
            out["omega"] = np.stack([_Pencil(c, M).omega(q, case["nbands"])
                                     for c, M, q in zip(cl, Ms, Q)])
        if case["solver"] == "lobpcg":
            p = torch.from_numpy(_params_of_shipped_net().astype(float)).to(dev)
            u = _net_forward(p, warmstart.CellPack(cl), Q.reshape(-1, 2), case["nk"])
            out["start"] = u.view(case["ncells"], case["nk"], NET_NVEC, -1)
        return out
    if k == "modes":
        c = _cell(case, seed)
        Q = _path(case["lattice"], case["nk"], c.h1, c.h2)
        U = _modes(case, seed)
        N, nk, nv = (2 * case["M"] + 1) ** 2, case["nk"], case["nvec"]
        S = _Pencil(c, case["M"]).stress(Q, U)
        Ut = torch.from_numpy(U).to(S.device)
        return {"stress": S, "field_u": _fields(Ut.view(nk, 2 * nv, N), Q, case["M"], case["G"]),
                "field_s": _fields(S.contiguous().view(nk, 3 * nv, N), Q, case["M"], case["G"])}
    pack, Q, p, V = _net(case, seed)
    p = torch.from_numpy(p.astype(float)).to(dev).requires_grad_(True)
    U = _net_forward(p, pack, Q, case["kper"]).transpose(1, 2)
    Vt = torch.from_numpy(V.astype(np.complex128)).to(dev).transpose(1, 2)
    Uh = U.conj().transpose(1, 2)
    B = Uh @ Vt
    G = Uh @ U + 1e-4 * torch.eye(NET_NVEC, dtype=U.dtype, device=dev)
    cap = (B.conj() * torch.linalg.solve(G, B)).real.sum((1, 2))
    v2 = Vt.abs().square().sum((1, 2))
    loss = (v2 - cap) / v2
    loss.mean().backward()
    return {"loss": loss.detach(), "grad": p.grad}
