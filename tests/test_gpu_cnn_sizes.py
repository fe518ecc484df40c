"""The warm-start network at the sizes where its kernels change over: one sample,
and enough samples for the wide product tiles; few and many output channels per
thread; a cell of more phases than the encoder's table holds.

The forward pass adds the terms of every output in one order, whatever the tile:
a cell alone and the same cell in a batch give the same bits.  The gradients are
held to the bound of the other gradient test (2e-3 of the norm of each layer).
"""
import numpy as np
import pytest

from oracle import warm_start_net as wn
from paper_1310_6380_gb300 import cells, warmstart

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

NV, MP = 12, 3
L = 2 * (2 * MP + 1) ** 2


@pytest.fixture(scope="module")
def net():
    n = warmstart.WarmStartNet(NV, MP, max_cells=72, max_samples=360, seed=3)
    yield n
    n.close()


@pytest.mark.parametrize("nc, kper, nb", [(1, 1, 1), (5, 3, 10), (72, 5, 16)])
def test_batch_and_single_cell_agree(net, nc, kper, nb):
    cl = [cells.config3_cell(i)["cell"] for i in range(nc - 1)] + [cells.voronoi_cell(64, 1400, seed=3)]
    pack = warmstart.CellPack(cl)
    rng = np.random.default_rng(nc)
    Q = rng.uniform(0, 0.5, (nc, kper, 2))
    V = (rng.standard_normal((nc, kper, nb, L)) +
         1j * rng.standard_normal((nc, kper, nb, L))).astype(np.complex64)
    U = net.predict(pack, Q)
    for c in {0, nc // 2, nc - 1}:
        assert np.array_equal(net.predict(pack.subset([c]), Q[c:c + 1])[0], U[c]), c
    x = np.stack([wn.encode(c.phase, c.lam, c.mu, c.rho) for c in cl])
    kf = np.stack([wn.kfeatures(Q[c, j], cl[c].lattice == "hex")
                   for c in range(nc) for j in range(kper)])
    p = net.params()
    loss = net.train_step(pack, Q, V, lr=0.0)
    g = net.grads()
    Vr = V.reshape(nc * kper, nb, L).transpose(0, 2, 1)
    lref, gref = wn.loss_and_grad(p.astype(np.float64), x, kf, kper, Vr, NV, MP)
    assert np.allclose(loss, lref, rtol=1e-4, atol=1e-5)
    o = 0
    for name, shape in wn.layout(NV, MP):
        n = int(np.prod(shape))
        a, b = g[o:o + n].astype(np.float64), gref[o:o + n]
        assert np.linalg.norm(a - b) <= 2e-3 * max(np.linalg.norm(b), 1e-30), name
        o += n
