"""Network products at sizes where the tiling can go wrong: odd layer sizes
(scalar loads), fewer rows than a tile, k ranges split over several CTAs, and
an input that is not 16-byte aligned, against FP64 numpy.

Tolerance: a sum of K FP32 products, each rounded once and added in FP32, is
off by at most K 2^-24 of the sum of magnitudes; the bound used is normwise
1e-5, more than K 2^-24 for every K here and far below any indexing mistake.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp_oracle as M
from paper_2112_03804_gb300 import kps

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("din,width,dout,rows,shift", [(7, 5, 3, 1, 0), (33, 65, 12, 63, 0), (64, 64, 32, 65, 0),
                                                       (100, 72, 4, 1100, 1), (1232, 256, 12, 700, 0)])
def test_gradients_at_odd_sizes(din, width, dout, rows, shift):
    r = np.random.default_rng(rows)
    m = kps.MLP(din, width, dout, seed=3)
    p = m.get(0).astype(np.float64)
    blocks = M.unpack(p, din, width, dout)
    # positive hidden layers: no ReLU decision near zero
    for i in (0, 2):
        blocks[i] = torch.from_numpy(np.abs(blocks[i])).bfloat16().double().numpy()
    blocks[4] = torch.from_numpy(blocks[4]).bfloat16().double().numpy()
    p = M.pack(blocks)
    m.set(p.astype(np.float32))
    X = r.uniform(0.1, 1.0, size=(rows, din)).astype(np.float32)
    nact = r.integers(1, dout + 1, size=rows).astype(np.int32)
    T = np.zeros((rows, dout), np.float32)
    for q in range(rows):
        T[q, :nact[q]] = r.dirichlet(np.ones(nact[q]))
    w = r.uniform(0.2, 2.0, size=rows).astype(np.float32)
    flat = torch.zeros(rows * din + shift, device="cuda")
    dX = flat[shift:]
    dX.copy_(torch.from_numpy(X).reshape(-1))
    dn, dT, dw = (torch.from_numpy(a).cuda() for a in (nact, T, w))
    loss = torch.zeros(1, device="cuda")
    m.gradients(dX, rows, dn, dT, dw, float(w.sum()), loss)
    torch.cuda.synchronize()
    L, g = M.loss_and_grads(p, X.astype(np.float64), nact, T.astype(np.float64), w.astype(np.float64), din, width, dout)
    got = m.get(1).astype(np.float64)
    assert abs(float(loss.item()) - L) <= 1e-5 * abs(L)
    for a, b in zip(M.unpack(got, din, width, dout), M.unpack(g, din, width, dout)):
        scale = np.max(np.abs(g))
        assert np.max(np.abs(a - b)) <= 1e-5 * max(np.max(np.abs(b)), 1e-3 * scale)
