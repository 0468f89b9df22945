"""Bias gradients where their rows are one part and where they are several (256
rows and 257), and the smallest minibatch, against FP64 numpy.  Each column sum adds
its rows in FP32, 8 interleaved runs per part and the parts in order: at most
rows / 8 + 8 + parts roundings a sum, each 2^-24 of the magnitudes added.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp_oracle as M
from paper_2112_03804_gb300 import kps

pytestmark = pytest.mark.gpu

DIN, WIDTH, DOUT = 24, 40, 5


@pytest.mark.parametrize("rows", [1, 64, 65, 256, 257, 4100])
def test_bias_gradients(rows):
    r = np.random.default_rng(rows)
    m = kps.MLP(DIN, WIDTH, DOUT, seed=3)
    blocks = M.unpack(m.get(0).astype(np.float64), DIN, WIDTH, DOUT)
    # positive hidden layers: no ReLU decision near zero
    for i in (0, 2):
        blocks[i] = np.abs(blocks[i])
    for i in (0, 2, 4):
        blocks[i] = torch.from_numpy(blocks[i]).bfloat16().double().numpy()
    p = M.pack(blocks)
    m.set(p.astype(np.float32))
    X = r.uniform(0.1, 1.0, size=(rows, DIN)).astype(np.float32)
    nact = np.full(rows, DOUT, np.int32)
    T = r.dirichlet(np.ones(DOUT), size=rows).astype(np.float32)
    w = r.uniform(0.2, 2.0, size=rows).astype(np.float32)
    dX, dn, dT, dw = (torch.from_numpy(a).cuda() for a in (X, nact, T, w))
    m.gradients(dX, rows, dn, dT, dw, float(w.sum()))
    torch.cuda.synchronize()
    x64 = X.astype(np.float64)
    _, g = M.loss_and_grads(p, x64, nact, T.astype(np.float64), w.astype(np.float64), DIN, WIDTH, DOUT)
    got, want = (M.unpack(a, DIN, WIDTH, DOUT) for a in (m.get(1).astype(np.float64), g))
    # a logit: three layers of at most WIDTH products each, rounded in FP32, against
    # the magnitudes added; a probability moves by no more than the largest logit does
    _, (_, _, _, _, H2, _) = M.forward(p, x64, nact, DIN, WIDTH, DOUT)
    dz = 3 * WIDTH * 2.0 ** -24 * float((H2 @ np.abs(blocks[4])).max())
    parts = 1 if rows <= 256 else -(-rows // max(64, -(-rows // 64)))
    eps = (rows / parts / 8 + 8 + parts) * 2.0 ** -24 + dz
    # magnitudes added: sum w / sum w = 1 a column at the logits, times the weights below
    mag = [1.0, float(np.abs(blocks[4]).sum(1).max())]
    mag.append(mag[1] * float(np.abs(blocks[2]).sum(1).max()))
    for i, k in ((5, 0), (3, 1), (1, 2)):
        assert np.max(np.abs(got[i] - want[i])) <= eps * mag[k]
