"""Batches in which the staged kernel leaves a game to the tensor-memory kernel:
a tie group of 30 hands lists 870 ordered pairs (less those that share a card), of
which one chunk of the hand order, or two if a chunk boundary cuts the group, would hold
more than the 256 it takes.  Products of every storage type against the oracle
(1e-5 FP32, one output rounding for 16 bits, on the rounded inputs) whichever
place the game has in the batch, and solver iterations, whose captured products
make both launches, against the FP64 solver.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.oracle import OracleGame
from paper_2112_03804_gb300 import kps, synth
from tests.gpu_util import from_library, library_order, normwise_error, to_library

pytestmark = pytest.mark.gpu

TOL = {torch.float32: 1e-5, torch.bfloat16: 2.0 ** -8, torch.float16: 2.0 ** -10}
CODE = {torch.float32: kps.F32, torch.bfloat16: kps.BF16, torch.float16: kps.F16}


def _tied(spec, at, n=30):
    s = np.asarray(spec["strength"])
    order = np.lexsort((np.arange(len(s)), s))
    s = np.empty(len(s), dtype=np.int64)
    s[order] = 10 * np.arange(len(s))
    s[order[at:at + n]] = s[order[at]]
    return dict(spec, strength=s.tolist())


def _specs(place):
    specs = [synth.river_spec(seed=3), synth.river_spec(seed=4, nboard=4, bet_frac=(0.5,))]
    specs.insert(place, _tied(synth.river_spec(seed=5), 100 + 120 * place))
    return specs


@pytest.mark.parametrize("dt", list(TOL))
@pytest.mark.parametrize("place", [0, 1, 2])
def test_products(place, dt):
    specs = _specs(place)
    games = [kps.Game(s) for s in specs]
    b = kps.Batch(games)
    ors = [OracleGame(s) for s in specs]
    orders = [library_order(s["strength"]) for s in specs]
    infs = [g.info() for g in games]
    for transpose in (False, True):
        pin = 0 if transpose else 1
        off = b.offsets(1 - pin)
        vs = [synth.simplex_vectors(o.sequences(pin)["nact"], o.H, 1, seed=9 + i)[0] for i, o in enumerate(ors)]
        flat = np.concatenate([to_library(v, o, i["hs"]).reshape(-1) for v, o, i in zip(vs, orders, infs)])
        out = torch.full((int(off[-1]),), float("nan"), device="cuda", dtype=dt)
        (b.matvec_AT if transpose else b.matvec_A)(torch.from_numpy(flat).to("cuda", dt), out)
        kps.device_status()
        assert b.shape(CODE[dt])["kernel"] == kps.BATCH_STAGED
        res = out.double().cpu().numpy()
        for i, o in enumerate(ors):
            want = (o.matvec_AT if transpose else o.matvec_A)(torch.from_numpy(vs[i]).to(dt).double().numpy()[None])[0]
            got = from_library(res[off[i]:off[i + 1]].reshape(-1, infs[i]["hs"]), orders[i], infs[i]["H"])
            assert normwise_error(got, want) <= TOL[dt], i


def test_solver():
    b = kps.Batch([kps.Game(s) for s in _specs(1)])
    e = {}
    for dt in (kps.F32, kps.F64):
        s = kps.Solver(b, dt)
        s.step(3)
        e[dt] = torch.zeros(3, dtype=torch.float64, device="cuda")
        s.exploitability(e[dt])
        s.status()
    # a strategy entry decided at the matching floor may differ; the value of the
    # averages of three iterations does not move by a thousandth of the pot for it
    assert float((e[kps.F32] - e[kps.F64]).abs().max()) <= 1e-3
    assert float(e[kps.F64].min()) > 0
