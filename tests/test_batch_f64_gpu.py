"""FP64 launch shapes of a batch: what kps_batch_shape_get and the tuner report
is what runs, a shape that is set takes effect, and a batch that the FP64
kernel refuses (a game of many ties) runs the vector-register variant, against
the oracle (1e-12 normwise, as every FP64 product).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.oracle import OracleGame
from paper_2112_03804_gb300 import kps, synth
from tests.gpu_util import from_library, library_order, normwise_error, to_library

pytestmark = pytest.mark.gpu


def _tied(spec, n):
    s = np.asarray(spec["strength"])
    rank = np.empty(len(s), dtype=np.int64)
    rank[np.lexsort((np.arange(len(s)), s))] = np.arange(len(s))
    return dict(spec, strength=(rank // n).tolist())


class _Case:
    def __init__(self, specs):
        self.ors = [OracleGame(s) for s in specs]
        self.orders = [library_order(s["strength"]) for s in specs]
        self.games = [kps.Game(s) for s in specs]
        self.infs = [g.info() for g in self.games]
        self.b = kps.Batch(self.games)
        self.v = [[synth.simplex_vectors(o.sequences(p)["nact"], o.H, 1, seed=9 + i)[0]
                   for i, o in enumerate(self.ors)] for p in (0, 1)]
        self.want = [[o.matvec_A(v[None])[0] for o, v in zip(self.ors, self.v[1])],
                     [o.matvec_AT(v[None])[0] for o, v in zip(self.ors, self.v[0])]]

    def products(self):
        """Both products, checked against the oracle."""
        outs = []
        for p in (0, 1):
            flat = np.concatenate([to_library(v, o, i["hs"]).reshape(-1)
                                   for v, o, i in zip(self.v[1 - p], self.orders, self.infs)])
            off = self.b.offsets(p)
            out = torch.full((int(off[-1]),), float("nan"), device="cuda", dtype=torch.float64)
            (self.b.matvec_AT if p else self.b.matvec_A)(torch.from_numpy(flat).cuda(), out)
            kps.device_status()
            res = out.cpu().numpy()
            for i, o in enumerate(self.orders):
                got = from_library(res[off[i]:off[i + 1]].reshape(-1, self.infs[i]["hs"]), o, self.infs[i]["H"])
                assert normwise_error(got, self.want[p][i]) <= 1e-12
            outs.append(out)
        return outs


def _rivers():
    return [synth.river_spec(seed=3), synth.river_spec(seed=5, nboard=4, bet_frac=(0.5,)), synth.river_spec(seed=6)]


def test_shapes_say_what_runs():
    c = _Case(_rivers())
    b = c.b
    own = b.shape(kps.F64)
    assert own["kernel"] == kps.BATCH_F64 and own["warps"] == 6
    first = c.products()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    # the other kernel: another order of summation, so other last bits
    ran = 0
    for w in range(1, 9):
        try:
            b.set_shape(kps.F64, w, sms, w & 1, kps.BATCH_TMEM)
        except kps.KpsError as e:
            assert e.status == kps.ENOTSUP
            continue
        sh = b.shape(kps.F64)
        assert (sh["kernel"], sh["warps"], sh["schedule"]) == (kps.BATCH_TMEM, w, w & 1)
        assert not all(torch.equal(a, o) for a, o in zip(first, c.products()))
        ran += 1
    assert ran >= 2
    for w, dt in ((4, kps.F64), (6, kps.F32)):
        with pytest.raises(kps.KpsError) as e:
            b.set_shape(dt, w, own["grid"], own["schedule"], kps.BATCH_F64)
        assert e.value.status == kps.ENOTSUP
    b.set_shape(kps.F64, own["warps"], own["grid"], own["schedule"], own["kernel"])
    assert all(torch.equal(a, o) for a, o in zip(first, c.products()))
    # river games: the tuner measures both kernels and finds the FP64 one faster
    sh = b.tune(kps.F64)
    assert sh["kernel"] == kps.BATCH_F64 and sh["ms_per_pair"] > 0
    assert all(torch.equal(a, o) for a, o in zip(first, c.products()))


def test_many_ties_take_the_other_kernel():
    c = _Case(_rivers()[:1] + [_tied(synth.river_spec(seed=7), 9), _tied(synth.river_spec(seed=8), 30)])
    assert c.b.shape(kps.F64)["kernel"] == kps.BATCH_TMEM
    c.products()
    with pytest.raises(kps.KpsError) as e:
        c.b.set_shape(kps.F64, 6, 10, 1, kps.BATCH_F64)
    assert e.value.status == kps.ENOTSUP
    assert c.b.tune(kps.F64)["kernel"] == kps.BATCH_TMEM
    c.products()


def test_first_call_while_capturing():
    """A first FP64 product under capture runs the vector-register variant, its
    tables made outside the graph; the batch takes the FP64 kernel afterwards."""
    specs = _rivers()[:2]
    c = _Case(specs)
    fresh = kps.Batch(c.games)
    flat = np.concatenate([to_library(v, o, i["hs"]).reshape(-1) for v, o, i in zip(c.v[1], c.orders, c.infs)])
    vin = torch.from_numpy(flat).cuda()
    off = fresh.offsets(0)
    out = torch.full((int(off[-1]),), float("nan"), device="cuda", dtype=torch.float64)
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=side):
        fresh.matvec_A(vin, out, stream=side)
    graph.replay()
    kps.device_status()
    res = out.cpu().numpy()
    for i, o in enumerate(c.orders):
        got = from_library(res[off[i]:off[i + 1]].reshape(-1, c.infs[i]["hs"]), o, c.infs[i]["H"])
        assert normwise_error(got, c.want[0][i]) <= 1e-12
    assert fresh.shape(kps.F64)["kernel"] == kps.BATCH_F64
