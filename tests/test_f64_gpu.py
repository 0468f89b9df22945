"""The FP64 product kernel at the sizes where it can go wrong: bit-exact on
dyadic games (tie groups, items of 8 to 32 columns), boards of 3 to 5
cards, games it does not take, padding entries that hold NaN, and many games in
one launch, against the oracle (1e-12 normwise, as every FP64 product).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.oracle import OracleGame
from paper_2112_03804_gb300 import kps, synth
from tests.dyadic import dyadic_river
from tests.gpu_util import from_library, library_order, normwise_error, to_library

pytestmark = pytest.mark.gpu


def _product(g, v, order, transpose):
    inf = g.info()
    vl = to_library(v, order, inf["hs"])
    vl[..., inf["H"]:] = np.nan                 # padding is ignored on input
    vin = torch.from_numpy(vl).cuda().contiguous()
    out = torch.full((v.shape[0], inf["n2"] if transpose else inf["n1"], inf["hs"]), float("nan"), device="cuda",
                     dtype=torch.float64)
    (kps.matvec_AT if transpose else kps.matvec_A)(g, vin, out, v.shape[0])
    torch.cuda.synchronize()
    o = out.cpu().numpy()
    assert np.all(o[..., inf["H"]:] == 0)
    return from_library(o, order, inf["H"])


@pytest.mark.parametrize("ties", [False, True], ids=["river", "river_ties4"])
@pytest.mark.parametrize("batch", [1, 5, 90, 300])
def test_river_bit_exact(ties, batch):
    spec = dyadic_river(seed=2, ties=ties)
    og, g = OracleGame(spec), kps.Game(spec)
    order = library_order(spec["strength"])
    inf = g.info()
    for transpose in (False, True):
        v = synth.integer_vectors(inf["n1"] if transpose else inf["n2"], og.H, batch, seed=11 + transpose)
        got = _product(g, v, order, transpose)
        assert g.kernel(int(transpose)) == "f64" or ties
        assert np.array_equal(got, og.matvec_AT(v) if transpose else og.matvec_A(v))


@pytest.mark.parametrize("nboard,batch", [(3, 2), (4, 33), (5, 7)])
@pytest.mark.parametrize("transpose", [False, True])
def test_boards(nboard, batch, transpose):
    spec = synth.river_spec(seed=5, nboard=nboard)
    og, g = OracleGame(spec), kps.Game(spec)
    order = library_order(spec["strength"])
    v = synth.simplex_vectors(og.sequences(0 if transpose else 1)["nact"], og.H, batch, seed=5)
    got = _product(g, v, order, transpose)
    assert g.kernel(int(transpose)) == "f64"
    assert normwise_error(got, og.matvec_AT(v) if transpose else og.matvec_A(v)) <= 1e-12


def test_many_ties_take_another_kernel():
    spec = synth.river_spec(seed=5)
    s = np.asarray(spec["strength"])
    rank = np.empty(len(s), dtype=np.int64)
    rank[np.lexsort((np.arange(len(s)), s))] = np.arange(len(s))
    spec["strength"] = (rank // 9).tolist()
    og, g = OracleGame(spec), kps.Game(spec)
    v = synth.simplex_vectors(og.sequences(1)["nact"], og.H, 3, seed=5)
    got = _product(g, v, library_order(spec["strength"]), False)
    assert g.kernel(0) == "vec"
    assert normwise_error(got, og.matvec_A(v)) <= 1e-12


@pytest.mark.parametrize("copies", [1, 40])
def test_many_games(copies):
    base = [synth.river_spec(seed=3), synth.river_spec(seed=5, nboard=4, bet_frac=(0.33, 0.66, 1.0)),
            synth.river_spec(seed=6, nboard=3, bet_frac=(0.5,), raise_cap=2),
            synth.micro_spec(seed=8, ranks=6, suits=3, nboard=4, ties=False)]
    games = [kps.Game(s) for s in base * copies]
    b = kps.Batch(games)
    ors = [OracleGame(s) for s in base]
    orders = [library_order(s["strength"]) for s in base]
    infs = [g.info() for g in games[:len(base)]]
    for transpose in (False, True):
        pin = 0 if transpose else 1
        off = b.offsets(1 - pin)
        vs = [synth.simplex_vectors(o.sequences(pin)["nact"], o.H, 1, seed=9 + i)[0] for i, o in enumerate(ors)]
        flat = np.concatenate([to_library(v, o, i["hs"]).reshape(-1) for v, o, i in zip(vs, orders, infs)] * copies)
        out = torch.full((int(off[-1]),), float("nan"), device="cuda", dtype=torch.float64)
        (b.matvec_AT if transpose else b.matvec_A)(torch.from_numpy(flat).cuda(), out)
        torch.cuda.synchronize()
        res = out.cpu().numpy()
        parts = [res[off[i]:off[i + 1]] for i in range(len(games))]
        for i, o in enumerate(ors):
            want = (o.matvec_AT if transpose else o.matvec_A)(vs[i][None])[0]
            got = from_library(parts[i].reshape(-1, infs[i]["hs"]), orders[i], infs[i]["H"])
            assert normwise_error(got, want) <= 1e-12
            for k in range(1, copies):
                assert np.array_equal(parts[i], parts[i + k * len(base)])
