"""The TMA-staged kernel's paired items (fold and call of one bet in one scan)
and its 16-bit storage: river batches around the 32-vector tile, the
eight-warp shape of small batches, 47, 48 and 49
cards left, decks too small for paired items, against the oracle on the
rounded inputs.  Tolerances: 1e-5 normwise for FP32, one output rounding
(2^-8 BF16, 2^-10 FP16) for 16-bit storage.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.oracle import OracleGame
from paper_2112_03804_gb300 import kps, synth
from tests.gpu_util import from_library, library_order, normwise_error, to_library

pytestmark = pytest.mark.gpu

TOL = {torch.float32: 1e-5, torch.bfloat16: 2.0 ** -8, torch.float16: 2.0 ** -10}
SPECS = {
    "river": lambda: synth.river_spec(seed=2),
    "turn_board": lambda: synth.river_spec(seed=3, nboard=4),
    "flop_board": lambda: synth.river_spec(seed=4, nboard=3),
    "small_deck": lambda: synth.micro_spec(seed=5, ranks=6, suits=4, nboard=3, ties=False),
    "one_card": lambda: synth.micro_spec(seed=6, ranks=12, suits=4, nboard=1, cards_per_hand=1, ties=False),
}


@pytest.mark.parametrize("dt", [torch.float64, torch.float32, torch.bfloat16])
@pytest.mark.parametrize("first", [0, 8])
def test_captured_after_the_other_alignment(dt, first):
    """A captured product whose kernel is not the one that the calls before
    it took (vectors 16-byte aligned or not): its tables are made outside the
    graph, and the replay gives what the same call gives without a graph."""
    spec = SPECS["river"]()
    g = kps.Game(spec)
    inf = g.info()
    nin, nout = 2 * inf["n2"] * inf["hs"], 2 * inf["n1"] * inf["hs"]
    buf = torch.randn(nin + 16, device="cuda", dtype=torch.float64).to(dt)
    out = torch.zeros(nout + 16, device="cuda", dtype=dt)
    es = buf.element_size()
    at = lambda off: (buf[off // es:][:nin], out[off // es:][:nout])
    kps.matvec_A(g, *at(first), 2)
    torch.cuda.synchronize()
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    vin, o = at(8 - first)
    with torch.cuda.graph(graph, stream=side):
        kps.matvec_A(g, vin, o, 2, stream=side)
    o.zero_()
    graph.replay()
    got = o.clone()
    kps.matvec_A(g, vin, o, 2)
    kps.device_status()
    err = (got.double() - o.double()).norm() / o.double().norm()
    assert err <= TOL.get(dt, 1e-12)


@pytest.mark.parametrize("dt", list(TOL))
@pytest.mark.parametrize("name,batch", [("river", 1), ("river", 33), ("turn_board", 5), ("flop_board", 5),
                                        ("river", 300), ("small_deck", 40), ("one_card", 3)])
@pytest.mark.parametrize("transpose", [False, True])
def test_products(name, batch, dt, transpose):
    spec = SPECS[name]()
    og, g = OracleGame(spec), kps.Game(spec)
    inf = g.info()
    order = library_order(spec["strength"])
    v = synth.simplex_vectors(og.sequences(0 if transpose else 1)["nact"], og.H, batch, seed=31 + batch)
    vin = torch.from_numpy(to_library(v, order, inf["hs"])).to("cuda", dt).contiguous()
    out = torch.full((batch, inf["n2"] if transpose else inf["n1"], inf["hs"]), float("nan"), device="cuda", dtype=dt)
    (kps.matvec_AT if transpose else kps.matvec_A)(g, vin, out, batch)
    kps.device_status()
    assert g.kernel(int(transpose)) == "tma" or name == "flop_board"   # its four chunks are too long
    o = out.double().cpu().numpy()
    assert np.all(o[..., inf["H"]:] == 0)
    rounded = torch.from_numpy(v).to(dt).double().numpy()
    want = og.matvec_AT(rounded) if transpose else og.matvec_A(rounded)
    assert normwise_error(from_library(o, order, inf["H"]), want) <= TOL[dt]
