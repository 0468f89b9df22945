"""The TMA-staged kernel's forms at the sizes where the choice changes: games of
1 to 26 boxes (four warps up to 4 boxes, the small form up to 24), one-card hands,
and 1128 hands, where eight warps take every batch, at one vector, a ragged tile
and several waves, against the oracle on the rounded inputs.  Tolerances: 1e-5
normwise for FP32, one output rounding (2^-8 BF16, 2^-10 FP16) for 16-bit storage.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.oracle import OracleGame
from paper_2112_03804_gb300 import kps, synth
from tests.gpu_util import from_library, library_order, normwise_error, to_library

pytestmark = pytest.mark.gpu

TOL = {torch.float32: 1e-5, torch.bfloat16: 2.0 ** -8, torch.float16: 2.0 ** -10}


def _deck(ranks, suits, nboard, cards=2):
    return lambda: synth.micro_spec(seed=5, ranks=ranks, suits=suits, nboard=nboard, cards_per_hand=cards, ties=False)


SPECS = {"box1": _deck(4, 2, 2), "box3": _deck(6, 2, 2), "box5": _deck(4, 3, 0), "box7": _deck(4, 4, 1),
         "box14": _deck(6, 4, 3), "box26": _deck(8, 4, 3), "one_card_box3": _deck(12, 4, 1, 1),
         "turn_board": lambda: synth.river_spec(seed=3, nboard=4, bet_frac=(0.5,))}


@pytest.mark.parametrize("dt", list(TOL))
@pytest.mark.parametrize("name,batch", [(n, b) for n in SPECS for b in (1, 33, 700) if n != "turn_board"] +
                         [("turn_board", b) for b in (1, 40, 330)])
def test_forms(name, batch, dt):
    spec = SPECS[name]()
    og, g = OracleGame(spec), kps.Game(spec)
    inf, order = g.info(), library_order(spec["strength"])
    for transpose in (False, True):
        v = synth.simplex_vectors(og.sequences(0 if transpose else 1)["nact"], og.H, batch, seed=31 + batch)
        vin = torch.from_numpy(to_library(v, order, inf["hs"])).to("cuda", dt).contiguous()
        out = torch.full((batch, inf["n2" if transpose else "n1"], inf["hs"]), float("nan"), device="cuda", dtype=dt)
        (kps.matvec_AT if transpose else kps.matvec_A)(g, vin, out, batch)
        kps.device_status()
        assert g.kernel(int(transpose)) == "tma"
        o = out.double().cpu().numpy()
        assert np.all(o[..., inf["H"]:] == 0)
        rounded = torch.from_numpy(v).to(dt).double().numpy()
        want = og.matvec_AT(rounded) if transpose else og.matvec_A(rounded)
        assert normwise_error(from_library(o, order, inf["H"]), want) <= TOL[dt]
