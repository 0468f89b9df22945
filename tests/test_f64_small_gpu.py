"""FP64 products of small decks, whose items are chosen by their fixed part as
much as by their boxes: 15 to 210 hands (1 to 27 boxes of 8 over 6 to 24 parts, so
parts without a box), one vector to several waves of items, and many games of
mixed sizes in one launch, against the oracle (1e-12 normwise).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.oracle import OracleGame
from paper_2112_03804_gb300 import kps, synth
from tests.gpu_util import from_library, library_order, normwise_error, to_library

pytestmark = pytest.mark.gpu

DECKS = [(4, 2, 2), (6, 2, 2), (4, 4, 1), (5, 4, 3), (6, 4, 3)]      # ranks, suits, board


def _spec(deck, seed=5):
    return synth.micro_spec(seed=seed, ranks=deck[0], suits=deck[1], nboard=deck[2], ties=False)


@pytest.mark.parametrize("batch", [1, 33, 150, 1000])
@pytest.mark.parametrize("deck", DECKS, ids=lambda d: "x".join(map(str, d)))
def test_one_game(deck, batch):
    spec = _spec(deck)
    og, g = OracleGame(spec), kps.Game(spec)
    inf, order = g.info(), library_order(spec["strength"])
    for transpose in (False, True):
        v = synth.simplex_vectors(og.sequences(0 if transpose else 1)["nact"], og.H, batch, seed=7)
        vin = torch.from_numpy(to_library(v, order, inf["hs"])).cuda()
        out = torch.full((batch, inf["n2" if transpose else "n1"], inf["hs"]), float("nan"), device="cuda",
                         dtype=torch.float64)
        (kps.matvec_AT if transpose else kps.matvec_A)(g, vin, out, batch)
        torch.cuda.synchronize()
        assert g.kernel(int(transpose)) == "f64"
        got = from_library(out.cpu().numpy(), order, inf["H"])
        assert normwise_error(got, og.matvec_AT(v) if transpose else og.matvec_A(v)) <= 1e-12


@pytest.mark.parametrize("copies", [1, 60])
def test_mixed_games(copies):
    specs = [_spec(d, 5 + i) for i, d in enumerate(DECKS)] + [synth.river_spec(seed=3, bet_frac=(0.5,))]
    games = [kps.Game(s) for s in specs * copies]
    b = kps.Batch(games)
    assert b.shape(kps.F64)["kernel"] == kps.BATCH_F64
    for transpose in (False, True):
        off, flat, want = b.offsets(1 if transpose else 0), [], []
        for i, s in enumerate(specs):
            og, inf = OracleGame(s), games[i].info()
            v = synth.simplex_vectors(og.sequences(0 if transpose else 1)["nact"], og.H, 1, seed=7)
            flat.append(to_library(v[0], library_order(s["strength"]), inf["hs"]).reshape(-1))
            want.append((og.matvec_AT if transpose else og.matvec_A)(v)[0])
        vin = torch.from_numpy(np.concatenate(flat * copies)).cuda()
        out = torch.full((int(off[-1]),), float("nan"), device="cuda", dtype=torch.float64)
        (b.matvec_AT if transpose else b.matvec_A)(vin, out)
        torch.cuda.synchronize()
        res = out.cpu().numpy()
        for i in range(len(games)):
            s, inf = specs[i % len(specs)], games[i].info()
            got = from_library(res[off[i]:off[i + 1]].reshape(-1, inf["hs"]), library_order(s["strength"]), inf["H"])
            assert normwise_error(got, want[i % len(specs)]) <= 1e-12
