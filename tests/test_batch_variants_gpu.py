"""The staged batched kernel's four variants (pairs or single rows, with or
without listed ties of more than 4 hands): one- and two-card hands, few games
(single rows in split items) and many (pairs), against the oracle game by game
(half precision: on the rounded inputs), each copy of a game the same bits.
Tolerances as for the other batched products: 1e-5, 2^-8, 2^-10 normwise.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.oracle import OracleGame
from paper_2112_03804_gb300 import kps, synth
from tests.gpu_util import from_library, library_order, normwise_error, to_library

pytestmark = pytest.mark.gpu

TOL = {torch.float32: 1e-5, torch.bfloat16: 2.0 ** -8, torch.float16: 2.0 ** -10}
# 43 sequences: two items of single rows, one of pairs
TREE = dict(bet_frac=(0.5, 1.0), raise_cap=3, allow_allin=False)


def _spec(cards, seed, tied):
    spec = (synth.river_spec(seed=seed, **TREE) if cards == 2 else
            synth.micro_spec(seed=seed, ranks=12, suits=4, nboard=1, cards_per_hand=1, stack=200.0, **TREE))
    s = np.asarray(spec["strength"])
    order = np.lexsort((np.arange(len(s)), s))
    s = np.empty(len(s), dtype=np.int64)
    s[order] = 10 * np.arange(len(s))
    if tied:
        at = len(s) // 3
        s[order[at:at + 6]] = s[order[at]]
    return dict(spec, strength=s.tolist())


@pytest.mark.parametrize("dt", list(TOL))
@pytest.mark.parametrize("copies", [3, 100])
@pytest.mark.parametrize("tied", [False, True], ids=["no_ties", "long_ties"])
@pytest.mark.parametrize("cards", [1, 2])
def test_variants(cards, tied, copies, dt):
    base = [_spec(cards, 3, tied), _spec(cards, 4, False)]
    games = [kps.Game(s) for s in base * copies]
    b = kps.Batch(games)
    ors = [OracleGame(s) for s in base]
    orders = [library_order(s["strength"]) for s in base]
    infs = [g.info() for g in games[:2]]
    for transpose in (False, True):
        pin = 0 if transpose else 1
        off = b.offsets(1 - pin)
        vs = [synth.simplex_vectors(o.sequences(pin)["nact"], o.H, 1, seed=9 + i)[0] for i, o in enumerate(ors)]
        flat = np.concatenate([to_library(v, o, i["hs"]).reshape(-1) for v, o, i in zip(vs, orders, infs)] * copies)
        out = torch.full((int(off[-1]),), float("nan"), device="cuda", dtype=dt)
        (b.matvec_AT if transpose else b.matvec_A)(torch.from_numpy(flat).to("cuda", dt), out)
        kps.device_status()
        res = out.double().cpu().numpy()
        assert b.shape({torch.float32: kps.F32, torch.bfloat16: kps.BF16, torch.float16: kps.F16}[dt])["kernel"] == kps.BATCH_STAGED
        parts = [res[off[i]:off[i + 1]] for i in range(len(games))]
        for i, o in enumerate(ors):
            want = (o.matvec_AT if transpose else o.matvec_A)(torch.from_numpy(vs[i]).to(dt).double().numpy()[None])[0]
            got = from_library(parts[i].reshape(-1, infs[i]["hs"]), orders[i], infs[i]["H"])
            assert normwise_error(got, want) <= TOL[dt]
            for k in range(1, copies):
                assert np.array_equal(parts[i], parts[i + 2 * k])
