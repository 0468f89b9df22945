"""The staged batched kernel's rows and ties: paired rows (fold and call of one
bet in one scan), items of 16 and of 32 rows, which its plan picks by the number of games, and
tie groups of 5 and more hands, with boards of 3 to 5 cards and every storage
type, against the oracle game by game (half precision: on the rounded inputs).
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


def _tied(spec, sizes, seed):
    """Groups of the given sizes at random places of the order."""
    s = np.asarray(spec["strength"])
    order = np.lexsort((np.arange(len(s)), s))
    s = np.empty(len(s), dtype=np.int64)
    s[order] = 10 * np.arange(len(s))
    r = np.random.default_rng(seed)
    for n in sizes:
        a = int(r.integers(0, len(s) - n + 1))
        s[order[a:a + n]] = s[order[a]]
    return dict(spec, strength=s.tolist())


def _specs(copies):
    base = [synth.river_spec(seed=3), _tied(synth.river_spec(seed=4), [5, 9, 6], 1),
            _tied(synth.river_spec(seed=5, nboard=4, bet_frac=(0.33, 0.66, 1.0)), [12], 2),
            synth.river_spec(seed=6, nboard=3, bet_frac=(0.5,), raise_cap=2),
            _tied(synth.river_spec(seed=7, nboard=3), [5, 5], 3),
            synth.micro_spec(seed=8, ranks=6, suits=3, nboard=4)]
    return base, base * copies


@pytest.mark.parametrize("copies", [1, 30, 70])
@pytest.mark.parametrize("dt", list(TOL))
def test_rows_and_ties(copies, dt):
    base, specs = _specs(copies)
    games = [kps.Game(s) for s in specs]
    b = kps.Batch(games)
    ors = [OracleGame(s) for s in base]
    orders = [library_order(s["strength"]) for s in base]
    infs = [g.info() for g in games[:len(base)]]
    for transpose in (False, True):
        pin = 0 if transpose else 1
        off = [b.offsets(p) for p in (0, 1)]
        vs = [synth.simplex_vectors(o.sequences(pin)["nact"], o.H, 1, seed=9 + i)[0] for i, o in enumerate(ors)]
        flat = np.concatenate([to_library(v, o, i["hs"]).reshape(-1) for v, o, i in zip(vs, orders, infs)] * copies)
        vin = torch.from_numpy(flat).to("cuda", dt)
        out = torch.full((int(off[1 - pin][-1]),), float("nan"), device="cuda", dtype=dt)
        (b.matvec_AT if transpose else b.matvec_A)(vin, out)
        kps.device_status()
        res = out.double().cpu().numpy()
        assert np.isfinite(res).all()
        parts = [res[off[1 - pin][i]:off[1 - pin][i + 1]] for i in range(len(specs))]
        for i, o in enumerate(ors):
            want = (o.matvec_AT if transpose else o.matvec_A)(torch.from_numpy(vs[i]).to(dt).double().numpy()[None])[0]
            got = from_library(parts[i].reshape(-1, infs[i]["hs"]), orders[i], infs[i]["H"])
            assert normwise_error(got, want) <= TOL[dt], (copies, i)
            for k in range(1, copies):       # the same game elsewhere in the launch: the same bits
                assert np.array_equal(parts[i], parts[i + k * len(base)])
