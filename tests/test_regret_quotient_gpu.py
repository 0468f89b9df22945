"""The solver's regret matching against the division, bit for bit, over the
exponent range: a checkpoint is loaded whose player-1 regrets are drawn here
(one large regret a node, the others down to the smallest subnormal, zeros and,
for a few hands, sums past 2^100) and whose player-2 strategy is zero, so that
player 1's values are zero, the update leaves the regrets as they are and the
next strategy is made of the quotients alone: x[sigma] = x[parent] R / sum R,
each step rounded once, as numpy rounds it.
"""
import struct

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2112_03804_gb300 import kps, synth

pytestmark = pytest.mark.gpu

HEADER = 120        # kps_solver_save: magic, 4 int32, 6 doubles, 7 64-bit integers


def _regrets(r, node, H, dt):
    """Per node one regret in [1, 16) of a power of two shared by the hand,
    the others spread over all exponents below it, a tenth of them zero."""
    low = -149 if dt == np.float32 else -1074
    top = r.integers(0, 41, size=H)      # above the noise floor
    top[::50] = 110                                     # past the range of the shared reciprocal
    out = np.zeros((len(node), H))
    for k in range(int(node.max()) + 1):
        rows = np.flatnonzero(node == k)
        big = r.integers(0, len(rows), size=H)
        for j, s in enumerate(rows):
            e = r.integers(low, top + 1)
            v = np.ldexp(r.uniform(1.0, 2.0, size=H), e)
            v[r.uniform(size=H) < 0.1] = 0.0
            out[s] = np.where(big == j, np.ldexp(r.uniform(1.0, 16.0, size=H), top), v)
    return out.astype(dt)


@pytest.mark.parametrize("code,dt", [(kps.F32, np.float32), (kps.F64, np.float64)], ids=["f32", "f64"])
@pytest.mark.parametrize("menu", [(0.5, 1.0), (0.25, 0.5, 0.75, 1.0, 1.5, 2.0)], ids=["few", "many_actions"])
def test_quotients_round_as_the_division(code, dt, menu):
    g = kps.Game(synth.river_spec(seed=2, bet_frac=menu, raise_cap=2))
    b = kps.Batch([g])
    s = kps.Solver(b, code)
    inf, seq = g.info(), g.sequences(0)
    n, hs, H, es = inf["n1"], inf["hs"], inf["H"], np.dtype(dt).itemsize
    R = np.zeros((n, hs), dt)
    R[:, :H] = _regrets(np.random.default_rng(7), seq["node"], H, dt)
    # header; then per player regrets, strategy sums, strategy, initial strategy
    state = bytearray(s.save())
    len1, len2 = n * hs, inf["n2"] * hs
    assert struct.unpack_from("<2q", state, 88) == (len1, len2) and len(state) == HEADER + (len1 + len2) * (3 * es + 4)
    state[HEADER:HEADER + len1 * es] = R.tobytes()
    y = HEADER + len1 * (3 * es + 4) + 2 * len2 * es
    state[y:y + len2 * es] = bytes(len2 * es)
    s.load(bytes(state))
    s.step(1)
    x = torch.zeros(len1, device="cuda", dtype=torch.float32 if dt == np.float32 else torch.float64)
    s.strategy(x, None)
    s.status()
    got = x.cpu().numpy().reshape(n, hs)[:, :H]
    want = np.zeros((n, H), dt)
    for k in range(int(seq["node"].max()) + 1):
        rows = np.flatnonzero(seq["node"] == k)
        tot = np.zeros(H, dt)
        for row in rows:
            tot = tot + R[row, :H]
        for row in rows:
            q = R[row, :H] / tot
            par = seq["parent"][row]
            want[row] = q if par < 0 else want[par] * q
    assert np.array_equal(got, want)
