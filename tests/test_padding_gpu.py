"""Padding entries of batch vectors (hands H .. hs - 1 of a row) hold anything
on input and are zero on output, on every batched kernel: products of vectors
whose padding is NaN equal, bit for bit, those whose padding is zero.  The
exploitability estimate reads FP32 averages that share their buffers with the FP64
ones of kps_solver_exploitability, so its padding holds whatever those left:
it has to agree with the FP64 value (FP32 rounding, about 1e-6 of values below
100 initial pots) after it.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2112_03804_gb300 import kps, synth

pytestmark = pytest.mark.gpu

TDT = {kps.F64: torch.float64, kps.F32: torch.float32, kps.BF16: torch.bfloat16, kps.F16: torch.float16}


def _one_card(seed):
    return synth.micro_spec(seed=seed, ranks=12, suits=4, nboard=1, cards_per_hand=1)


def _tied(seed, n):
    spec = synth.river_spec(seed=seed)
    s = np.asarray(spec["strength"])
    order = np.lexsort((np.arange(len(s)), s))
    s[order] = 2 * np.arange(len(s))
    s[order[300:300 + n]] = s[order[300]]
    return dict(spec, strength=s.tolist())


MIXES = {
    "river": lambda: [synth.river_spec(seed=s, nboard=nb) for s, nb in ((3, 5), (4, 4), (5, 3))],
    "small": lambda: [synth.micro_spec(seed=s, ranks=6, suits=4, nboard=3) for s in range(5)],
    "long_ties": lambda: [synth.river_spec(seed=3), _tied(4, 9), _tied(5, 30)],
    "many": lambda: [synth.river_spec(seed=s % 7, raise_cap=2) for s in range(120)],
    "one_card": lambda: [_one_card(s) for s in range(3)],
}


def _vectors(b, games, p, dt):
    """A random batch vector of player p with zero padding, and its padding."""
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    off = b.offsets(p)
    pad = torch.zeros(int(off[-1]), dtype=torch.bool, device="cuda")
    for i, game in enumerate(games):
        inf = game.info()
        pad[off[i]:off[i + 1]].view(-1, inf["hs"])[:, inf["H"]:] = True
    v = torch.rand(int(off[-1]), device="cuda", generator=g)
    return v.masked_fill(pad, 0.0).to(dt), pad


@pytest.mark.parametrize("dt", list(TDT), ids=["f64", "f32", "bf16", "f16"])
@pytest.mark.parametrize("mix", list(MIXES))
def test_batch_padding_is_ignored(mix, dt):
    games = [kps.Game(s) for s in MIXES[mix]()]
    b = kps.Batch(games)
    shapes = [b.shape(dt)]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    shapes += [dict(warps=w, grid=sms, schedule=0, kernel=kps.BATCH_TMEM) for w in (2, 4, 8)]
    for k, sh in enumerate(shapes):
        try:
            b.set_shape(dt, sh["warps"], sh["grid"], sh["schedule"], sh["kernel"])
        except kps.KpsError as e:
            assert k > 0 and e.status == kps.ENOTSUP     # a warp count these games do not fit
            continue
        for p in (0, 1):
            v, pad = _vectors(b, games, p, TDT[dt])
            assert int(pad.sum()) > 0
            out = [torch.full((int(b.offsets(1 - p)[-1]),), float("nan"), device="cuda", dtype=TDT[dt])
                   for _ in range(2)]
            for o, x in zip(out, (v, v.masked_fill(pad, float("nan")))):
                (b.matvec_A if p == 1 else b.matvec_AT)(x, o)
            kps.device_status()
            assert torch.isfinite(out[0]).all()
            assert torch.equal(out[0], out[1])


@pytest.mark.parametrize("dt", list(TDT), ids=["f64", "f32", "bf16", "f16"])
@pytest.mark.parametrize("mix", ["river", "small"])
def test_estimate_after_the_exact_value(mix, dt):
    b = kps.Batch([kps.Game(s) for s in MIXES[mix]()])
    s = kps.Solver(b, dt)
    e, f = (torch.zeros(len(b.games), dtype=torch.float64, device="cuda") for _ in range(2))
    for _ in range(8):
        s.step(5)
        s.exploitability(e)
        s.exploitability_estimate(f)
        s.status()
        assert torch.isfinite(f).all()
        assert float((e - f).abs().max()) <= 1e-4
