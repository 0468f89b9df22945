"""A plan whose device memory is not to be had: the product runs on the kernel
that needs less, reports no error of the allocation that failed, and a later
call, with memory there, takes the plan's kernel.  The shortage is made by
the library's test hook (KPS_TEST_FAIL_ALLOC=n: allocations of n bytes and more
ask for 2^60 bytes, which cudaMalloc refuses).  Tolerances as for the other products:
1e-12 FP64, 1e-5 FP32, 2^-8 BF16, 2^-10 FP16 normwise, on the rounded inputs.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.oracle import OracleGame
from paper_2112_03804_gb300 import kps, synth
from tests.gpu_util import from_library, library_order, normwise_error, to_library

pytestmark = pytest.mark.gpu

TOL = {torch.float64: 1e-12, torch.float32: 1e-5, torch.bfloat16: 2.0 ** -8, torch.float16: 2.0 ** -10}
DTS = list(TOL)
CODE = {torch.float64: kps.F64, torch.float32: kps.F32, torch.bfloat16: kps.BF16, torch.float16: kps.F16}
PLAN_BYTES = "16384"          # below a river game's plan, above its tile tables
SCRATCH_BYTES = "10000000"    # below the staged batched kernel's scratch area, above a small solver's arrays


def _check(got, spec, info, v, dt):
    og = OracleGame(spec)
    want = og.matvec_A(torch.from_numpy(v).to(dt).double().numpy())
    assert normwise_error(from_library(got, library_order(spec["strength"]), info["H"]), want) <= TOL[dt]


@pytest.mark.parametrize("dt", DTS)
def test_single_game(dt, monkeypatch):
    spec = synth.river_spec(seed=3)
    g = kps.Game(spec)
    g.upload()
    inf = g.info()
    v = synth.simplex_vectors(g.sequences(1)["nact"], inf["H"], 3, seed=4)
    vin = torch.from_numpy(to_library(v, library_order(spec["strength"]), inf["hs"])).to("cuda", dt)
    for short in (True, True, False):
        if short:
            monkeypatch.setenv("KPS_TEST_FAIL_ALLOC", PLAN_BYTES)
        else:
            monkeypatch.delenv("KPS_TEST_FAIL_ALLOC")
        out = torch.full((3, inf["n1"], inf["hs"]), float("nan"), device="cuda", dtype=dt)
        kps.matvec_A(g, vin, out, 3)
        kps.device_status()
        assert g.kernel(0) == ({torch.float64: "vec"}.get(dt, "tmem") if short else
                               {torch.float64: "f64"}.get(dt, "tma"))
        _check(out.double().cpu().numpy(), spec, inf, v, dt)


@pytest.mark.parametrize("dt", DTS)
def test_batch(dt, monkeypatch):
    spec = synth.river_spec(seed=3)
    g = kps.Game(spec)
    b = kps.Batch([g])
    inf = g.info()
    v = synth.simplex_vectors(g.sequences(1)["nact"], inf["H"], 1, seed=4)
    vin = torch.from_numpy(to_library(v, library_order(spec["strength"]), inf["hs"])).to("cuda", dt).reshape(-1)
    for short in (True, True, False):
        if short:
            monkeypatch.setenv("KPS_TEST_FAIL_ALLOC", PLAN_BYTES)
        else:
            monkeypatch.delenv("KPS_TEST_FAIL_ALLOC")
        out = torch.full((1, inf["n1"], inf["hs"]), float("nan"), device="cuda", dtype=dt)
        b.matvec_A(vin, out)
        kps.device_status()
        kernel = b.shape(CODE[dt])["kernel"]
        assert kernel == (kps.BATCH_TMEM if short else kps.BATCH_F64 if dt == torch.float64 else kps.BATCH_STAGED)
        _check(out.double().cpu().numpy(), spec, inf, v, dt)


def test_solver(monkeypatch):
    """A solver made while the staged kernel's scratch area is not to be had
    steps on the other kernel, in its captured iterations too, and goes on when
    it is."""
    b = kps.Batch([kps.Game(synth.river_spec(seed=3))])
    monkeypatch.setenv("KPS_TEST_FAIL_ALLOC", SCRATCH_BYTES)
    s = kps.Solver(b, kps.F32)
    assert b.shape(kps.F32)["kernel"] == kps.BATCH_TMEM
    s.step(5)
    s.status()
    monkeypatch.delenv("KPS_TEST_FAIL_ALLOC")
    s.step(5)
    s.step(7)
    s.status()
    assert b.shape(kps.F32)["kernel"] == kps.BATCH_STAGED
    e, f = (torch.zeros(1, dtype=torch.float64, device="cuda") for _ in range(2))
    s.exploitability(e)
    s.exploitability_estimate(f)
    s.status()
    t = kps.Solver(kps.Batch(b.games), kps.F32)
    t.step(17)
    ref = torch.zeros(1, dtype=torch.float64, device="cuda")
    t.exploitability(ref)
    t.status()
    # FP32 rounding of the products, amplified by 17 iterations
    assert abs(float(e - f)) <= 1e-4 and abs(float(e - ref)) <= 1e-2 * float(ref)


def test_solver_shares_the_batch_plans():
    """A solver's products (plain rows) run on the batch's own plans: creating
    one takes its state's memory, not a second set of records and scratch areas
    (20 MB each)."""
    def make():
        b = kps.Batch([kps.Game(synth.river_spec(seed=3))])
        x = torch.zeros(int(b.offsets(1)[-1]), device="cuda")
        b.matvec_A(x, torch.zeros(int(b.offsets(0)[-1]), device="cuda"))
        torch.cuda.synchronize()
        return b

    keep = kps.Solver(make(), kps.F32)          # loads every kernel
    keep.step(2)
    torch.cuda.synchronize()
    b = make()
    before, _ = torch.cuda.mem_get_info()
    s = kps.Solver(b, kps.F32)
    torch.cuda.synchronize()
    after, _ = torch.cuda.mem_get_info()
    assert before - after < 16 << 20
    s.step(2)
    s.status()
