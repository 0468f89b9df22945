"""First products of one game by several threads at once, each on its own
stream: tables and plans are built once, every thread's result is the one that
a later call gives, bit for bit, whichever kernel runs.
"""
import threading

import pytest

torch = pytest.importorskip("torch")

from paper_2112_03804_gb300 import kps, synth

pytestmark = pytest.mark.gpu

THREADS = 8


@pytest.mark.parametrize("dt,kernel", [(torch.float32, "tma"), (torch.bfloat16, "tma"), (torch.float64, "f64"),
                                       (torch.float32, "tmem"), (torch.float64, "vec")],
                         ids=["f32", "bf16", "f64", "f32_tmem", "f64_vec"])
def test_first_products_by_threads(dt, kernel, monkeypatch):
    monkeypatch.setenv("KPS_KERNEL", kernel)
    for seed in range(3):
        g = kps.Game(synth.river_spec(seed=seed))
        inf = g.info()
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        vin = [torch.rand(2, n, inf["hs"], device="cuda", generator=gen).to(dt) for n in (inf["n1"], inf["n2"])]
        outs = [[torch.zeros(2, n, inf["hs"], device="cuda", dtype=dt) for n in (inf["n1"], inf["n2"])]
                for _ in range(THREADS)]
        streams = [torch.cuda.Stream() for _ in range(THREADS)]
        torch.cuda.synchronize()
        start, errors = threading.Barrier(THREADS), []

        def work(t):
            try:
                start.wait()
                kps.matvec_A(g, vin[1], outs[t][0], 2, stream=streams[t])
                kps.matvec_AT(g, vin[0], outs[t][1], 2, stream=streams[t])
            except Exception as e:      # reported by the main thread
                errors.append(e)

        threads = [threading.Thread(target=work, args=(t,)) for t in range(THREADS)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not errors
        torch.cuda.synchronize()
        kps.device_status()
        assert g.kernel(0) == kernel and g.kernel(1) == kernel
        want = [torch.zeros_like(o) for o in outs[0]]
        kps.matvec_A(g, vin[1], want[0], 2)
        kps.matvec_AT(g, vin[0], want[1], 2)
        torch.cuda.synchronize()
        for o in outs:
            assert torch.equal(o[0], want[0]) and torch.equal(o[1], want[1])
