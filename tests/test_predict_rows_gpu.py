"""The predictor's first-layer products of a game are the same sums whether the
batch has few rows (one thread an output) or many (tiles): a game's predictions
do not depend on the batch it is in, bit for bit.
"""
import pytest

torch = pytest.importorskip("torch")

from paper_2112_03804_gb300 import kps, synth

pytestmark = pytest.mark.gpu


def test_predictions_do_not_depend_on_the_batch():
    games = [kps.Game(synth.river_spec(seed=3 + i, raise_cap=1 + i % 2)) for i in range(3)]
    m = kps.MLP(seed=2)
    got = []
    for copies in (1, 86):                       # 6 and 516 rows of game features
        b = kps.Batch(games * copies)
        beh = [torch.zeros(int(b.offsets(p)[-1]), device="cuda") for p in (0, 1)]
        kps.warm_predict(b, m, beh[0], beh[1])
        kps.device_status()
        got.append(beh)
    for one, many in zip(*got):
        assert torch.isfinite(one).all() and float(one.abs().sum()) > 0
        assert torch.equal(many.view(86, -1), one.expand(86, -1))
