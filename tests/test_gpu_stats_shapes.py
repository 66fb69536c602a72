"""The statistics kernel with two warps per 32 chains (few stars) and with one (many): the same
records bit for bit, at the edges of chains and warps and on windows of few points."""
import numpy as np
import pytest

import synth
from paper_2302_01293_gb300 import qlpbls

pytestmark = pytest.mark.gpu


def _edges(equal):
    stars = []
    for n in (40, 63, 64, 65, 127, 128, 129, 511, 512, 513, 575, 577, 1023, 1025, 2000, 4097):
        rng = np.random.default_rng(n)
        t = synth.T_START + np.arange(n) / 48.0
        dy = np.full(n, 1e-3) if equal else 1e-3 * rng.uniform(0.7, 1.4, n)
        period = min(1.37, n / 48.0 / 3.0)
        y = 1.0 + dy * rng.standard_normal(n)
        y -= 8e-3 * synth.box_mask(t, period, synth.T_START + 0.3 * period,
                                   synth.circular_duration_days(period, 1.41, 1.0))
        stars.append((t, y, dy))
    return stars


def _records(stars):
    offs = np.zeros(len(stars) + 1, np.int64)
    offs[1:] = np.cumsum([s[0].shape[0] for s in stars])
    plan = qlpbls.Plan(offs, *(np.concatenate([s[i] for s in stars]) for i in range(3)),
                       np.full(len(stars), 1.41), np.ones(len(stars)))
    out = plan.search()
    plan.snr(out)
    st = plan.candidate_stats(out)
    assert plan.device_status() == 0
    return plan.stats_host(st), plan.best_host(out)


@pytest.mark.parametrize("equal", [True, False])
def test_records_do_not_depend_on_the_batch(gpu_lib, equal):
    import torch
    stars = _edges(equal)
    alone, best = _records(stars)
    assert np.count_nonzero(alone["iterations"] > 0) >= 12
    rng = np.random.default_rng(3)
    t = synth.T_START + np.arange(40) / 24.0
    filler = [(t, 1.0 + 1e-3 * rng.standard_normal(40), np.full(40, 1e-3)) for _ in range(50)]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    many, best_many = _records(stars + [filler[i % 50] for i in range(8 * sms)])  # past the rule's line
    k = len(stars)
    assert np.array_equal(best_many[:k], best)
    assert np.array_equal(many[:k].view(np.uint8), alone.view(np.uint8))
    few, _ = _records(filler)
    assert np.array_equal(many[k: k + 50].view(np.uint8), few.view(np.uint8))
