"""The host call's chunks: the same records and spectra as one plan of all stars, and no more
chunks than a batch has work to hide."""
import time

import numpy as np
import pytest

from paper_2302_01293_gb300 import qlpbls
from test_gpu_launch_rules import _regular_star

pytestmark = pytest.mark.gpu


def _batch(n, points, spoil=False):
    stars = [_regular_star(points + s % 7, s) for s in range(n)]
    if spoil:  # time stamps and fluxes that are not numbers, at the ends and between
        for s in range(0, n, 3):
            stars[s][0][: s % 5] = np.nan
            stars[s][1][len(stars[s][1]) - 1 - s % 3:] = np.nan
            stars[s][0][len(stars[s][0]) // 2] = np.inf
    offs = np.zeros(n + 1, np.int64)
    offs[1:] = np.cumsum([s[0].shape[0] for s in stars])
    t, y, dy = (np.concatenate([s[i] for s in stars]) for i in range(3))
    return offs, t, y, dy, np.full(n, 1.41), np.ones(n)


def _one_plan(batch):
    plan = qlpbls.Plan(*batch)
    out = plan.search()
    plan.snr(out)
    return plan, out, plan.best_host(out)


@pytest.mark.parametrize("n,points,spoil", [(199, 1200, False), (200, 1200, True), (450, 1000, True), (1100, 300, False),
                                            (300, 2, False)])
def test_chunks_give_one_plans_result(gpu_lib, n, points, spoil):
    batch = _batch(n, points, spoil)
    plan, out, want = _one_plan(batch)
    nf = plan.n_freq_total
    got = qlpbls.run_host(*batch, sr_capacity=nf + 1)
    assert got["n_freq_total"] == nf
    assert np.array_equal(got["best"], want)
    assert np.array_equal(got["sr"][:nf], out["sr"].cpu().numpy()[:nf])
    assert np.array_equal(got["snr"][:nf], out["snr"].cpu().numpy()[:nf])


@pytest.mark.parametrize("n", [600, 999])
def test_short_light_curves_are_not_slower_than_one_plan(gpu_lib, n):
    """200 points over 4 days: host and device together take a few ms, a chunk 0.4 of its own."""
    batch = _batch(n, 200)
    best = []
    for call in (lambda: _one_plan(batch)[0].close(), lambda: qlpbls.run_host(*batch)):
        v = []
        for _ in range(12):
            t0 = time.perf_counter()
            call()
            v.append(time.perf_counter() - t0)
        best.append(min(v))
    assert best[1] <= 1.15 * best[0]
