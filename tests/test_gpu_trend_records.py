"""S/N from given trend records: the node counts a record can hold, and counts that none can,
which are read as a record without a trend."""
import numpy as np
import pytest

from paper_2302_01293_gb300 import qlpbls
from test_gpu_launch_rules import _regular_star

pytestmark = pytest.mark.gpu

NODES = 40  # a record's room


def _score(counts):
    import torch
    stars = [_regular_star(900 + i, i) for i in range(len(counts))]
    offs = np.zeros(len(stars) + 1, np.int64)
    offs[1:] = np.cumsum([s[0].shape[0] for s in stars])
    plan = qlpbls.Plan(offs, *(np.concatenate([s[i] for s in stars]) for i in range(3)),
                       np.full(len(stars), 1.41), np.ones(len(stars)))
    out = plan.search()
    rng = np.random.default_rng(4)
    rec = np.zeros((len(stars), qlpbls.TREND_DOUBLES))
    for s, c in enumerate(counts):
        f = plan.freqs[plan.star_slice(s)]
        rec[s, 0], rec[s, 1] = c, 2.5e-6
        rec[s, 4: 4 + NODES] = np.sort(rng.uniform(f[0], f[-1], NODES))
        rec[s, 4 + NODES: 4 + 2 * NODES] = rng.uniform(1e-5, 1e-4, NODES)
    plan.snr(out, trend_in=torch.from_numpy(rec.reshape(-1)).cuda())
    assert plan.device_status() == 0
    return plan, out["sr"].cpu().numpy().astype(np.float64), out["snr"].cpu().numpy(), plan.best_host(out), rec


def test_records_of_one_to_forty_nodes(gpu_lib):
    counts = [1, 2, 3, 17, 39, 40]
    plan, sr, snr, best, rec = _score(counts)
    for s, c in enumerate(counts):
        sl = plan.star_slice(s)
        f = plan.freqs[sl]
        tr = np.interp(f, rec[s, 4: 4 + c], rec[s, 4 + NODES: 4 + NODES + c])
        want = (sr[sl] - tr) / rec[s, 1]
        # one FP32 rounding; FP64 rounding of the values that meet, scaled by sigma
        slope = np.max(np.abs(np.diff(rec[s, 4 + NODES: 4 + NODES + c]) / np.diff(rec[s, 4: 4 + c]))) if c > 1 else 0.0
        tol = 2.0 ** -23 * np.abs(want) + 8 * 2.0 ** -52 * (np.abs(sr[sl]) + 1e-4 + slope * f) / rec[s, 1]
        assert np.all(np.abs(snr[sl] - want) <= tol), c
        assert best[s]["f_idx"] == int(np.argmax(snr[sl])) and best[s]["status"] == 0


def test_counts_that_no_record_holds(gpu_lib):
    counts = [0, -3, 41, 84, 1e9, -1e300, np.inf, np.nan, 12]
    plan, _, snr, best, _ = _score(counts)
    for s, c in enumerate(counts[:-1]):
        assert best[s]["f_idx"] == -1 and best[s]["status"] == qlpbls.STAR_ZERO_MAD, c
        assert not snr[plan.star_slice(s)].any(), c
    assert best[len(counts) - 1]["f_idx"] >= 0 and snr[plan.star_slice(len(counts) - 1)].any()
