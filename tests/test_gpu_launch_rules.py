"""GPU launch rules that may not change a result: the preparation's cluster size (it follows
the number of stars) and the point path's warps (they follow the bins and points). Every
output of a star is compared bit for bit between the launches, and one of them with the
oracle."""
import numpy as np
import pytest

import oracle
from paper_2302_01293_gb300 import qlpbls
from parity import compare_spectrum

pytestmark = pytest.mark.gpu

FIELDS = ("sr", "qidx", "kbin", "s", "r", "snr")


def _regular_star(n, seed, gap=0):
    """n points at 30-minute spacing, `gap` cells missing in the middle, unequal errors."""
    rng = np.random.default_rng(seed)
    k = np.arange(n) + np.where(np.arange(n) >= n // 2, gap, 0)
    t = 2880.0 + k / 48.0
    dy = 1e-3 * rng.uniform(0.7, 1.4, n)
    y = 1.0 + dy * rng.standard_normal(n) - 3e-3 * (np.mod(k, 97) < 5)
    return t, y, dy


def _outputs(stars, params, rho=1.41):
    offs = np.zeros(len(stars) + 1, np.int64)
    offs[1:] = np.cumsum([s[0].shape[0] for s in stars])
    t, y, dy = (np.concatenate([s[i] for s in stars]) for i in range(3))
    plan = qlpbls.Plan(offs, t, y, dy, np.full(len(stars), rho), np.ones(len(stars)), params)
    out = plan.search()
    plan.snr(out)
    assert plan.device_status() == 0
    return plan, {k: out[k].cpu().numpy() for k in FIELDS}


@pytest.mark.parametrize("sum_mode", [qlpbls.SUM_FIXED, qlpbls.SUM_FIXED64])
@pytest.mark.parametrize("n,gap", [(289, 0), (480, 31), (511, 32), (512, 1), (513, 200), (1025, 65), (4097, 33)])
def test_prep_cluster_size(gpu_lib, sum_mode, n, gap):
    star = _regular_star(n, 3 * n + gap, gap)
    params = qlpbls.Params(sum_mode=sum_mode, method=qlpbls.METHOD_CELLS)
    plan, alone = _outputs([star], params)
    assert plan.n_exact_stars == 1
    pl = oracle.plan_star(*star, 1.41, 1.0)
    compare_spectrum(pl, oracle.bls_star(pl), alone, plan.star_slice(0), label=f"n {n} gap {gap}", tight=True)
    other = _regular_star(300, 1)
    for copies in (200, 400, 700, 1300):  # clusters of 8 alone, then 4, 4 or 2, 2 and 1
        if copies * n > 3_000_000 and copies < 1300:
            continue
        first = [other] * (copies - 1)
        plan, got = _outputs(first + [star], params)
        sl = plan.star_slice(copies - 1)
        for k in FIELDS:
            assert np.array_equal(got[k][sl], alone[k][: sl.stop - sl.start]), (copies, k)


@pytest.mark.parametrize("n,span,rho", [(40, 6.0, 1.0), (33, 27.4, 10.0), (900, 27.4, 1.41), (4200, 27.4, 5.0),
                                        (3000, 54.0, 30.0), (11000, 27.4, 1.0)])
@pytest.mark.parametrize("sum_mode", [qlpbls.SUM_FIXED, qlpbls.SUM_PLAIN])
def test_point_path_warps(gpu_lib, n, span, rho, sum_mode):
    rng = np.random.default_rng(n)
    stars = []
    for m in (n, max(2, n // 3)):
        t = 2880.0 + np.sort(rng.uniform(0.0, span, m))
        t[0], t[-1] = 2880.0, 2880.0 + span
        dy = 1e-3 * rng.uniform(0.7, 1.4, m)
        stars.append((t, 1.0 + dy * rng.standard_normal(m), dy))
    ref = None
    for warps in (8, 0):  # as many as fit per item, and a fixed count
        plan, got = _outputs(stars, qlpbls.Params(method=qlpbls.METHOD_POINTS, sum_mode=sum_mode,
                                                  warps_per_block=warps), rho)
        assert plan.work_points > 0
        if ref is None:
            ref = got
        for k in FIELDS:
            assert np.array_equal(got[k], ref[k]), (warps, k)
