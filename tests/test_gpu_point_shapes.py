"""Launch shapes of the point path: how a plan cuts its work may not change a result, and the
shape that the planner chooses may not cost more than a fixed one of 8 warps."""
import numpy as np
import pytest

import oracle
from paper_2302_01293_gb300 import qlpbls
from parity import compare_spectrum
from test_gpu_launch_rules import FIELDS, _outputs

pytestmark = pytest.mark.gpu


def _stars(n, points, span):
    rng = np.random.default_rng(n * points)
    stars = []
    for _ in range(n):
        t = 2880.0 + np.sort(rng.uniform(0.0, span, points))
        t[0], t[-1] = 2880.0, 2880.0 + span
        dy = 1e-3 * rng.uniform(0.7, 1.4, points)
        stars.append((t, 1.0 + dy * rng.standard_normal(points), dy))
    return stars


# short stars (small blocks), one wave of items, bins that leave room for few warps, several tiles
@pytest.mark.parametrize("n,points,span,rho", [(1, 33, 8.0, 1.0), (1, 300, 27.4, 1.41), (2, 1000, 27.4, 5.0),
                                               (6, 900, 20.0, 1.0), (1, 4200, 27.4, 0.5), (1, 11000, 27.4, 1.0)])
@pytest.mark.parametrize("kw", [dict(), dict(sum_mode=qlpbls.SUM_PLAIN), dict(phase_mode=qlpbls.PHASE_FP64)])
def test_items_and_warps_do_not_change_a_result(gpu_lib, n, points, span, rho, kw):
    stars = _stars(n, points, span)
    kw = dict(method=qlpbls.METHOD_POINTS, **kw)
    plan, ref = _outputs(stars, qlpbls.Params(warps_per_block=8, **kw), rho)
    assert plan.work_points > 0
    if points < 1000 and kw.get("sum_mode") != qlpbls.SUM_PLAIN:
        pl = oracle.plan_star(*stars[0], rho, 1.0)
        compare_spectrum(pl, oracle.bls_star(pl), ref, plan.star_slice(0), label=f"{points} points")
    for chunk in (0, 1, 7, 8, 16, 31, 32, 33, 100, 2 ** 31 - 1):
        _, got = _outputs(stars, qlpbls.Params(chunk_freqs=chunk, **kw), rho)
        for k in FIELDS:
            assert np.array_equal(got[k], ref[k]), (chunk, k)


def _ms(stars, params, rho):
    import torch
    offs = np.zeros(len(stars) + 1, np.int64)
    offs[1:] = np.cumsum([s[0].shape[0] for s in stars])
    plan = qlpbls.Plan(offs, *(np.concatenate([s[i] for s in stars]) for i in range(3)), np.full(len(stars), rho),
                       np.ones(len(stars)), params)
    out = plan.search()
    best = np.inf
    for _ in range(20):
        e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        torch.cuda.synchronize()
        e0.record()
        plan.search(out)
        e1.record()
        e1.synchronize()
        best = min(best, e0.elapsed_time(e1))
    return best


@pytest.mark.parametrize("n,points,span,rho,kw", [
    (1, 300, 27.4, 1.41, {}), (1, 14000, 27.4, 1.0, {}), (1, 14000, 27.4, 1.0, dict(phase_mode=qlpbls.PHASE_FP64)),
    (30, 500, 27.4, 1.0, dict(sum_mode=qlpbls.SUM_PLAIN)), (8, 300, 27.4, 5.0, dict(chunk_freqs=8)),
    (60, 900, 15.0, 1.0, dict(chunk_freqs=16)), (1, 9000, 27.4, 1.0, dict(tile_points=512))])
def test_chosen_shape_is_not_slower_than_eight_warps(gpu_lib, n, points, span, rho, kw):
    stars = _stars(n, points, span)
    kw = dict(method=qlpbls.METHOD_POINTS, **kw)
    fixed = _ms(stars, qlpbls.Params(warps_per_block=8, **kw), rho)
    assert _ms(stars, qlpbls.Params(**kw), rho) <= 1.2 * fixed
