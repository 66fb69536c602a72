"""GPU work splits that may not change a result: the windows an exact table is cut into,
the CTAs of a weight gradient, and the warps and chains of the candidate statistics."""
import numpy as np
import pytest

import synth
from paper_2302_01293_gb300 import qlpbls
from test_gpu_launch_rules import _outputs, _regular_star
from test_gpu_stats import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,gap", [(700, 0), (1300, 2000), (4097, 33)])
@pytest.mark.parametrize("window", [32, 64, 352, 2048])
def test_windowed_table_is_the_whole_table(gpu_lib, n, gap, window):
    """Windows shorter than a cycle, longer than one, with empty cells and a short last one:
    the integer bin sums, and so every output, are the whole 64-bit table's."""
    star = _regular_star(n, n + gap, gap)
    kw = dict(sum_mode=qlpbls.SUM_FIXED64, method=qlpbls.METHOD_CELLS)
    plan, whole = _outputs([star], qlpbls.Params(cell_window=1 << 20, **kw))
    assert plan.n_exact_stars == 1
    plan, got = _outputs([star], qlpbls.Params(cell_window=window, **kw))
    assert plan.n_exact_stars == 1
    for k in whole:
        assert np.array_equal(got[k], whole[k]), k


@pytest.mark.parametrize("batch,length", [(1, 128), (151, 128), (152, 128), (153, 128), (77, 256), (304, 128),
                                          (305, 128)])
def test_weight_gradient_ctas(gpu_lib, batch, length):
    """Whole numbers up to 2: every sum is below 2^24, so FP32 holds it exactly in any order."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(batch)
    dy, x = (torch.randint(-2, 3, (batch, length, 64), device="cuda", generator=gen).to(torch.bfloat16)
             for _ in range(2))
    dw, db = qlpbls.conv64_wgrad(dy, x)
    d64, x64 = dy.double(), torch.nn.functional.pad(x.double(), (0, 0, 4, 4))
    want = torch.stack([torch.einsum("blo,bli->oi", d64, x64[:, k: k + length]) for k in range(9)])
    assert torch.equal(dw.double(), want)
    assert torch.equal(db.double(), d64.sum((0, 1)))


@pytest.mark.parametrize("n", [511, 512, 513, 575, 577, 1023, 1025, 2000])
@pytest.mark.parametrize("equal", [True, False])
def test_statistics_at_the_edges_of_chains_and_warps(gpu_lib, n, equal):
    rng = np.random.default_rng(n)
    t = synth.T_START + np.arange(n) / 48.0
    dy = np.full(n, 1e-3) if equal else 1e-3 * rng.uniform(0.7, 1.4, n)
    period = 1.37
    y = 1.0 + dy * rng.standard_normal(n)
    y -= 8e-3 * synth.box_mask(t, period, synth.T_START + 0.4, synth.circular_duration_days(period, 1.41, 1.0))
    _check(synth._assemble("edges", [t], [y], [dy], [1.41], [1.0], [True], [period], [0.0], [8e-3], [0.1]))


@pytest.mark.parametrize("n,rho", [(11900, 5.0), (16000, 1.0), (30001, 2.0)])
@pytest.mark.parametrize("sum_mode", [qlpbls.SUM_FIXED, qlpbls.SUM_PLAIN])
def test_point_path_warps_over_several_tiles(gpu_lib, n, rho, sum_mode):
    """Stars longer than one tile of points: as many warps as an item's bins leave room for,
    and a fixed count of 8, whose tile is the same."""
    rng = np.random.default_rng(n)
    stars = []
    for m in (n, 4000):
        t = 2880.0 + np.sort(rng.uniform(0.0, 27.4, m))
        t[0], t[-1] = 2880.0, 2907.4
        dy = 1e-3 * rng.uniform(0.7, 1.4, m)
        stars.append((t, 1.0 + dy * rng.standard_normal(m), dy))
    ref = None
    for warps in (8, 0):
        plan, got = _outputs(stars, qlpbls.Params(method=qlpbls.METHOD_POINTS, sum_mode=sum_mode,
                                                  warps_per_block=warps), rho)
        if ref is None:
            ref = got
        for k in ref:
            assert np.array_equal(got[k], ref[k]), k


def test_host_call_in_chunks_within_the_budget_of_one(gpu_lib):
    """250 stars run in two chunks; where the budget holds the buffers of one plan of all of
    them, but not of two, in one, with the same result."""
    b = synth.tiny_batch(n_stars=250, seed=3, n_min=200, n_max=400, span_days=8.0)

    def held(lo, hi):
        """Bytes of a plan of stars lo .. hi - 1 and its outputs, and the best records."""
        at0, base = int(b.offsets[lo]), qlpbls.device_bytes_held()
        sl = slice(at0, int(b.offsets[hi]))
        plan = qlpbls.Plan(b.offsets[lo: hi + 1] - at0, b.t[sl], b.y[sl], b.dy[sl], b.rho[lo:hi], b.rstar[lo:hi])
        out = plan.search()
        plan.snr(out)
        best = plan.best_host(out)
        n = qlpbls.device_bytes_held() - base + 21 * plan.n_freq_total + qlpbls.BEST_DTYPE.itemsize * (hi - lo)
        del out
        plan.close()
        return n + 16 * 256, best  # each buffer starts on a 256-byte boundary

    one, want = held(0, 250)
    assert held(0, 125)[0] + held(125, 250)[0] > one + 16 * 256
    base = qlpbls.device_bytes_held()
    for budget in (base + one, 0):
        qlpbls.set_device_budget(budget)
        try:
            got = qlpbls.run_host(b.offsets, b.t, b.y, b.dy, b.rho, b.rstar)["best"]
        finally:
            qlpbls.set_device_budget(0)
        assert np.array_equal(got, want)
    assert qlpbls.device_bytes_held() == base
