"""GPU calls after a device allocation that was refused: the refusal is the failing call's
result alone, and no later call takes it for its own. The device refuses memory it does not
have (nothing is taken), the budget memory it may not hand out."""
import gc

import numpy as np
import pytest

from paper_2302_01293_gb300 import qlpbls
from test_gpu_launch_rules import _outputs, _regular_star

pytestmark = pytest.mark.gpu


def _refused_by_device():
    import torch
    batch = 2 * torch.cuda.get_device_properties(0).total_memory // (4 * 4096)  # its logits alone take twice that
    return lambda: qlpbls.CNN(max_batch=int(batch), length=4096)


def _refused_by_budget():
    def call():
        qlpbls.set_device_budget(qlpbls.device_bytes_held() + 1)
        try:
            qlpbls.CNN(max_batch=1, length=128)
        finally:
            qlpbls.set_device_budget(0)
    return call


@pytest.mark.parametrize("refusal", [_refused_by_device, _refused_by_budget])
def test_calls_after_a_refused_allocation(gpu_lib, refusal):
    import torch
    refused = refusal()
    star = _regular_star(900, 3)
    params = qlpbls.Params(grid_mode=1, coarse_bins=256)
    plan, _ = _outputs([star], params)
    out = plan.search()
    plan.snr(out)
    w = torch.randn(9, 64, 64, device="cuda")
    x = torch.randn(1, 128, 64, device="cuda").to(torch.bfloat16)
    z = torch.randn(2, 256, device="cuda")
    x0 = torch.ones(2, 256, qlpbls.CNN_IN_CH, dtype=torch.bfloat16, device="cuda")
    calls = dict(peaks=lambda: plan.top_peaks(out, 4), tensor=lambda: plan.coarse_tensor(out),
                 statistics=lambda: plan.candidate_stats(out), search=lambda: plan.search(out),
                 snr=lambda: plan.snr(out), pack=lambda: qlpbls.pack_w64(w), topk=lambda: qlpbls.topk(z, x0, 3),
                 conv=lambda: qlpbls.conv64(x, qlpbls.pack_w64(w)), wgrad=lambda: qlpbls.conv64_wgrad(x, x),
                 plan=lambda: _outputs([star], params))
    for name, call in calls.items():
        with pytest.raises(qlpbls.QlpError) as ei:
            refused()
        assert ei.value.code == qlpbls.ERR_NOMEM
        call()
        torch.cuda.synchronize()
        assert plan.device_status() == 0, name


def test_host_call_after_its_chunks_were_refused(gpu_lib):
    """200 stars of a sector: two chunks; within a budget of one plan of all of them the second
    chunk is refused by cudaMalloc and the batch runs as one, with the same result."""
    gc.collect()  # nothing of earlier tests is freed between the counts
    stars = [_regular_star(1250 + s % 50, s) for s in range(200)]
    offs = np.zeros(201, np.int64)
    offs[1:] = np.cumsum([s[0].shape[0] for s in stars])
    t, y, dy = (np.concatenate([s[i] for s in stars]) for i in range(3))
    rho = np.full(200, 1.41)

    def held(lo, hi):
        base, sl = qlpbls.device_bytes_held(), slice(int(offs[lo]), int(offs[hi]))
        plan = qlpbls.Plan(offs[lo: hi + 1] - offs[lo], t[sl], y[sl], dy[sl], rho[lo:hi], np.ones(hi - lo))
        n = qlpbls.device_bytes_held() - base + 21 * plan.n_freq_total + qlpbls.BEST_DTYPE.itemsize * (hi - lo)
        plan.close()
        return n

    slack = 16 * 256  # each buffer starts on a 256-byte boundary
    one = held(0, 200) + slack
    assert held(0, 100) + held(100, 200) > one
    base = qlpbls.device_bytes_held()
    got = []
    for budget in (0, base + one):
        qlpbls.set_device_budget(budget)
        try:
            got.append(qlpbls.run_host(offs, t, y, dy, rho, np.ones(200))["best"])
        finally:
            qlpbls.set_device_budget(0)
    assert np.array_equal(got[0], got[1])
    assert qlpbls.device_bytes_held() == base
