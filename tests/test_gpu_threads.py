"""Launches from two host threads at once, one with small shared-memory needs and one with
large ones: neither may be refused, and both give what they give alone."""
import os
import subprocess
import sys
import threading

import numpy as np
import pytest

from paper_2302_01293_gb300 import qlpbls
from test_gpu_launch_rules import _regular_star

pytestmark = pytest.mark.gpu

ROUNDS = 10000


def _together(calls):
    import torch
    refused = [0] * len(calls)

    def work(i):
        stream = torch.cuda.Stream()
        for _ in range(ROUNDS):
            try:
                calls[i](stream)
            except qlpbls.QlpError:
                refused[i] += 1
        stream.synchronize()

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(calls))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert refused == [0] * len(calls)


def _searched(points, **kw):
    plan = qlpbls.Plan(np.array([0, points], np.int64), *_regular_star(points, points), np.array([1.41]),
                       np.ones(1), qlpbls.Params(**kw))
    out = plan.search()
    plan.snr(out)
    return plan, out, {k: out[k].cpu().numpy() for k in ("sr", "snr", "best")}


def _check(case):
    plan, out, alone = case
    assert plan.device_status() == 0
    for k, v in alone.items():
        assert np.array_equal(out[k].cpu().numpy(), v), k


def test_snr_launches(gpu_lib):
    cases = [_searched(n) for n in (100, 3000)]
    _together([lambda st, c=c: c[0].snr(c[1], stream=st) for c in cases])
    for c in cases:
        _check(c)


def test_topk_launches(gpu_lib):
    import torch
    topk, check, calls, rows = qlpbls.lib().qlp_cnn_topk, qlpbls._check, [], []
    for length in (64, 30000):
        z = torch.randn(2, length, device="cuda", generator=torch.Generator(device="cuda").manual_seed(length))
        x0 = torch.ones(2, length, qlpbls.CNN_IN_CH, dtype=torch.bfloat16, device="cuda")
        bins = torch.empty(2, 2, dtype=torch.int32, device="cuda")
        rows.append((z, x0, bins))
        args = (z.data_ptr(), x0.data_ptr(), 2, length, 2, bins.data_ptr())  # the library's own call: no allocation
        calls.append(lambda st, a=args: check(topk(*a, qlpbls._stream_ptr(st)), "qlp_cnn_topk"))
    torch.cuda.synchronize()
    _together(calls)
    for z, _, bins in rows:
        assert torch.equal(bins.long(), torch.topk(z, 2).indices)


@pytest.mark.parametrize("kw", [dict(method=qlpbls.METHOD_POINTS), dict(method=qlpbls.METHOD_CELLS)])
def test_search_launches(gpu_lib, kw):
    cases = [_searched(n, **kw) for n in (300, 3000)]
    _together([lambda st, c=c: c[0].search(c[1], stream=st) for c in cases])
    for c in cases:
        _check(c)


def test_first_tensor_core_calls_of_a_process(gpu_lib):
    """Eight host threads whose first CUDA call of all needs the driver's tensor-map encoder, in
    processes of their own: each has to make its context current, and the one that looks the
    encoder up must not leave the others without it."""
    code = """
import threading, torch
from paper_2302_01293_gb300 import qlpbls
x = torch.randint(-1, 2, (1, 128, 64), device="cuda").to(torch.bfloat16)
wp = qlpbls.pack_w64(torch.randn(9, 64, 64, device="cuda"))
L, gate, bad = qlpbls.lib(), threading.Barrier(8), []
ys, errs = [torch.empty_like(x) for _ in range(4)], torch.zeros(8, dtype=torch.int32, device="cuda")
ws = [torch.empty(L.qlp_cnn_wgrad64_workspace(1, 128), device="cuda") for _ in range(4)]
dws = [torch.empty(9 * 64 * 64 + 64, device="cuda") for _ in range(4)]
streams = [torch.cuda.Stream() for _ in range(8)]
calls = []
for i in range(8):
    tail = (errs[i:].data_ptr(), qlpbls._stream_ptr(streams[i]))
    if i < 4:
        calls.append((L.qlp_cnn_conv64, (x.data_ptr(), wp.data_ptr(), None, None, ys[i].data_ptr(), 1, 128, 1) + tail))
    else:
        calls.append((L.qlp_cnn_conv64_wgrad, (x.data_ptr(), x.data_ptr(), ws[i - 4].data_ptr(),
                                               dws[i - 4].data_ptr(), 1, 128) + tail))
torch.cuda.synchronize()
def work(i):
    gate.wait()
    if calls[i][0](*calls[i][1]):
        bad.append(i)
threads = [threading.Thread(target=work, args=(i,)) for i in range(8)]
[t.start() for t in threads]
[t.join() for t in threads]
torch.cuda.synchronize()
assert not bad, bad
assert not errs.any()
assert all(torch.equal(y, ys[0]) for y in ys) and all(torch.equal(d, dws[0]) for d in dws)
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    for _ in range(4):
        run = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
        assert run.returncode == 0, run.stderr[-2000:]
