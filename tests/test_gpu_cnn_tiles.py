"""The network's kernels where a CTA walks several tiles: seams between tiles of a sample, ring
buffers and accumulators used again, short last tiles. Every layer on the GPU's own stored
tensors against FP64 (torch), element by element, as test_gpu_cnn.py does at one tile per CTA."""
import math

import numpy as np
import pytest

from oracle import cnn as oc
from paper_2302_01293_gb300 import qlpbls

pytestmark = pytest.mark.gpu

U23 = 2.0 ** -23
SMS = 152  # of a GB300


def _shift(x, k):
    import torch
    s = k - 4
    pad = torch.nn.functional.pad(x, (0, 0, max(-s, 0), max(s, 0)))
    return pad[:, max(s, 0): max(s, 0) + x.shape[1]]


def _conv(x, W, b=0.0):
    return sum(_shift(x, k) @ W[k].T for k in range(9)) + b


def _conv_back(x, W, dy):
    """dW, db, dx of conv(x, W, b)."""
    import torch
    flat = dy.reshape(-1, dy.shape[2])
    dW = torch.stack([flat.T @ _shift(x, k).reshape(-1, x.shape[2]) for k in range(9)])
    dx = sum(_shift(dy, 8 - k) @ W[k] for k in range(9))
    return dW, flat.sum(0), dx


def _check_bf16(g, z, e, keep, label):
    import torch
    lo, hi = (torch.where(keep, v, torch.zeros_like(v)).to(torch.bfloat16).double() for v in (z - e, z + e))
    bad = (g < lo) | (g > hi)
    assert not bool(bad.any()), f"{label}: {int(bad.sum())} of {g.numel()}, first at {bad.nonzero()[0].tolist()}"


def _check(g, z, e, label):
    bad = ~((g - z).abs() <= e)
    assert not bool(bad.any()), (f"{label}: {int(bad.sum())} of {g.numel()}, first at {bad.nonzero()[0].tolist()}, "
                                 f"worst {float(((g - z).abs() / e).max())} of the bound")


# one tile and one of 8 rows; two seams, the last tile of 144 rows; 11 tiles a CTA of every kernel;
# more one-tile samples than CTAs
@pytest.mark.parametrize("B,L", [(2, 512), (3, 1152), (305, 640), (500, 128)])
def test_network_over_several_tiles(gpu_lib, B, L):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(B * L)
    x0 = torch.randn(B, L, qlpbls.CNN_IN_CH, device="cuda", generator=gen)
    x0[..., 1] = (torch.rand(B, L, device="cuda", generator=gen) > 0.1).float()
    x0 = x0.to(torch.bfloat16)
    labels = (torch.rand(B, L, device="cuda", generator=gen) < 0.02).float()
    params = oc.init_params(3).astype(np.float32)
    net = qlpbls.CNN(max_batch=B, length=L, seed=1)
    net.set_params(params)
    net.backward(x0, labels, 30.0)
    p = {k: torch.from_numpy(v).cuda() for k, v in oc.unflatten(params.astype(np.float64)).items()}
    for k in range(2, 6):  # as the tensor cores use them
        p[f"W{k}"] = p[f"W{k}"].to(torch.bfloat16).double()
    take = lambda which, k: torch.from_numpy(net.tensor(which, k, B)).cuda().double()
    act = {0: x0.double(), **{k: take(qlpbls.CNN_ACT, k) for k in range(1, 6)}}
    gact = {k: take(qlpbls.CNN_GACT, k) for k in range(1, 6)}
    logit, dlogit = take(qlpbls.CNN_LOGIT, 0), take(qlpbls.CNN_DLOGIT, 0)
    _, grad = net.params(with_grads=True)
    g = {k: torch.from_numpy(v).cuda() for k, v in oc.unflatten(grad.astype(np.float64)).items()}

    for k in range(1, 6):
        n = 9 * act[k - 1].shape[2] + 1
        z = _conv(act[k - 1], p[f"W{k}"], p[f"b{k}"])
        e = n * U23 * _conv(act[k - 1].abs(), p[f"W{k}"].abs(), p[f"b{k}"].abs())
        lo, hi = ((z + s * e).clamp(min=0.0).to(torch.bfloat16).double() for s in (-1, 1))
        bad = (act[k] < lo) | (act[k] > hi)
        assert not bool(bad.any()), f"layer {k} output: {int(bad.sum())}, first at {bad.nonzero()[0].tolist()}"
    W6, b6 = p["W6"], p["b6"]
    _check(logit, _conv(act[5], W6, b6)[..., 0], 577 * U23 * _conv(act[5].abs(), W6.abs(), b6.abs())[..., 0], "logits")

    # FP32 roundings on the way to a weight gradient: a thread's or an accumulator's chain (16
    # products and a sum per matrix instruction), then the CTAs' parts, eight side by side
    tiles = B * L // 128
    each = math.ceil(tiles / min(tiles, SMS))
    joined = 8 + SMS // 8 + 1 + 8
    d = dlogit[..., None]
    dW, db, dx = _conv_back(act[5], W6, d)
    aW, ab, ax = _conv_back(act[5].abs(), W6.abs(), d.abs())
    chain = 8 * math.ceil(B * L / 64 / min(B * L // 64, 3 * SMS)) + 2 + 4 + 3 * joined
    _check(g["W6"], dW, chain * U23 * aW, "W6 gradient")
    _check(g["b6"], db, chain * U23 * ab, "b6 gradient")
    _check_bf16(gact[5], dx, 10 * U23 * ax, act[5] > 0, "layer 5 pre-activation gradient")
    for k in range(5, 0, -1):
        W = p[f"W{k}"]
        dW, db, dx = _conv_back(act[k - 1], W, gact[k])
        aW, ab, ax = _conv_back(act[k - 1].abs(), W.abs(), gact[k].abs())
        per_acc = math.ceil(each / 8) if k == 1 else each  # the first layer has eight accumulators
        _check(g[f"W{k}"], dW, (17 * 8 * per_acc + 8 + joined) * U23 * aW, f"W{k} gradient")
        _check(g[f"b{k}"], db, (16 * each + 8 + joined) * U23 * ab, f"b{k} gradient")
        if k >= 2:
            _check_bf16(gact[k - 1], dx, 577 * U23 * ax, act[k - 1] > 0, f"layer {k - 1} pre-activation gradient")
    net.close()


@pytest.mark.parametrize("batch,length", [(305, 640), (305, 1024)])
def test_weight_gradient_ring_is_reused(gpu_lib, batch, length):
    """11 and 17 tiles a CTA through the ring of six buffers; whole numbers up to 2, whose sums
    FP32 holds exactly."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(length)
    dy, x = (torch.randint(-2, 3, (batch, length, 64), device="cuda", generator=gen).to(torch.bfloat16)
             for _ in range(2))
    dw, db = qlpbls.conv64_wgrad(dy, x)
    want, want_b, _ = _conv_back(x.double(), torch.zeros(9, 64, 64, device="cuda", dtype=torch.float64), dy.double())
    assert torch.equal(dw.double(), want)
    assert torch.equal(db.double(), want_b)


@pytest.mark.parametrize("mask", [False, True])
def test_conv64_over_several_tiles(gpu_lib, mask):
    """13 and 14 tiles a CTA (six buffers, four accumulators, two staging tiles): whole numbers
    whose sums BF16 holds exactly."""
    import torch
    B, L = 200, 1280
    gen = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randint(-1, 2, (B, L, 64), device="cuda", generator=gen).to(torch.bfloat16)
    w = torch.zeros(9, 64, 64, device="cuda")
    for k in range(9):  # 27 terms of magnitude at most 1 for every output
        for j in range(3):
            w[k, torch.arange(64), (torch.arange(64) * 5 + 7 * k + 11 * j) % 64] = float(1 - 2 * ((j + k) % 2))
    keep = torch.randint(-1, 2, (B, L, 64), device="cuda", generator=gen).to(torch.bfloat16) if mask else None
    y = qlpbls.conv64(x, qlpbls.pack_w64(w), mask=keep, relu=False)
    want = _conv(x.double(), w.double())
    if mask:
        want = torch.where(keep > 0, want, torch.zeros_like(want))
    assert torch.equal(y.double(), want)
