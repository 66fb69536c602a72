"""GPU selections on crafted inputs: the S/N kernel's medians, trend and MAD on spectra
chosen for its selection passes (ties, wide and narrow ranges, constant, lengths from one
entry to longer than its cached keys), and the top-k bins at short and ragged rows."""
import numpy as np
import pytest

from oracle import snr as osn
from paper_2302_01293_gb300 import qlpbls

pytestmark = pytest.mark.gpu

# S/N is one FP32 rounding of FP64 arithmetic whose sigma comes from an FP32 MAD: two
# roundings of 2^-24, with a hair for the quotient
RTOL_RAW = 2.5 * 2.0 ** -24


def _spectrum(kind, n, rng):
    if kind == "noise":
        return (1e-5 * rng.chisquare(4, n)).astype(np.float32)
    if kind == "constant":
        return np.full(n, 3e-5, np.float32)
    if kind == "two_values":
        return np.where(rng.uniform(size=n) < 0.5, 1e-5, 2e-5).astype(np.float32)
    if kind == "few_levels":  # long runs of equal keys beside close neighbours
        return np.float32(1e-5) * (1 + rng.integers(0, 3, n) * np.float32(2.0 ** -22)).astype(np.float32)
    if kind == "wide":  # zeros, tiny and large values: the key range is nearly all 32 bits
        v = np.exp(rng.uniform(-80, 5, n))
        v[rng.uniform(size=n) < 0.1] = 0.0
        return v.astype(np.float32)
    raise ValueError(kind)


def _plan(lengths, params=None):
    """A plan of stars whose grids have the given lengths, windows cut from one long grid."""
    n = 6000
    t = 2880.0 + np.arange(n) * 0.02
    one = qlpbls.star_grid(t, np.ones(n), np.ones(n), 1.0)["freqs"]
    lo, hi = [], []
    for m in lengths:
        lo.append(one[0])
        hi.append(0.5 * (one[m - 1] + one[m]))
    k = len(lengths)
    offs = np.arange(k + 1, dtype=np.int64) * n
    rng = np.random.default_rng(1)
    win = (np.arange(k + 1, dtype=np.int64), np.asarray(lo), np.asarray(hi))
    return qlpbls.Plan(offs, np.tile(t, k), 1.0 + 1e-3 * rng.standard_normal(n * k), np.full(n * k, 1e-3),
                       np.ones(k), np.ones(k), params, windows=win)


@pytest.mark.parametrize("kind", ["noise", "constant", "two_values", "few_levels", "wide"])
@pytest.mark.parametrize("mad", [qlpbls.MAD_RAW, qlpbls.MAD_RESID])
def test_snr_selection(gpu_lib, kind, mad):
    import torch
    lengths = [1, 2, 3, 31, 64, 65, 127, 512, 513, 1024, 1025, 4095, 12288, 12289, 14001]
    plan = _plan(lengths, qlpbls.Params(mad_mode=mad))
    assert [int(x) for x in np.diff(plan.freq_offsets)] == lengths
    rng = np.random.default_rng(7)
    out = plan.search()
    sr = np.concatenate([_spectrum(kind, m, rng) for m in lengths])
    out["sr"].copy_(torch.from_numpy(sr))
    trend = plan.alloc_trend()
    plan.snr(out, trend_out=trend)
    assert plan.device_status() == 0
    got = out["snr"].cpu().numpy().astype(np.float64)
    rec = trend.cpu().numpy().reshape(len(lengths), -1)
    best = plan.best_host(out)
    for s, m in enumerate(lengths):
        sl = plan.star_slice(s)
        f, v = plan.freqs[sl], sr[sl].astype(np.float64)
        _, xs, ys = osn.trend_curve(f, v)
        assert int(rec[s, 0]) == len(xs)
        assert np.array_equal(rec[s, 4:4 + len(xs)], xs) and np.array_equal(rec[s, 44:44 + len(ys)], ys)
        ref, tr, sigma = osn.spectral_snr(f, v, "raw" if mad == qlpbls.MAD_RAW else "resid")
        # FP32 residuals: the medians move by half an ulp of the residuals
        eps = 0.0 if mad == qlpbls.MAD_RAW else 2.0 ** -24 * float(np.median(np.abs(v - tr)))
        if sigma <= 8.0 * eps * 1.4826:  # (nearly) no spread: either zero or rounding
            continue
        assert rec[s, 1] == pytest.approx(sigma, rel=2.0 ** -23 + 4.0 * eps / sigma)
        tol = (RTOL_RAW + 4.0 * eps * 1.4826 / sigma) * np.abs(ref) + 1e-30
        assert np.all(np.abs(got[sl] - ref) <= tol), (m, float(np.max(np.abs(got[sl] - ref) - tol)))
        k = int(np.argmax(got[sl]))
        assert best[s]["f_idx"] in (k, -1)
    if kind == "constant":
        assert not got.any() and np.all(best["f_idx"] == -1)


@pytest.mark.parametrize("length,k", [(1, 1), (31, 5), (256, 32), (257, 32), (4096, 64), (9001, 40), (300, 300)])
def test_topk_rows(gpu_lib, length, k):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(length)
    z = torch.randn(5, length, device="cuda", generator=gen)
    z[1] = torch.round(z[1])                      # ties: the lower bin first
    z[2] = -3.0e38                                # the smallest value that can be taken
    x0 = torch.zeros(5, length, qlpbls.CNN_IN_CH, dtype=torch.bfloat16, device="cuda")
    x0[:, :, 1] = 1
    x0[3, torch.rand(length, device="cuda", generator=gen) < 0.9, 1] = 0  # fewer valid bins than k
    x0[4, :, 1] = 0
    got = qlpbls.topk(z, x0, k).cpu().numpy()
    zh, ok = z.cpu().numpy(), x0[:, :, 1].float().cpu().numpy() > 0
    for r in range(5):
        order = [i for i in np.argsort(-zh[r], kind="stable") if ok[r, i]][:k]
        assert got[r].tolist() == order + [-1] * (k - len(order)), r
