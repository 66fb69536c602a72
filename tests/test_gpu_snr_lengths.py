"""The S/N kernel in both of its launches and on spectra shorter and longer than its cached
keys: batches of at least as many stars as the chip has SMs cache 6,144 keys, smaller ones
24,576. Trend, sigma, S/N and the best record against the oracle, both MAD modes."""
import numpy as np
import pytest

from oracle import snr as osn
from paper_2302_01293_gb300 import qlpbls
from test_gpu_select import RTOL_RAW, _spectrum

pytestmark = pytest.mark.gpu


def _plan(lengths, mad):
    """Stars whose grids have the given lengths: windows from the low end of one long grid."""
    t = 2880.0 + np.arange(500) * 0.6
    one = qlpbls.star_grid(t, np.ones(500), np.ones(500), 1.0)["freqs"]
    hi = [0.5 * (one[m - 1] + one[m]) for m in lengths]
    k = len(lengths)
    rng = np.random.default_rng(2)
    win = (np.arange(k + 1, dtype=np.int64), np.full(k, one[0]), np.asarray(hi))
    return qlpbls.Plan(np.arange(k + 1, dtype=np.int64) * 500, np.tile(t, k),
                       1.0 + 1e-3 * rng.standard_normal(500 * k), np.full(500 * k, 1e-3), np.ones(k), np.ones(k),
                       qlpbls.Params(mad_mode=mad), windows=win)


LENGTHS = {"many": [1, 2, 5, 63, 64, 65, 511, 512, 513, 1500, 6143, 6144, 6145, 14001] * 11,
           "few": [1, 2, 1023, 1024, 1025, 6144, 14001, 24575, 24576, 24577, 30000]}


@pytest.mark.parametrize("kind", ["noise", "few_levels", "two_values", "wide"])
@pytest.mark.parametrize("mad", [qlpbls.MAD_RAW, qlpbls.MAD_RESID])
@pytest.mark.parametrize("batch", ["many", "few"])
def test_snr_lengths(gpu_lib, kind, mad, batch):
    import torch
    lengths = LENGTHS[batch]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert (len(lengths) >= sms) == (batch == "many")
    plan = _plan(lengths, mad)
    assert [int(x) for x in np.diff(plan.freq_offsets)] == lengths
    rng = np.random.default_rng(len(lengths))
    n = plan.n_freq_total
    box = dict(sr=np.concatenate([_spectrum(kind, m, rng) for m in lengths]),
               qidx=rng.integers(0, 14, n).astype(np.uint8), kbin=rng.integers(0, 40, n).astype(np.int32),
               s=-rng.uniform(1e-4, 1e-2, n).astype(np.float32), r=rng.uniform(0.01, 0.3, n).astype(np.float32))
    out = plan.alloc_outputs()
    for name, v in box.items():
        out[name].copy_(torch.from_numpy(v))
    trend = plan.alloc_trend()
    plan.snr(out, trend_out=trend)
    assert plan.device_status() == 0
    snr, best = out["snr"].cpu().numpy().astype(np.float64), plan.best_host(out)
    rec = trend.cpu().numpy().reshape(len(lengths), -1)
    reported = 0
    for s, m in enumerate(lengths):
        sl = plan.star_slice(s)
        f, v, got = plan.freqs[sl], box["sr"][sl].astype(np.float64), snr[sl]
        _, xs, ys = osn.trend_curve(f, v)
        assert int(rec[s, 0]) == len(xs)
        assert np.array_equal(rec[s, 4:4 + len(xs)], xs) and np.array_equal(rec[s, 44:44 + len(ys)], ys)
        ref, tr, sigma = osn.spectral_snr(f, v, "raw" if mad == qlpbls.MAD_RAW else "resid")
        # FP32 residuals: the medians move by half an ulp of the residuals
        eps = 0.0 if mad == qlpbls.MAD_RAW else 2.0 ** -24 * float(np.median(np.abs(v - tr)))
        if rec[s, 1] > 0.0:  # a spread: the first maximum's box is the record
            k = int(np.argmax(got))
            i = sl.start + k
            r = float(box["r"][i])
            assert best[s]["f_idx"] == k and best[s]["f"] == f[k] and best[s]["period"] == 1.0 / f[k]
            assert best[s]["j"] == box["qidx"][i] and best[s]["k"] == box["kbin"][i]
            assert best[s]["snr"] == got[k] and best[s]["sr"] == v[k]
            assert best[s]["depth"] == -float(box["s"][i]) / (r * (1.0 - r))
            assert best[s]["status"] == 0
            reported += 1
        else:
            assert best[s]["f_idx"] == -1 and best[s]["status"] == qlpbls.STAR_ZERO_MAD and not got.any()
        if sigma <= 8.0 * eps * 1.4826:  # (nearly) no spread: either zero or rounding
            continue
        assert rec[s, 1] == pytest.approx(sigma, rel=2.0 ** -23 + 4.0 * eps / sigma)
        tol = (RTOL_RAW + 4.0 * eps * 1.4826 / sigma) * np.abs(ref) + 1e-30
        assert np.all(np.abs(got - ref) <= tol), (m, float(np.max(np.abs(got - ref) - tol)))
    assert reported >= len(lengths) // 2 or kind in ("two_values", "few_levels")
