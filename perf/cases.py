"""Performance cases: the work a user of the transit search has the framework do.

A case is a dict of plain values. `prepare` makes, from a seed, what a user's program
holds before the call (light curves, plans, networks, output buffers), `run` is one pass
through the public entry points, `work` what that pass cannot do without and `exact` the
same outputs in 64 bits, without the framework's code.

Kinds:
  search   light curves with a plan: the periodogram of every star and its spectral S/N
  coarse   the learned path's first stage: log-period spectra, S/N with its trend record,
           the network input
  refine   its last stage: the grid inside the proposed period windows, scored on the
           coarse trend
  vetting  the statistics of each star's best candidate and its strongest peaks
  host     host light curves in, best candidates out, in one call (planning included)
  propose  the proposal network on a batch of coarse spectra, and the top bins
  train    one training step of that network
  layer    one 64-channel layer by itself: forward, input gradient, weight gradient
"""
import math
import os
import tempfile

import numpy as np
import torch

from paper_2302_01293_gb300 import qlpbls

SECTOR = 27.4            # days
T_START = 2880.0         # time stamps of the size TESS uses (BTJD)
G_SI = 6.67430e-11
N_Q = 14                 # durations q_min exp(0.1 j) up to 2 q_circ, from 0.5 q_circ
NET_LEN, NET_CH = 4096, 6
DEV = "cuda"
EXACT_PAIRS = 3.0e10     # point-frequency pairs the 64-bit search takes within its time


def listed():
    return [
        # one newly downloaded star, 30-minute cadence, one sector: latency and launches
        dict(name="star_30min", kind="search", stars=1, sectors=1, cadence=1800, rho_lo=1.41, rho_hi=1.41,
             red=False, errors="equal", method=0),
        # a camera's handful of targets with per-point errors, 200-second cadence, ragged by gaps
        dict(name="sector_150", kind="search", stars=150, sectors=1, cadence=200, rho_lo=0.1, rho_hi=10.0, red=False,
             errors="scattered", method=0),
        # the production batch: 4,096 uneven single-sector stars
        dict(name="sector_4096", kind="search", stars=4096, sectors=1, cadence=200, rho_lo=0.1, rho_hi=10.0,
             red=False, errors="equal", method=0),
        # stars near the ecliptic pole: 1-13 sectors with red noise, tables in time windows
        dict(name="multi_sector_40", kind="search", stars=40, sectors=13, cadence=200, rho_lo=1.41, rho_hi=1.41,
             red=True, errors="equal", method=0),
        # irregularly sampled stars (ground-based, or cadences cut by quality flags): every point folded
        dict(name="irregular_77", kind="search", stars=77, sectors=1, cadence=0, rho_lo=0.3, rho_hi=5.0, red=False,
             errors="scattered", method=0),
        # the learned path's coarse spectra of 1-4 sector stars
        dict(name="coarse_256", kind="coarse", stars=256, sectors=4),
        # and its refined search inside 32 proposed windows per star
        dict(name="refine_256", kind="refine", stars=256, sectors=4, proposals=32),
        # vetting of a batch's candidates
        dict(name="vetting_1000", kind="vetting", stars=1000, peaks=5),
        # the whole call from host arrays, host planning included
        dict(name="host_600", kind="host", stars=600),
        # the network on a batch of spectra, 32 proposals each
        dict(name="propose_256", kind="propose", batch=256, k=32),
        # one training step at the training batch size
        dict(name="train_128", kind="train", batch=128),
        # a small layer by itself: few tiles
        dict(name="layer_12x1920", kind="layer", batch=12, length=1920),
    ]


def draw(rng):
    def logint(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["search"] * 5 + ["coarse", "refine", "vetting", "host", "propose", "train", "layer"])
    if kind == "search":
        form = rng.choice(["few", "sector", "sector", "multi", "irregular", "points"])
        c = dict(kind=kind, stars=logint(20, 2500), sectors=1, cadence=200, rho_lo=0.1, rho_hi=10.0, red=False,
                 errors=rng.choice(["equal", "scattered"]), method=0)
        if form == "few":
            c.update(stars=logint(1, 12), cadence=rng.choice([200, 600, 1800]), rho_lo=1.0, rho_hi=3.0)
        elif form == "multi":
            c.update(stars=logint(5, 40), sectors=rng.randint(2, 13), rho_lo=1.0, rho_hi=2.0, red=rng.random() < 0.7)
        elif form == "irregular":
            c.update(stars=logint(4, 200), cadence=0, rho_lo=0.3, rho_hi=5.0)
        elif form == "points":  # every point folded on request, as the precision studies do
            c.update(stars=logint(4, 60), method=1, rho_lo=0.3, rho_hi=5.0)
        return c
    if kind == "coarse":
        return dict(kind=kind, stars=logint(16, 700), sectors=rng.randint(1, 4))
    if kind == "refine":
        return dict(kind=kind, stars=logint(16, 700), sectors=rng.randint(1, 4), proposals=rng.randint(4, 32))
    if kind == "vetting":
        return dict(kind=kind, stars=logint(32, 3000), peaks=rng.randint(1, 16))
    if kind == "host":
        return dict(kind=kind, stars=logint(8, 2000))
    if kind == "propose":
        return dict(kind=kind, batch=logint(1, 700), k=rng.randint(1, 32))
    if kind == "train":
        return dict(kind=kind, batch=logint(4, 300))
    return dict(kind=kind, batch=logint(1, 160), length=128 * logint(2, 40))


# ---------------------------------------------------------------- light curves

def _kepler_q(period_days, rho):
    """Circular, central transit duration over the period."""
    ps = np.asarray(period_days, np.float64) * 86400.0
    a_r = np.cbrt(G_SI * np.asarray(rho, np.float64) * 1000.0 * ps * ps / (3.0 * math.pi))
    return np.arcsin(np.minimum(1.0, 1.0 / a_r)) / math.pi


def _p_min(rho):
    return np.sqrt(3.0 * math.pi * 8.0 / (G_SI * np.asarray(rho, np.float64) * 1000.0)) / 86400.0


def _star_mix(case):
    """What does not depend on the seed: each star's density and its sectors, evenly spread
    over the case's ranges, so that the amount of work is the case's."""
    n = case["stars"]
    lo, hi = case.get("rho_lo", 0.1), case.get("rho_hi", 10.0)
    u = (np.arange(n) * 0.6180339887498949 + 0.5) % 1.0
    rho = np.exp(math.log(lo) + u * (math.log(hi) - math.log(lo)))
    sectors = 1 + np.arange(n) * 7 % case.get("sectors", 1)
    return rho, sectors


def _times(case, rng, sectors):
    """Gaps and irregular times are the seed's; a star's first and last time stamps are the
    case's, and with them its number of trial frequencies."""
    cadence = case.get("cadence", 200)
    out = []
    for s, ns in enumerate(sectors):
        start = T_START + (0.37 * s) % 1.0
        if cadence == 0:
            inside = np.sort(rng.uniform(0.0, SECTOR, int(rng.integers(900, 4200))))
            out.append(start + np.concatenate([[0.0], inside, [SECTOR]]))
            continue
        n = int(round(SECTOR * 86400.0 / cadence))
        keep = np.ones(n * ns, bool)
        if ns == 1:
            gaps = int(rng.integers(0, 7)) if cadence == 200 else 1
            for _ in range(gaps):
                a = rng.uniform(0.1, SECTOR - 2.1)
                lost = slice(int(a / SECTOR * n), int((a + rng.uniform(0.5, 2.0)) / SECTOR * n))
                if keep.sum() > 0.62 * n:
                    keep[lost] = False
        grid = np.arange(n) * (cadence / 86400.0)
        base = np.concatenate([k * (SECTOR + 1.0) + grid for k in range(ns)])
        out.append(start + base[keep])
    return out


def _red_noise(rng, n, sigma, phi=0.9, block=256):
    """A stationary AR(1) sequence, block by block (phi^256 is 2e-12)."""
    m = -(-n // block)
    e = rng.standard_normal((m, block)) * (sigma * math.sqrt(1.0 - phi * phi))
    i = np.arange(block)
    part = e @ np.tril(phi ** np.abs(i[:, None] - i[None, :])).T
    part[1:] += part[:-1, -1:] * phi ** (i + 1)
    return part.reshape(-1)[:n]


def _light_curves(case, seed):
    """(offsets, t, y, dy, rho, rstar): host arrays, as a reader of light curves hands them over."""
    rng = np.random.default_rng([seed, 11])
    n = case["stars"]
    rho, sectors = _star_mix(case)
    ts = _times(case, rng, sectors)
    offsets = np.zeros(n + 1, np.int64)
    offsets[1:] = np.cumsum([t.shape[0] for t in ts])
    t = np.concatenate(ts)
    sigma = np.exp(rng.uniform(math.log(2e-4), math.log(2e-3 if case["kind"] in ("coarse", "refine") else 1e-2), n))
    if case.get("red"):
        sigma[:] = 1e-3
    dy = np.repeat(sigma, np.diff(offsets))
    if case.get("errors") == "scattered":
        dy *= rng.uniform(0.8, 1.2, dy.shape[0])
    y = rng.standard_normal(t.shape[0], dtype=np.float32) * dy
    if case.get("red"):
        y += _red_noise(rng, t.shape[0], 1e-3)
    y += 1.0
    for s in range(n):  # transits in about a third of the stars
        if n > 1 and rng.uniform() > 0.35:
            continue
        a, b = int(offsets[s]), int(offsets[s + 1])
        span = (t[b - 1] - t[a]) / 2.2
        period = math.exp(rng.uniform(math.log(0.6), math.log(span)))
        t0 = t[a] + rng.uniform(0.0, period)
        half = 0.5 * period * float(_kepler_q(period, rho[s]))
        phase = np.mod(t[a:b] - t0 + 0.5 * period, period) - 0.5 * period
        y[a:b] -= math.exp(rng.uniform(math.log(3e-4), math.log(1e-2))) * (np.abs(phase) < half)
    return offsets, t, y, dy, rho, np.ones(n)


# ---------------------------------------------------------------- spectra and networks

def _spectra(batch, seed):
    """Network input as qlp_bls_coarse_tensor lays it out (BF16 [batch][4096][6]) and labels:
    noise spectra with a peak and its aliases in half of the rows, searched between two
    period limits of the star's own."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    dev = torch.device(DEV)
    snr = 1.3 * torch.randn(batch, NET_LEN, device=dev, generator=gen)
    k = torch.arange(NET_LEN, device=dev)
    lo = 600 + torch.randint(0, 500, (batch, 1), device=dev, generator=gen)
    hi = 2400 + torch.randint(0, 1000, (batch, 1), device=dev, generator=gen)
    mask = (k >= lo) & (k < hi)
    peak = lo + ((hi - lo) * torch.rand(batch, 1, device=dev, generator=gen)).long()
    has = torch.rand(batch, 1, device=dev, generator=gen) < 0.5
    height = torch.exp(1.5 + 2.5 * torch.rand(batch, 1, device=dev, generator=gen))
    d2, d3 = 342, 542
    for shift, share in ((0, 1.0), (d2, 0.6), (-d2, 0.5), (d3, 0.4)):
        snr += has * share * height * torch.exp(-0.5 * ((k - peak - shift) / 2.0) ** 2)
    a = torch.where(mask, torch.asinh(0.25 * snr), torch.zeros((), device=dev)).to(torch.bfloat16)
    x = torch.zeros(batch, NET_LEN, NET_CH, dtype=torch.bfloat16, device=dev)
    x[:, :, 0] = a
    x[:, :, 1] = mask
    for c, d in ((2, d2), (3, -d2), (4, d3), (5, -d3)):
        there = torch.roll(a, -d, 1)
        there = torch.where(((k + d >= 0) & (k + d < NET_LEN)) & mask, there, torch.zeros((), device=dev).to(a.dtype))
        x[:, :, c] = there
    labels = (has & mask & ((k - peak).abs() <= 1)).float()
    return x.contiguous(), labels.contiguous()


def _net_params(seed):
    """Weights of the network's initial distribution, in the order of its flat parameters."""
    rng = np.random.default_rng([seed, 7])
    parts = []
    for co, ci in ((64, NET_CH), (64, 64), (64, 64), (64, 64), (64, 64), (1, 64)):
        parts += [rng.standard_normal(9 * co * ci) * math.sqrt((2.0 if co > 1 else 1.0) / (9 * ci)),
                  0.02 * rng.standard_normal(co) - (0.0 if co > 1 else 4.0)]
    return np.concatenate(parts).astype(np.float32)


def _network(case, seed):
    net = qlpbls.CNN(case["batch"], NET_LEN, seed=seed)
    net.set_params(_net_params(seed))
    return net


def _warm_moments(net, seed):
    """Training resumed from a checkpoint: Adam's moments are those of a run under way (after
    the file's header come the parameters and the two moment vectors in FP32)."""
    rng = np.random.default_rng([seed, 5])
    fd, path = tempfile.mkstemp(suffix=".ckpt")
    os.close(fd)
    try:
        net.save(path)
        with open(path, "rb") as f:
            raw = f.read()
        n = net.n_params
        head = raw[: len(raw) - 12 * n]
        params = np.frombuffer(raw[len(head): len(head) + 4 * n], "<f4")
        m = (1e-4 * rng.standard_normal(n)).astype("<f4")
        v = (1e-6 * rng.uniform(0.5, 2.0, n)).astype("<f4")
        with open(path, "wb") as f:
            f.write(head + params.tobytes() + m.tobytes() + v.tobytes())
        net.load(path)
    finally:
        os.unlink(path)


def _layer_inputs(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    b, n = case["batch"], case["length"]
    r = lambda *s: torch.randn(*s, device=DEV, generator=gen)  # noqa: E731
    x = torch.relu(r(b, n, 64)).to(torch.bfloat16)       # the layer below's output
    dy = (r(b, n, 64) * (r(b, n, 64) > 0)).to(torch.bfloat16)  # gradients through this layer's ReLU
    return x, dy, r(9, 64, 64) * math.sqrt(2.0 / 576.0), 0.1 * r(64)


# ---------------------------------------------------------------- preparation

def _coarse_params():
    return qlpbls.Params(grid_mode=1)


def _proposed_windows(case, coarse):
    """Each star's proposals: coarse bins spread over those it searched (the same for every
    seed, so that the refined grids are)."""
    rng = np.random.default_rng([case["stars"], case["proposals"], 3])
    bins = np.full((case["stars"], case["proposals"]), -1, np.int32)
    for s in range(case["stars"]):
        sl = coarse.star_slice(s)
        if sl.stop <= sl.start:
            continue
        k = qlpbls.coarse_bins(1.0 / coarse.freqs[sl], coarse.params)
        take = rng.choice(k, min(case["proposals"], k.shape[0]), replace=False)
        bins[s, : take.shape[0]] = take
    return qlpbls.proposal_windows(bins, coarse.params, 1.0)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind in ("search", "vetting"):
        lc = _light_curves(case, seed)
        st["plan"] = qlpbls.Plan(*lc, params=qlpbls.Params(method=case.get("method", 0)))
        st["out"] = st["plan"].alloc_outputs()
        if kind == "vetting":  # the search came before
            st["plan"].search(st["out"])
            st["plan"].snr(st["out"])
            st["stats"] = st["plan"].candidate_stats(st["out"])
    elif kind in ("coarse", "refine"):
        lc = _light_curves(case, seed)
        coarse = qlpbls.Plan(*lc, params=_coarse_params())
        st["plan"], st["out"], st["trend"] = coarse, coarse.alloc_outputs(), coarse.alloc_trend()
        if kind == "refine":  # the coarse stage came before
            coarse.search(st["out"])
            coarse.snr(st["out"], trend_out=st["trend"])
            st["plan"] = qlpbls.Plan.windows_from(coarse, _proposed_windows(case, coarse))
            st["out"] = st["plan"].alloc_outputs()
    elif kind == "host":
        st["lc"] = _light_curves(case, seed)
    elif kind == "propose":
        st["net"] = _network(case, seed)
        st["x0"], _ = _spectra(case["batch"], seed)
        st["logits"] = torch.empty(case["batch"], NET_LEN, dtype=torch.float32, device=DEV)
    elif kind == "train":
        st["net"] = _network(case, seed)
        st["x0"], st["labels"] = _spectra(case["batch"], seed)
        _warm_moments(st["net"], seed)
    else:
        x, dy, w, bias = _layer_inputs(case, seed)
        st.update(x=x, dy=dy, bias=bias, wf=qlpbls.pack_w64(w), wb=qlpbls.pack_w64(w, transpose=True),
                  err=torch.zeros(1, dtype=torch.int32, device=DEV), y=torch.empty_like(x), dx=torch.empty_like(x))
    torch.cuda.synchronize()
    return st


# ---------------------------------------------------------------- one pass

def _best_fields(raw, n):
    """The records' whole numbers and their FP64 fields, as views of the device buffer."""
    rec = raw[: n * qlpbls.BEST_DTYPE.itemsize].view(n, qlpbls.BEST_DTYPE.itemsize)
    return dict(f_idx=rec[:, :8].view(torch.int64), values=rec[:, 8:64].view(torch.float64),
                counts=rec[:, 64:88].view(torch.int32))


def _spectrum(out, plan):
    nf, n = plan.n_freq_total, plan.n_stars
    got = {k: out[k][:nf] for k in ("sr", "qidx", "kbin", "s", "r", "snr")}
    got["best"] = _best_fields(out["best"], n)
    return got


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "search":
        st["plan"].search(st["out"])
        st["plan"].snr(st["out"])
        return _spectrum(st["out"], st["plan"])
    if kind == "coarse":
        st["plan"].search(st["out"])
        st["plan"].snr(st["out"], trend_out=st["trend"])
        x0, rows = st["plan"].coarse_tensor(st["out"], snr_rows=True)
        got = _spectrum(st["out"], st["plan"])
        got.update(trend=st["trend"], x0=x0, rows=rows)
        return got
    if kind == "refine":
        st["plan"].search(st["out"])
        st["plan"].snr(st["out"], trend_in=st["trend"])
        return _spectrum(st["out"], st["plan"])
    if kind == "vetting":
        stats = st["plan"].candidate_stats(st["out"], stats=st["stats"])
        peaks = st["plan"].top_peaks(st["out"], case["peaks"])
        n = st["plan"].n_stars
        rec = stats[: n * qlpbls.STATS_DTYPE.itemsize].view(n, qlpbls.STATS_DTYPE.itemsize)
        return dict(fit=rec[:, :80].view(torch.float64), counts=rec[:, 80:112].view(torch.int32), peaks=peaks)
    if kind == "host":
        best = qlpbls.run_host(*st["lc"])["best"]
        return {k: np.ascontiguousarray(best[k]) for k in best.dtype.names}
    if kind == "propose":
        logits = st["net"].forward(st["x0"], out=st["logits"])
        return dict(logits=logits, bins=qlpbls.topk(logits, st["x0"], case["k"]))
    if kind == "train":
        st["net"].train_step(st["x0"], st["labels"], 16.0, 3e-4)
        params, grads = st["net"].params(with_grads=True)
        return dict(params=params, grads=grads)
    y = qlpbls.conv64(st["x"], st["wf"], bias=st["bias"], relu=True, out=st["y"], err=st["err"])
    dx = qlpbls.conv64(st["dy"], st["wb"], mask=st["x"], relu=False, out=st["dx"], err=st["err"])
    dw, db = qlpbls.conv64_wgrad(st["dy"], st["x"])
    return dict(y=y, dx=dx, dw=dw, db=db)


# ---------------------------------------------------------------- work

def _points_of(case, sectors):
    if case.get("cadence", 200) == 0:
        return np.full(case["stars"], 2550.0)
    per = SECTOR * 86400.0 / case.get("cadence", 200)
    return np.where(sectors == 1, 0.87, 1.0) * sectors * per


def _grid_sums(case):
    """Over all stars: points, trial frequencies, phase bins, bin edges (cycles x bins)."""
    rho, sectors = _star_mix(case)
    pts = _points_of(case, sectors)
    base = np.where(sectors == 1, SECTOR, sectors * (SECTOR + 1.0) - 1.0)
    nf = nb = ne = pairs = 0.0
    for r, t, p in zip(rho[:512], base, pts):
        f = np.linspace(2.0 / t, 1.0 / _p_min(r), 400)
        q = 0.5 * _kepler_q(1.0 / f, r)
        if case["kind"] in ("coarse", "refine"):
            per = NET_LEN / math.log(4000.0) / f  # log-spaced: density per unit frequency
        else:
            per = 2.0 * t / q
        if case["kind"] == "refine":
            share = min(1.0, case["proposals"] * 2.0 / (NET_LEN * math.log(f[-1] / f[0]) / math.log(4000.0)))
            per = share * 2.0 * t / q
        w = per * (f[1] - f[0])
        nf, nb, ne = nf + w.sum(), nb + (w * 3.0 / q).sum(), ne + (w * 3.0 / q * f * t).sum()
        pairs += w.sum() * p
    scale = case["stars"] / min(case["stars"], 512)
    return float(pts.sum()), nf * scale, nb * scale, ne * scale, pairs * scale


def work(case):
    kind = case["kind"]
    if kind in ("search", "coarse", "refine", "host", "vetting"):
        pts, nf, nb, ne, _ = _grid_sums(case)
        if kind == "vetting":  # the S/N read once by the peaks, the points once by the fit and the residuals
            return dict(bytes=24.0 * pts + 12.0 * nf + 200.0 * case["stars"], flops=60.0 * pts)
        # two sums per bin edge (per point-frequency pair when points are folded one by one is
        # more); per start bin two running sums and nine scores of six operations
        flops = 2.0 * ne + nb * (22.0 + 54.0)
        out = 88.0 * case["stars"] + (0.0 if kind == "host" else 21.0 * nf)
        if kind == "coarse":
            out += case["stars"] * NET_LEN * (2.0 * NET_CH + 4.0)
        return dict(bytes=24.0 * pts + out, flops=flops)
    if kind == "layer":
        pos = case["batch"] * case["length"]
        return dict(bytes=pos * 64 * 2 * 6.0 + 2 * 73728.0 + 147712.0, flops=3.0 * 73728 * pos)
    pos = case["batch"] * NET_LEN
    fwd = pos * (2.0 * 54 * 64 + 4 * 73728 + 2.0 * 576)
    if kind == "propose":
        return dict(bytes=pos * (12.0 + 4.0) + 0.6e6 + 4.0 * case["batch"] * case["k"], flops=fwd)
    return dict(bytes=pos * (12.0 + 4.0) + 4 * 0.6e6, flops=3.0 * fwd)


# ---------------------------------------------------------------- 64 bits

def _grids64(lc):
    """Per star: trial frequencies and shortest durations by the spacing rule, all stars together."""
    offsets, t, _, _, rho, _ = lc
    first, last = t[offsets[:-1]], t[offsets[1:] - 1]
    base = last - first
    fmax = 1.0 / _p_min(rho)
    f = 1.0 / (base / 2.0)
    fs = []
    on = f <= fmax
    while on.any():
        q = 0.5 * _kepler_q(1.0 / f, rho)
        fs.append((np.where(on, f, np.nan), q))
        f = np.where(on, f + q / (2.0 * base), f)
        on = on & (f <= fmax)
    ff, qq = np.stack([a for a, _ in fs], 1), np.stack([b for _, b in fs], 1)
    return [(ff[s][~np.isnan(ff[s])], qq[s][~np.isnan(ff[s])]) for s in range(rho.shape[0])]


def _coarse_grids64(lc):
    offsets, t, _, _, rho, _ = lc
    per = 0.1 * 4000.0 ** (np.arange(NET_LEN) / (NET_LEN - 1.0))
    got = []
    for s in range(rho.shape[0]):
        base = t[offsets[s + 1] - 1] - t[offsets[s]]
        p = per[(per >= _p_min(rho[s])) & (per <= base / 2.0)][::-1]
        got.append((1.0 / p, 0.5 * _kepler_q(p, rho[s])))
    return got


def _search64(t, y, dy, f, q):
    """SR, s, r of every frequency's best box, on the GPU in FP64: each point's phase bin, the
    prefix sums at the bins' edges, every box of every duration."""
    dev = torch.device(DEV)
    tp = torch.from_numpy(t - t[0]).to(dev)
    w = torch.from_numpy(dy).to(dev) ** -2
    w = w / w.sum()
    yy = torch.from_numpy(y).to(dev)
    wd = w * (yy - (w * yy).sum())
    zero = torch.zeros(1, dtype=torch.float64, device=dev)
    cum = torch.stack([torch.cat([zero, w.cumsum(0)]), torch.cat([zero, wd.cumsum(0)])])
    sr, sb, rb = (np.zeros(f.shape[0]) for _ in range(3))
    nbs = np.ceil(3.0 / q).astype(np.int64)
    k = 0
    while k < f.shape[0]:
        room = 6_000_000 // max(t.shape[0], int((t[-1] - t[0]) * f[k] + 2) * int(nbs[k]))
        e = min(f.shape[0], k + max(1, room))
        fk, nb = torch.from_numpy(f[k:e]).to(dev), torch.from_numpy(nbs[k:e]).to(dev)
        x = tp[None, :] * fk[:, None]
        c = x.floor()
        b = torch.minimum(((x - c) * nb[:, None]).floor().long(), nb[:, None] - 1)
        g = c.long() * nb[:, None] + b                       # the point's bin, counted over all cycles
        n_edge = int(g[:, -1].max()) + 2
        edges = torch.arange(n_edge, device=dev)[None, :].expand(e - k, n_edge)
        at = torch.searchsorted(g, edges.contiguous())
        nmax = int(nb.max())
        phase = torch.remainder(edges[:, :-1], nb[:, None])
        h = []
        for row in cum:
            at_edges = row[at]
            acc = torch.zeros(e - k, nmax, dtype=torch.float64, device=dev)
            h.append(acc.scatter_add_(1, phase, at_edges[:, 1:] - at_edges[:, :-1]))
        col = torch.arange(nmax + 16, device=dev)[None, :]
        wrap = torch.remainder(col, nb[:, None])
        hw, hy = (torch.gather(a, 1, wrap) for a in h)
        qk = torch.from_numpy(q[k:e]).to(dev)
        widths = torch.stack([((qk * math.exp(0.1 * j) * nb) + 0.5).floor().long().clamp(min=1) for j in range(N_Q)])
        best = torch.zeros(e - k, dtype=torch.float64, device=dev)
        bs, br = torch.zeros_like(best), torch.zeros_like(best)
        rw = torch.zeros(e - k, nmax, dtype=torch.float64, device=dev)
        ry = torch.zeros_like(rw)
        start = col[:, :nmax] < nb[:, None]
        for m in range(1, int(widths.max()) + 1):
            rw = rw + hw[:, m - 1: m - 1 + nmax]
            ry = ry + hy[:, m - 1: m - 1 + nmax]
            used = (widths == m).any(0)
            if not bool(used.any()):
                continue
            ok = start & used[:, None] & (rw > 1e-14) & (rw < 1.0 - 1e-14)
            v = torch.where(ok, ry * ry / (rw * (1.0 - rw)), zero)
            top, i = v.max(1)
            up = top > best
            best = torch.where(up, top, best)
            bs = torch.where(up, torch.gather(ry, 1, i[:, None])[:, 0], bs)
            br = torch.where(up, torch.gather(rw, 1, i[:, None])[:, 0], br)
        sr[k:e], sb[k:e], rb[k:e] = best.cpu().numpy(), bs.cpu().numpy(), br.cpu().numpy()
        k = e
    return sr, sb, rb


def _trend64(f, sr):
    """Median-binned trend nodes (Sturges) and 1.4826 MAD."""
    n = int(math.floor(1.0 + 3.322 * math.log10(f.shape[0]) + 0.5))
    span = f[-1] - f[0]
    which = np.zeros(f.shape[0], np.int64) if span <= 0 else np.minimum(n - 1, np.floor((f - f[0]) * n / span)).astype(int)
    xs = [f[0] + (i + 0.5) * span / n for i in range(n) if (which == i).any()]
    ys = [np.median(sr[which == i]) for i in range(n) if (which == i).any()]
    med = np.median(sr)
    return np.asarray(xs), np.asarray(ys), med, 1.4826 * np.median(np.abs(sr - med))


def _search_exact(case, seed):
    if _grid_sums(case)[4] > EXACT_PAIRS:
        return None
    lc = _light_curves(case, seed)
    offsets, t, y, dy = lc[:4]
    grids = _coarse_grids64(lc) if case["kind"] == "coarse" else _grids64(lc)
    got = {k: [] for k in ("sr", "s", "r", "snr")}
    trend = np.zeros((case["stars"], 84))
    for s, (f, q) in enumerate(grids):
        sl = slice(int(offsets[s]), int(offsets[s + 1]))
        sr, sb, rb = _search64(t[sl], y[sl], dy[sl], f, q)
        xs, ys, med, sigma = _trend64(f, sr)
        trend[s, :3] = len(xs), sigma, med
        trend[s, 4: 4 + len(xs)] = xs
        trend[s, 44: 44 + len(ys)] = ys
        for k, v in (("sr", sr), ("s", sb), ("r", rb), ("snr", (sr - np.interp(f, xs, ys)) / sigma)):
            got[k].append(v)
    out = {k: np.concatenate(v) for k, v in got.items()}
    if case["kind"] == "coarse":
        out["trend"] = trend.reshape(-1)
    return out


def _conv64bit(x, w):
    """Same-padded convolution over positions: x [B][L][ci], w [9][co][ci]."""
    n = x.shape[1]
    xp = torch.nn.functional.pad(x, (0, 0, 4, 4))
    return sum(xp[:, k: k + n] @ w[k].T for k in range(9))


def _network64(p, x):
    """The logits from the flat parameters: conv(6->64), four conv(64->64), conv(64->1)."""
    o = 0

    def take(*shape):
        nonlocal o
        n = math.prod(shape)
        v = p[o: o + n].view(*shape)
        o += n
        return v

    h = torch.relu(_conv64bit(x, take(9, 64, NET_CH)) + take(64))
    for _ in range(4):
        h = torch.relu(_conv64bit(h, take(9, 64, 64)) + take(64))
    return _conv64bit(h, take(9, 64)[:, None, :])[:, :, 0] + take(1)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("search", "coarse"):
        return _search_exact(case, seed)
    if kind == "layer":
        x, dy, w, bias = _layer_inputs(case, seed)
        x64, dy64, w64 = x.double(), dy.double(), w.to(torch.bfloat16).double()
        n = x.shape[1]
        xp = torch.nn.functional.pad(x64, (0, 0, 4, 4))
        dw = torch.stack([torch.einsum("blo,bli->oi", dy64, xp[:, k: k + n]) for k in range(9)])
        dx = _conv64bit(dy64, w64.flip(0).transpose(1, 2)) * (x64 > 0)
        return dict(y=torch.relu(_conv64bit(x64, w64) + bias.double()), dx=dx, dw=dw, db=dy64.sum((0, 1)))
    if kind in ("propose", "train"):
        x0, labels = _spectra(case["batch"], seed)
        p = torch.from_numpy(_net_params(seed)).to(DEV).double()
        if kind == "propose":
            return dict(logits=torch.cat([_network64(p, x.double()) for x in x0.split(16)]))
        p.requires_grad_(True)
        for x, lab in zip(x0.split(8), labels.split(8)):
            z = _network64(p, x.double())
            loss = torch.nn.functional.binary_cross_entropy_with_logits(
                z, lab.double(), reduction="sum", pos_weight=torch.tensor(16.0, dtype=torch.float64, device=DEV))
            (loss / labels.numel()).backward()
        return dict(grads=p.grad.detach())
    return None
