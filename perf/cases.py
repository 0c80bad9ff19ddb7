"""Workloads of the resampled CrossCorr search, each one pass through the public API.

listed() gives the fixed cases, draw(rng) further ones of the same ranges, prepare() the
inputs and the plan a user's program holds before the call, run() one pass, work() the bytes
and operations a pass cannot do without, and exact() what run() returns, in 64 bits, written
directly from the definitions (plain torch, no code of the package).

Data: heterodyned complex series of two (or three) detectors, Gaussian noise in the locked
T_sft blocks, gaps in between, a weak signal from a circular binary orbit; a synthetic Earth
orbit and rotation; antenna functions that vary over a sidereal day; random orbital templates
around the Sco X-1 values (a_p ~ 1.44 s, P = 68023.7 s).
"""
import math

import numpy as np
import torch

import paper_1712_06515_gb300 as cc
from paper_1712_06515_gb300 import learned_interp, multiband

T0 = 1.1264e9
T_ASC = 1131415400.0
PERIOD = 68023.70
DAY = 86400.0
DT = 1.0
MU_F = 0.1
F_BAND = 0.5
PAD = 2048.0        # the ephemeris reaches this far beyond both ends of the data [s]


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------
def _search(name=None, **kw):
    case = {"kind": "search", "n_samples": 4096, "T_sft": 64, "T_short": 128, "T_max": 128, "f_h": 120.0, "f_band": F_BAND,
            "n_t": 4, "n_det": 2, "D": 8, "duty": 0.6, "lock": 21600.0, "jitter": 0.0, "ecc": False, "learned": False,
            "bf16": False}
    case.update(kw)
    if name:
        case["name"] = name
    return case


def _days(d):
    return int(round(d * DAY))


def listed():
    return [
        # a first look at about an hour of data, a handful of templates: launches and latency count
        _search("first_look", duty=0.85, lock=600.0, jitter=0.2),
        # one day, 1 Hz at 100 Hz, short segments and no lag, a 64-template grid
        _search("day_100hz", n_samples=_days(1), T_sft=240, T_short=240, T_max=0, f_h=100.0, f_band=1.0, n_t=64, duty=0.8),
        # a three-detector network, half-hour segments, the wider stencil, noise levels that vary per block
        _search("three_detectors", n_samples=_days(10), T_sft=360, T_short=1800, T_max=1800, f_h=110.0, n_t=48, n_det=3, D=16,
                jitter=0.2),
        # the single band of an observing run: 120 days, one-hour segments and lag, two batches of the template grid
        _search("o1_band", n_samples=_days(120), T_sft=360, T_short=3600, T_max=3600, f_h=150.0, n_t=144),
        # a month with a ragged end, 42-minute segments, eccentric orbits, the learned interpolator
        _search("ragged_learned", n_samples=_days(29.53) + 1, T_sft=360, T_short=2520, T_max=2520, f_h=150.0, n_t=97, ecc=True,
                learned=True, jitter=0.1),
        # the precision follow-up: ten-hour lag, few templates, the resampled series stored in BF16
        _search("long_lag_bf16", n_samples=_days(120), T_sft=360, T_short=36000, T_max=36000, f_h=150.0, n_t=16, bf16=True),
        # many bands from one graph launch, segment length by band frequency
        {"kind": "multiband", "name": "multiband", "n_samples": _days(10), "bands": "0,6,12,18,24,31", "n_t": 48},
        # the three stages called one by one, their outputs kept (a user who looks at the spectra)
        dict(_search("stages", n_samples=_days(20), T_sft=360, T_short=3600, T_max=3600, f_h=150.0, n_t=3), kind="stages"),
        # the detector-frame statistic for comparison, the method's pair loop (the default form)
        dict(_search("demod_pairs", n_samples=_days(30), T_sft=360, T_short=3600, T_max=3600, f_h=150.0, n_t=16), kind="demod",
             separable=False),
        # the same statistic in separable form over the whole run
        dict(_search("demod_separable", n_samples=_days(120), T_sft=360, T_short=3600, T_max=3600, f_h=150.0, n_t=16),
             kind="demod", separable=True),
        # input preparation: the SFTs of one detector's 120 days to the heterodyned series
        {"kind": "sft_series", "name": "sft_series", "n_blocks": 28800, "n_prime": 360, "T_sft": 360.0, "f_h": 150.0, "duty": 0.6},
        # candidates: the best (template, bin) of 2000 templates of the 120-day band
        {"kind": "topk", "name": "topk", "n_t": 2000, "T_max": 3600, "k": 100},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the listed ranges: the kinds weighted as they are listed, sizes spread over the logarithm of their
    ranges, template counts kept to the cost of the largest listed case."""
    kind = rng.choice(["search"] * 6 + ["multiband", "stages", "demod", "demod", "sft_series", "topk"])
    if kind == "multiband":
        bands = sorted(rng.sample(range(32), rng.randint(2, 6)))
        return {"kind": kind, "n_samples": _days(_log(rng, 2, 10)), "bands": ",".join(map(str, bands)), "n_t": rng.randint(3, 48)}
    if kind == "sft_series":
        n_prime = rng.choice([60, 72, 90, 120, 144, 180, 225, 240, 300, 360, 450, 480, 600, 720, 900, 1024])
        n_blocks = int(_log(rng, 100, 10368000 / n_prime))
        return {"kind": kind, "n_blocks": n_blocks, "n_prime": n_prime, "T_sft": float(n_prime), "f_h": float(rng.randint(20, 250)),
                "duty": rng.uniform(0.4, 1.0)}
    if kind == "topk":
        return {"kind": kind, "n_t": int(_log(rng, 1, 2000)), "T_max": 60 * rng.randint(5, 60), "k": int(_log(rng, 1, 1000))}
    if kind in ("stages", "demod"):
        T = 360 * rng.randint(4, 11)
        days = _log(rng, 2, 20 if kind == "stages" else 60)
        n_t = rng.randint(1, 3) if kind == "stages" else rng.randint(3, 16)
        case = _search(n_samples=_days(days) + rng.randint(0, 359), T_sft=360, T_short=T, T_max=T, f_h=rng.uniform(40.0, 250.0), n_t=n_t,
                       duty=rng.uniform(0.5, 0.9), jitter=rng.choice([0.0, 0.2]), D=rng.choice([8, 16]))
        case["kind"] = kind
        if kind == "demod":
            case["separable"] = rng.random() < 0.5
        return case
    # searches: segment lengths from two minutes to an hour (and ten hours with BF16 storage), whole minutes or odd numbers of
    # samples, with the segment's own lag or none
    long_lag = rng.random() < 0.15
    learned = not long_lag and rng.random() < 0.25
    n_s = 360 * rng.randint(30, 100) if long_lag else int(_log(rng, 120, 4000))
    if not long_lag and rng.random() < 0.7:
        n_s = 60 * max(2, n_s // 60)
    f_band = 0.5 if learned else rng.choice([0.1, 0.25, 0.5])     # the network is trained for 0.5 Hz bands
    days = _log(rng, 20, 120) if long_lag else _log(rng, max(0.05, 8 * n_s / DAY), 120)
    n_samples = _days(days) + rng.randint(0, 59)
    n_det = 3 if not long_lag and n_s <= 2048 and rng.random() < 0.2 else 2
    cost = n_samples * n_det * (4.0 if n_det == 3 else 3.0 if n_s < 1000 else 1.2)
    most = max(1, int(144 * 2 * 10368000 / cost / (2 if long_lag else 1)))
    n_t = max(1, min(int(_log(rng, 1, 400)), most))
    return _search(n_samples=n_samples, T_sft=360 if n_s % 360 == 0 else max(60, n_s // 4), T_short=n_s, T_max=n_s if rng.random() < 0.85 or long_lag else 0,
                   f_h=rng.uniform(40.0, 250.0), f_band=f_band, n_t=n_t, n_det=n_det, D=rng.choice([8, 8, 16, 12]),
                   duty=rng.uniform(0.5, 1.0), lock=_log(rng, 1800, 43200), jitter=rng.choice([0.0, 0.2]), ecc=rng.random() < 0.2,
                   learned=learned, bf16=long_lag)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
class Config:
    """The attributes CrossCorrPlan reads."""


class Detector:
    pass


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _lock_mask(n, duty, mean, rng):
    """Lock state per block: geometric lock and unlock lengths, trimmed at their ends to the duty cycle."""
    target = int(round(duty * n))
    if target >= n:
        return np.ones(n, bool)
    mean = max(mean, 1.0)
    gap = max(mean * (1.0 - duty) / duty, 1.0)
    mask, i, on = np.zeros(n, bool), 0, bool(rng.random() < duty)
    while i < n:
        m = int(rng.geometric(1.0 / (mean if on else gap)))
        mask[i:i + m] = on
        i += m
        on = not on
    while mask.sum() != target:
        extra = int(mask.sum()) - target
        on = extra > 0                      # flip blocks of this state, at the ends of their runs
        edge = np.flatnonzero(mask == on)
        inner = edge[(edge > 0) & (edge < n - 1)]
        ends = inner[(mask[inner - 1] != on) | (mask[inner + 1] != on)]
        pick = ends if len(ends) else edge
        mask[rng.choice(pick, size=min(abs(extra), max(1, len(pick) // 2)), replace=False)] = not on
    return mask


def _earth(t, q):
    """Detector position along the source direction [s]: a circular orbit of 499 s and the Earth's rotation."""
    return (0.94 * 499.0047838 * np.cos(6.1087 + 2 * np.pi * t / 31558149.76)
            + 0.0175 * np.cos(0.4 + 1.3 * q + 2 * np.pi * t / 86164.0905) - 0.003)


def _antenna(t, q):
    h = 0.7 + 1.1 * q + 2 * np.pi * t / 86164.0905
    a = 0.12 + 0.41 * np.cos(2 * h + 0.3 * q) + 0.09 * np.sin(h)
    b = 0.38 * np.sin(2 * h - 0.2 * q) + 0.21 * np.cos(h + 0.5)
    return a, b


def _templates(case, rng):
    n = case["n_t"]
    t = np.stack([rng.uniform(1.36, 1.52, n), T_ASC + rng.uniform(-300, 300, n), PERIOD + rng.uniform(-0.1, 0.1, n),
                  rng.uniform(0.0, 0.3, n) if case["ecc"] else np.zeros(n), rng.uniform(0, 2 * np.pi, n) if case["ecc"] else np.zeros(n)], 1)
    return t if case["ecc"] else t[:, :3].copy()


def _dataset(case, seed):
    """(config, detectors, x [Q, N_t] complex64 on the device, templates [n, 3 or 5] float64 on the host)."""
    dev = _device()
    rng = np.random.default_rng([seed, 11])
    gen = torch.Generator(device=dev)
    gen.manual_seed(7919 * int(seed) + 17)
    cfg = Config()
    cfg.t0, cfg.dt, cfg.n_samples, cfg.f_h, cfg.f_band = T0, DT, case["n_samples"], case["f_h"], case["f_band"]
    cfg.T_sft, cfg.T_max, cfg.T_short, cfg.mu_f = float(case["T_sft"]), float(case["T_max"]), float(case["T_short"]), MU_F
    cfg.D, cfg.n_det, cfg.pair_mode = case["D"], case["n_det"], 0
    n, nsft = cfg.n_samples, case["T_sft"]
    n_blk = -(-n // nsft)
    templates = _templates(case, rng)
    dets, xs = [], []
    for q in range(cfg.n_det):
        d = Detector()
        d.eph_t0, d.eph_dt, d.ab_t0, d.ab_dt = -PAD, 8.0, 0.0, 60.0
        d.ssb_delay = _earth(d.eph_t0 + d.eph_dt * np.arange(int(math.ceil((n + 2 * PAD) / d.eph_dt)) + 1), q)
        d.a_tab, d.b_tab = _antenna(d.ab_dt * np.arange(int(math.ceil(n / d.ab_dt)) + 2), q)
        lock = _lock_mask(n_blk, case["duty"], case["lock"] / nsft, rng)
        sig = 1.0 + case["jitter"] * (2.0 * rng.random(n_blk) - 1.0)
        d.sigma = np.where(lock, sig, 0.0)
        dets.append(d)
        s = torch.from_numpy(d.sigma).to(dev, torch.float32).repeat_interleave(nsft)[:n]
        noise = torch.randn(n, 2, generator=gen, device=dev) * (s * math.sqrt(0.5))[:, None]
        # a weak signal near the middle of the band, from the first template's orbit
        tau, _ = _source_time(d, templates[0], torch.arange(n, device=dev, dtype=torch.float64), cfg)
        tt = torch.arange(n, device=dev, dtype=torch.float64)
        f0 = cfg.f_h + 0.1462 * cfg.f_band
        cyc = torch.remainder(f0 * tau, 1.0) + torch.remainder((f0 - cfg.f_h) * tt, 1.0)
        amp = (0.035 * (s > 0)).to(torch.float64)
        sig_c = torch.polar(amp, 2 * math.pi * cyc).to(torch.complex64)
        xs.append(torch.view_as_complex(noise) + sig_c)
    return cfg, dets, torch.stack(xs), templates


def _band_case(case, b):
    """Band b of 32 over 20..250 Hz: segments from 240 s to an hour."""
    x = b / 31.0
    T = 60 * int(round(4.0 * 15.0 ** x))
    return _search(n_samples=case["n_samples"], T_sft=T, T_short=T, T_max=T, f_h=20.0 + 230.0 * x, n_t=case["n_t"])


def _plan(case, cfg, dets):
    return cc.CrossCorrPlan(cfg, dets, store=cc.STORE_BF16 if case["bf16"] else cc.STORE_FP32,
                            interp=cc.INTERP_LEARNED if case["learned"] else cc.INTERP_EXACT)


def _topk_case(case):
    return _search(n_samples=10 * case["T_max"], T_sft=case["T_max"] // 5, T_short=case["T_max"], T_max=case["T_max"], f_h=150.0, n_t=1)


def _rho_input(case, seed, n_f):
    gen = torch.Generator(device=_device())
    gen.manual_seed(104729 * int(seed) + 3)
    rho = torch.randn(case["n_t"], n_f, generator=gen, device=_device())
    rng = np.random.default_rng([seed, 5])
    for _ in range(5):                          # a few candidates above the noise
        rho[int(rng.integers(case["n_t"])), int(rng.integers(n_f))] = float(rng.uniform(6.0, 30.0))
    return rho


def _series_input(case, seed):
    dev = _device()
    rng = np.random.default_rng([seed, 23])
    gen = torch.Generator(device=dev)
    gen.manual_seed(15485863 + 31 * int(seed))
    lock = _lock_mask(case["n_blocks"], case["duty"], 60.0, rng)
    block = np.full(case["n_blocks"], -1, np.int64)
    block[lock] = np.arange(int(lock.sum()))
    n_sft = max(1, int(lock.sum()))
    band = torch.view_as_complex(torch.randn(n_sft, case["n_prime"], 2, generator=gen, device=dev) * math.sqrt(0.5 * case["n_prime"]))
    return band, torch.from_numpy(block).to(dev)


def prepare(case, seed):
    kind = case["kind"]
    state = {"kind": kind, "case": case}
    if kind == "sft_series":
        state["band"], state["block"] = _series_input(case, seed)
        state["out"] = torch.empty(case["n_blocks"] * case["n_prime"], dtype=torch.complex64, device=_device())
        return state
    if kind == "topk":
        cfg, dets, _, _ = _dataset(_topk_case(case), seed)
        state["plan"] = cc.CrossCorrPlan(cfg, dets)
        state["rho"] = _rho_input(case, seed, state["plan"].N_f)
        return state
    if kind == "multiband":
        bands = []
        for b in case["bands"].split(","):
            cfg, dets, x, tm = _dataset(_band_case(case, int(b)), seed + 1009 * int(b))
            bands.append((cfg, dets, x, torch.from_numpy(tm).to(x.device)))
        state["search"] = multiband.MultiBandSearch(bands).capture()
        return state
    cfg, dets, x, tm = _dataset(case, seed)
    state["x"], state["tm"] = x, torch.from_numpy(tm).to(x.device)
    state["plan"] = _plan(case, cfg, dets)
    if kind == "demod":
        state["plan"].demod_prepare(x)
        state["plan"].set_demod_form(case["separable"])
    return state


def run(state):
    kind = state["kind"]
    if kind == "sft_series":
        return cc.sfts_to_series(state["band"], state["block"], state["case"]["T_sft"], state["case"]["f_h"], out=state["out"])
    if kind == "multiband":
        return state["search"].run()
    plan = state["plan"]
    if kind == "topk":
        hits = plan.topk(state["rho"], state["case"]["k"])
        return {name: np.ascontiguousarray(hits[name]) for name in ("tmpl", "bin", "freq", "rho")}
    if kind == "demod":
        return plan.demod_search(state["tm"])
    if kind == "stages":
        n_t = state["tm"].shape[0]
        ab, norm = plan.resample(state["x"], state["tm"])
        F = plan.segment_fft(ab, n_t)
        return {"ab": ab, "norm": norm, "F": F, "rho": plan.pair_accumulate(F, norm, n_t)}
    return plan.search(state["x"], state["tm"])


# ---------------------------------------------------------------------------
# Floors
# ---------------------------------------------------------------------------
def _layout(case):
    """Segments, resolution and output bins of a search (the definitions of the method)."""
    n_s = case["T_short"]
    r = case["T_max"] // n_s
    t_coh = 2.0 * case["T_max"] + n_s
    dlf = math.sqrt(6.0 * MU_F / math.pi) / t_coh
    n0 = (1.0 / DT / dlf) * math.ceil(dlf * t_coh)
    n_fft = 1
    while n_fft < n0:
        n_fft *= 2
    t_fft = n_fft * DT
    fb = case["f_band"]
    n_f = int(math.floor(fb / dlf))
    a, b = -fb / 2.0, 1.0 / t_fft
    f_r = a - math.copysign(1.0, a) * math.floor(abs(a) / b) * b
    f_fft = case["f_h"] + f_r - 0.5 / DT
    k0 = int(math.floor((case["f_h"] - fb / 2.0 - f_fft) * t_fft + 1e-9))
    kbar = k0 + np.floor(dlf * DT * n_fft * np.arange(n_f, dtype=np.float64)).astype(np.int64)
    return {"N_s": n_s, "M": case["n_samples"] // n_s, "R": r, "N_FFT": n_fft, "N_f": n_f, "f_r": f_r, "f_FFT": f_fft, "T_FFT": t_fft,
            "kbar": kbar}


def _search_work(case):
    """Inputs and rho once; operations of the locked part of the data: the interpolation, one
    zero-padded transform of twice the segment per (detector, weight, segment) (twice the
    length holds every lag of two segments), the pair products on that grid, one transform to
    the output resolution per template."""
    p = _layout(case)
    q, n_t, duty = case["n_det"], case["n_t"], case["duty"]
    taps = 8 if case["learned"] else 2 * case["D"] + 1
    g = 2 * p["N_s"]
    per = duty * q * p["M"] * p["N_s"] * (8.0 * taps + 30.0)
    per += 2 * duty * q * p["M"] * 5.0 * g * math.log2(g)
    per += 2 * duty * p["M"] * g * 8.0 * (p["R"] + 1)
    per += 5.0 * p["N_FFT"] * math.log2(p["N_FFT"])
    tables = q * (case["n_samples"] / 8.0 * 8 + case["n_samples"] / 60.0 * 8 + case["n_samples"] / case["T_sft"] * 8)
    return {"bytes": q * case["n_samples"] * 8.0 + tables + n_t * (40.0 + 4.0 * p["N_f"]), "flops": n_t * per}


def work(case):
    kind = case["kind"]
    if kind == "sft_series":
        n = case["n_prime"]
        return {"bytes": 8.0 * n * case["n_blocks"] * (1.0 + case["duty"]) + 8.0 * case["n_blocks"],
                "flops": case["duty"] * case["n_blocks"] * (5.0 * n * math.log2(n) + 8.0 * n)}
    if kind == "topk":
        return {"bytes": 4.0 * case["n_t"] * _layout(_topk_case(case))["N_f"], "flops": 0.0}
    if kind == "multiband":
        parts = [_search_work(_band_case(case, int(b))) for b in case["bands"].split(",")]
        return {k: sum(w[k] for w in parts) for k in ("bytes", "flops")}
    if kind == "stages":
        w = _search_work(case)
        p = _layout(case)
        series = case["n_t"] * 2 * 2 * p["M"] * p["N_s"] * 8.0
        spectra = case["n_t"] * 2 * 2 * p["M"] * p["N_f"] * 8.0
        return {"bytes": w["bytes"] + 2 * series + 2 * spectra, "flops": w["flops"]}
    if kind == "demod":
        n_blk = case["n_samples"] // case["T_sft"]
        p = _layout(case)
        sfts = case["duty"] * 2 * n_blk
        lags = case["T_max"] // case["T_sft"]
        pairs = sfts * (case["duty"] * 2 * lags + 0.5 * case["duty"])
        per = sfts * (97.0 if case["separable"] else 30.0) + (0.0 if case["separable"] else 12.0 * pairs)
        return {"bytes": sfts * (case["f_band"] * case["T_sft"] + 60) * 8.0 + case["n_t"] * (40.0 + 4.0 * p["N_f"]),
                "flops": case["n_t"] * p["N_f"] * per}
    return _search_work(case)


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------
def _lerp(t0, dt, tab, t):
    u = (t - t0) / dt
    i = torch.floor(u).clamp_(0, tab.numel() - 2).to(torch.int64)
    f = u - i
    v = tab[i]
    return v + f * (tab[i + 1] - v)


def _orbit(tm):
    a, tasc, P = (float(v) for v in tm[:3])
    e, w = (float(tm[3]), float(tm[4])) if len(tm) >= 5 else (0.0, 0.0)
    tp = tasc - T0
    if e != 0.0:
        E = 2.0 * math.atan2(math.sqrt(1 - e) * math.sin(-0.5 * w), math.sqrt(1 + e) * math.cos(-0.5 * w))
        tp -= (E - e * math.sin(E)) * P / (2 * math.pi)
    return a, tp, P, e, w


def _binary(orb, u, rate=False):
    """Roemer delay of the binary orbit at solar-system time u (and its rate)."""
    a, tp, P, e, w = orb
    om = 2 * math.pi / P
    M = 2 * math.pi * torch.remainder((u - tp) / P, 1.0)
    if e == 0.0:
        return (a * torch.sin(M), a * om * torch.cos(M)) if rate else a * torch.sin(M)
    E = M + e * torch.sin(M)
    for _ in range(12):
        E = E - (E - e * torch.sin(E) - M) / (1.0 - e * torch.cos(E))
    sE, cE, q = torch.sin(E), torch.cos(E), math.sqrt(1 - e * e)
    R = a * (math.sin(w) * (cE - e) + math.cos(w) * q * sE)
    return (R, a * (-math.sin(w) * sE + math.cos(w) * q * cE) * om / (1.0 - e * cE)) if rate else R


def _source_time(d, tm, t, cfg):
    """tau(t) - t and dtau/dt at detector times t."""
    tab = torch.from_numpy(np.asarray(d.ssb_delay)).to(t.device)
    u = (t - d.eph_t0) / d.eph_dt
    i = torch.floor(u).clamp_(0, tab.numel() - 2).to(torch.int64)
    slope = tab[i + 1] - tab[i]
    dl = tab[i] + (u - i) * slope
    R, dR = _binary(_orbit(tm), t + dl, rate=True)
    return dl - R, (1.0 + slope / d.eph_dt) * (1.0 - dR)


def _learned_taps(u, case, model):
    w, lo, hi = model
    nu = learned_halfwidth(case)
    s = torch.stack([2.0 * u - 1.0, torch.full_like(u, (2.0 * nu - lo - hi) / (hi - lo))], -1)
    h = torch.tanh(s @ w[0] + w[1])
    h = torch.tanh(h @ w[2] + w[3])
    return h @ w[4] + w[5]


def learned_halfwidth(case):
    """Half-width of the data's band in cycles per sample: the searched half-band and the Doppler wings."""
    return min(0.5, DT * (0.5 * case["f_band"] + 2.5e-4 * case["f_h"]))


def _resampled(case, cfg, d, x, tm, p, model):
    """x'_r with the heterodyne correction, the weights alpha, beta and sigma^2 at t(tau_r), r < M N_s."""
    dev = x.device
    n = p["M"] * p["N_s"]
    tau = torch.arange(n, device=dev, dtype=torch.float64) * DT
    orb = _orbit(tm)
    b = torch.zeros_like(tau)
    for _ in range(6):                          # contraction ~1e-4 a step
        b = _binary(orb, tau + b)
    tab = torch.from_numpy(np.asarray(d.ssb_delay)).to(dev)
    dl = _lerp(d.eph_t0, d.eph_dt, tab, tau)
    for _ in range(6):
        dl = _lerp(d.eph_t0, d.eph_dt, tab, (tau + b) - dl)
    dly = dl - b
    g = 0.5 - dly / DT
    fl = torch.floor(g)
    js = torch.arange(n, device=dev) + fl.to(torch.int64)
    de = (g - 0.5) - fl
    del tau, dl, g, fl, b
    N = x.numel()
    acc = torch.zeros(n, dtype=torch.complex128, device=dev)
    if model is not None:
        j0 = torch.where(de < 0, js - 1, js)
        c = _learned_taps(torch.where(de < 0, de + 1.0, de), case, model)
        for m in range(c.shape[1]):
            j = j0 - 3 + m
            acc += torch.where((j >= 0) & (j < N), x[j.clamp(0, N - 1)], 0.0) * c[:, m]
    else:
        D = case["D"]
        s = torch.sin(math.pi * de) / math.pi
        zero = de == 0
        for m in range(-D, D + 1):
            win = 0.54 - 0.46 * math.cos(math.pi * (m + D) / D)
            q = de - m
            c = torch.where(zero, 1.0 if m == 0 else 0.0, (-1.0 if m % 2 else 1.0) * s / torch.where(q == 0, 1.0, q)) * win
            j = js + m
            acc += torch.where((j >= 0) & (j < N), x[j.clamp(0, N - 1)], 0.0) * c
    acc *= torch.polar(torch.ones_like(dly), -2 * math.pi * torch.remainder(cfg.f_h * dly, 1.0))
    t = js.to(torch.float64) + de
    a = _lerp(d.ab_t0, d.ab_dt, torch.from_numpy(d.a_tab).to(dev), t)
    bb = _lerp(d.ab_t0, d.ab_dt, torch.from_numpy(d.b_tab).to(dev), t)
    nsft = case["T_sft"]
    q = torch.div(js, nsft, rounding_mode="floor")
    blk = torch.where((js - q * nsft == 0) & (de < 0), q - 1, q)
    sig = torch.from_numpy(d.sigma).to(dev)
    s2 = torch.where((blk >= 0) & (blk < sig.numel()), sig[blk.clamp(0, sig.numel() - 1)], 0.0) ** 2
    inv = torch.where(s2 > 0, 1.0 / torch.where(s2 > 0, s2, 1.0), 0.0)
    return acc, a * inv, bb * inv, s2


def _model(case, dev):
    if not case["learned"]:
        return None
    z = np.load(learned_interp.WEIGHTS)
    w = [torch.from_numpy(np.asarray(z[k], np.float64)).to(dev) for k in ("W1", "b1", "W2", "b2", "W3", "b3")]
    return w, float(z["nu_c_range"][0]), float(z["nu_c_range"][1])


def _pair_sums(F, R, first, acc):
    """acc += Re sum over the unordered pairs whose later segment is at index >= first of F [Q, K, w, N_f]."""
    Q, K = F.shape[:2]
    same = torch.zeros_like(F[0, first:])
    for X in range(Q):
        acc += (F[X, first:].conj() * same).real.sum((0, 1))
        same = same + F[X, first:]
    S = F.sum(0)
    for lag in range(1, R + 1):
        lo = max(first, lag)
        if lo < K:
            acc += (S[lo:].conj() * S[lo - lag:K - lag]).real.sum((0, 1))


def _template_exact(case, cfg, dets, x, tm, p, model, keep=False):
    """rho of one template; with `keep` also a_r and b_r, the segment norms and the spectra."""
    dev = x.device
    Q, M, N_s, N, R = len(dets), p["M"], p["N_s"], p["N_FFT"], p["R"]
    bins = torch.from_numpy(p["kbar"]).to(dev)
    idx = torch.remainder(bins - N // 2, N)
    r = torch.arange(M * N_s, device=dev, dtype=torch.float64)
    rot = torch.polar(torch.ones_like(r), -2 * math.pi * torch.remainder(p["f_r"] * r * DT, 1.0))
    ab = torch.empty(Q, 2, M, N_s, dtype=torch.complex128, device=dev)
    norm = torch.empty(Q, M, 3, dtype=torch.float64, device=dev)
    for X, d in enumerate(dets):
        xr, al, be, s2 = _resampled(case, cfg, d, x[X], tm, p, model)
        xr *= rot
        ab[X, 0] = (xr * al).view(M, N_s)
        ab[X, 1] = (xr * be).view(M, N_s)
        for i, v in enumerate((al * al * s2, be * be * s2, al * be * s2)):
            norm[X, :, i] = v.view(M, N_s).sum(1)
    raw = torch.zeros(p["N_f"], dtype=torch.float64, device=dev)
    spectra = torch.empty(Q, M, 2, p["N_f"], dtype=torch.complex128, device=dev) if keep else None
    step = max(R + 1, int(4e9 / (16.0 * N * Q * 2)))
    k0 = 0
    while k0 < M:
        lo, hi = max(0, k0 - R), min(M, k0 + step)
        Y = torch.fft.fft(ab[:, :, lo:hi].transpose(1, 2), n=N)[..., idx]
        # the segment-start phase exp(-2 pi i (kbar - N/2) K N_s / N), its index reduced exactly
        seg = torch.arange(lo, hi, device=dev) * N_s
        ph = torch.remainder(seg[:, None] * torch.remainder(bins - N // 2, N)[None, :], N).to(torch.float64)
        Y *= torch.polar(torch.ones(ph.shape, dtype=torch.float64, device=dev), -2 * math.pi * ph / N)[None, :, None, :]
        _pair_sums(Y, R, k0 - lo, raw)
        if keep:
            spectra[:, lo:hi] = Y
        k0 = hi
    D = 0.0
    for K in range(R + 1):
        for X in range(Q):
            for Yd in range(Q):
                if K == 0 and X >= Yd:
                    continue
                u, v = norm[X, :M - K], norm[Yd, K:]
                D += float((u[:, 0] * v[:, 0] + u[:, 1] * v[:, 1] + 2 * u[:, 2] * v[:, 2]).sum())
    rho = raw * (math.sqrt(2.0) / math.sqrt(D)) if D > 0 else torch.zeros_like(raw)
    if not keep:
        return rho
    return rho, ab.reshape(Q, 2, M * N_s), torch.cat([norm, torch.zeros_like(norm[..., :1])], -1), spectra


def _demod_exact(case, cfg, dets, x, templates, p):
    """The detector-frame statistic: two sinc-weighted bins per SFT, every pair of SFTs within T_max."""
    dev = x.device
    n = case["T_sft"]
    n_blk = case["n_samples"] // n
    T = n * DT
    lags = int(math.floor(case["T_max"] / T + 1e-9))
    df = (p["f_r"] - 0.5 / DT) + torch.from_numpy(p["kbar"]).to(dev).to(torch.float64) / p["T_FFT"]
    f = cfg.f_h + df
    tmid = (torch.arange(n_blk, device=dev, dtype=torch.float64) + 0.5) * T
    z, ah, bh = [], [], []
    for X, d in enumerate(dets):
        sig = torch.from_numpy(d.sigma).to(dev)[:n_blk]
        on = sig > 0
        sc = torch.where(on, 1.0 / torch.where(on, sig, 1.0), 0.0)
        z.append(torch.fft.fft(x[X, :n_blk * n].view(n_blk, n), dim=1) * (sc / math.sqrt(n))[:, None])
        for out, tab in ((ah, d.a_tab), (bh, d.b_tab)):
            out.append(math.sqrt(n) * sc * _lerp(d.ab_t0, d.ab_dt, torch.from_numpy(tab).to(dev), tmid))
    rows = []
    for tm in templates:
        src = [_source_time(d, tm, tmid, cfg) for d in dets]
        parts = []
        width = max(1, int(1.5e8 / n_blk))
        for c0 in range(0, f.numel(), width):
            fc, dfc = f[c0:c0 + width], df[c0:c0 + width]
            Y, XI = [], []
            for X in range(len(dets)):
                dly, dtau = src[X]
                pos = ((dtau - 1.0)[:, None] * fc[None, :] + dfc[None, :]) * T
                m0 = torch.floor(pos)
                k0 = m0 - pos                      # in (-1, 0]
                k1 = k0 + 1.0
                s0, s1 = torch.special.sinc(k0), torch.special.sinc(k1)
                i0 = torch.remainder(m0, n).to(torch.int64)
                sg = 1.0 - 2.0 * torch.remainder(m0, 2.0)
                v = sg * (s0 * torch.gather(z[X], 1, i0) - s1 * torch.gather(z[X], 1, torch.remainder(i0 + 1, n)))
                cyc = torch.remainder(dly[:, None] * fc[None, :], 1.0) + torch.remainder(tmid[:, None] * dfc[None, :], 1.0)
                Y.append(v * torch.polar(torch.ones_like(cyc), -2 * math.pi * cyc))
                XI.append(s0 * s0 + s1 * s1)
            raw, den = torch.zeros_like(fc), torch.zeros_like(fc)
            for lag in range(lags + 1):
                if lag >= n_blk:
                    break
                for X in range(len(dets)):
                    for V in range(len(dets)):
                        if lag == 0 and X >= V:
                            continue
                        a, b = slice(0, n_blk - lag), slice(lag, n_blk)
                        g = ((ah[X][a] * ah[V][b] + bh[X][a] * bh[V][b]) / 10.0)[:, None]
                        y, w = Y[X][a], Y[V][b]
                        raw += 2.0 * (g * (y.real * w.real + y.imag * w.imag)).sum(0)
                        den += (g * g * XI[X][a] * XI[V][b]).sum(0)
            parts.append(torch.where(den > 0, raw / torch.sqrt(2.0 * torch.where(den > 0, den, 1.0)), 0.0))
        rows.append(torch.cat(parts))
    return torch.stack(rows)


def _search_exact(case, seed):
    cfg, dets, x, templates = _dataset(case, seed)
    x = x.to(torch.complex128)
    p = _layout(case)
    model = _model(case, x.device)
    return torch.stack([_template_exact(case, cfg, dets, x, tm, p, model) for tm in templates])


def exact(case, seed):
    kind = case["kind"]
    if kind == "sft_series":
        band, block = _series_input(case, seed)
        n = case["n_prime"]
        j = torch.arange(n, device=band.device)
        y = torch.fft.ifft(band.to(torch.complex128), dim=1) * (n / case["T_sft"]) * (1.0 - 2.0 * (j % 2))
        K = torch.arange(case["n_blocks"], device=band.device, dtype=torch.float64)
        ph = torch.polar(torch.ones_like(K), -2 * math.pi * torch.remainder(case["f_h"] * (K * case["T_sft"]), 1.0))
        return (torch.where((block >= 0)[:, None], y[block.clamp(min=0)], 0.0) * ph[:, None]).reshape(-1)
    if kind == "topk":
        p = _layout(_topk_case(case))
        rho = _rho_input(case, seed, p["N_f"]).cpu().numpy().reshape(-1)
        k = min(case["k"], rho.size)
        part = np.flatnonzero(rho >= np.partition(rho, rho.size - k)[rho.size - k])
        order = part[np.lexsort((part, -rho[part].astype(np.float64)))][:k]
        b = order % p["N_f"]
        return {"tmpl": (order // p["N_f"]).astype(np.int64), "bin": b.astype(np.int32),
                "freq": p["f_FFT"] + p["kbar"][b] / p["T_FFT"], "rho": rho[order]}
    if kind == "multiband":
        return [_search_exact(_band_case(case, int(b)), seed + 1009 * int(b)) for b in case["bands"].split(",")]
    if kind == "search":
        # 64-bit time of a template, seconds on the device (measured): 0.1 for 120 days of two detectors
        if case["n_t"] * case["n_samples"] * case["n_det"] > 144 * 2 * 10368000:
            return None
        return _search_exact(case, seed)
    cfg, dets, x, templates = _dataset(case, seed)
    x = x.to(torch.complex128)
    p = _layout(case)
    if kind == "demod":
        return _demod_exact(case, cfg, dets, x, templates, p)
    rows = [_template_exact(case, cfg, dets, x, tm, p, None, keep=True) for tm in templates]
    return {"ab": torch.stack([r[1] for r in rows]), "norm": torch.stack([r[2] for r in rows]),
            "F": torch.stack([r[3] for r in rows]), "rho": torch.stack([r[0] for r in rows])}
