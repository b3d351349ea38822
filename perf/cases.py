"""The work users of this library have it do, as cases that can be timed and compared.

Every case goes through the public Python entry points (the same names as the C ABI):

  search   one light curve from device-resident inputs: resample, linear search with its three
           outputs, periodic search (Plan + DeviceSearch.run)
  host     the same from host buffers, as a script calls it (cetra_linear_search, then
           cetra_periodic_search, or several rounds of search-and-mask)
  events   single-transit events of one curve (resample, linear search, greedy events)
  batch    many curves of uneven length in one run (Batch.run)
  propose  the learned-proposal search of a batch (Batch.search_proposed)
  forward  transit probabilities of a chunk of curves (CNN.forward)
  train    loss and gradients of one mini-batch (CNN.backward)
  comb     interval scores of proposal maps (cetra_cnn_comb)

Inputs are synthetic light curves made from the seed: white noise, planets, gaps, dropped points.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2503_20875_gb300 as cetra
from paper_2503_20875_gb300 import _native

DAY_S = 86400.0
HOUR = 1.0 / 24.0
BINS = 4096      # feature bins of a curve (the proposal network's input length)
EVENTS = 10      # single-transit events asked for
SECTOR = 27.4    # days of one observing sector of a batch curve, 1 d of gap between sectors


def _search(name, cadence_s, days, n_dur, d_lo, d_hi, n_per, p_lo, p_hi, step_s=0.0,
            precision="fp32", gap=0.0, offset=0.0, drop=0.0, kind="search", rounds=1):
    """step_s = 0: the t0 step is the cadence; durations in hours, log-spaced; periods in days,
    log-spaced; gap: days missing from the middle; drop: fraction of the points missing."""
    c = dict(kind=kind, cadence_s=float(cadence_s), days=float(days), n_dur=int(n_dur),
             d_lo=float(d_lo), d_hi=float(d_hi), n_per=int(n_per), p_lo=float(p_lo),
             p_hi=float(p_hi), step_s=float(step_s or cadence_s), precision=precision,
             gap=float(gap), offset=float(offset), drop=float(drop), rounds=int(rounds))
    return dict(c, name=name) if name else c


def listed():
    return [
        # One sector of 30-min full-frame data, a short period grid: the smallest useful call,
        # where launches and latency count.
        _search("search_30min_sector", 1800, 27.4, 16, 1, 16, 200, 0.5, 13.7, step_s=600),
        # 27 d of 2-min TESS data, 2,000 periods: the ordinary single-target search.
        _search("search_2min_27d", 120, 27, 10, 0.5, 6, 2000, 0.5, 13.5),
        # 27 d of 20-s TESS data with a mid-sector gap, 50,000 periods: high cadence.
        _search("search_20s_27d", 20, 27, 20, 0.5, 12, 50000, 0.5, 13.5, gap=1.0),
        # The same curve with compensated sums (the precision form).
        _search("search_20s_27d_kahan", 20, 27, 20, 0.5, 12, 50000, 0.5, 13.5, gap=1.0,
                precision="kahan"),
        # Four years of 1-min data at Julian dates, 100,000 periods up to 700 d: the largest.
        _search("search_1min_4yr", 60, 1461, 30, 1, 16, 100000, 1, 700, offset=2.45e6),
        # Search and three rounds of mask-and-search of an ordinary curve from host buffers.
        _search("host_2min_27d", 120, 27, 10, 0.5, 6, 2000, 0.5, 13.5, kind="host", rounds=3),
        # Single-transit events of the four-year curve.
        _search("events_1min_4yr", 60, 1461, 30, 1, 16, 0, 1, 700, offset=2.45e6, kind="events"),
        # A survey batch: 64 curves of 1 to 13 sectors at 30 min, every period from 0.5 d to half
        # of each baseline.
        dict(name="batch_64", kind="batch", curves=64, sectors=13, n_dur=16),
        # The learned proposal on a larger batch: 5 % of the period intervals are folded.
        dict(name="propose_128", kind="propose", curves=128, sectors=13, n_dur=16, frac=0.05),
        # The proposal network on a chunk of curves.
        dict(name="forward_256", kind="forward", curves=256, n_dur=16),
        # One mini-batch of its training.
        dict(name="train_32", kind="train", curves=32, n_dur=16),
        # Interval scores of a chunk of proposal maps.
        dict(name="comb_256", kind="comb", curves=256, sectors=13, intervals=512),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search"] * 6 + ["host", "events", "batch", "propose", "forward", "train",
                                        "comb"])
    if kind in ("search", "host", "events"):
        cad = rng.choice([20, 60, 120, 120, 200, 600, 1800])
        most = min(1461.0, 2.1e6 * cad / DAY_S) if kind == "events" else \
            min(1461.0, 3e5 * cad / DAY_S)
        days = math.exp(rng.uniform(math.log(13.0), math.log(max(14.0, most))))
        step = cad * rng.choice([1.0, 1.0, 1.0, 2.0, 1.0 / 3.0 if cad >= 600 else 1.0])
        n_dur = rng.randint(5, 30)
        d_lo = max(rng.uniform(0.5, 2.0), 3.0 * cad / 3600.0)
        d_hi = rng.uniform(5.0, 16.0)
        n_per = _log_int(rng, 101, 50000)
        cells = days * DAY_S / step * n_dur
        n_per = max(64, min(n_per, int(2.0e11 / cells)))  # well below the largest listed case
        if kind == "events":
            n_per = 0
        if kind == "host":
            n_per = min(n_per, 9001)
        p_lo = rng.uniform(0.5, 1.5)
        return _search("", cad, round(days, 3), n_dur, round(d_lo, 3), round(d_hi, 3), n_per,
                       round(p_lo, 3), round(rng.uniform(0.3, 0.5) * days, 3), step_s=step,
                       precision="kahan" if rng.random() < 0.25 else "fp32",
                       gap=rng.choice([0.0, 0.0, 1.0]), offset=rng.choice([0.0, 2.45e6]),
                       drop=rng.choice([0.0, 0.03]), kind=kind,
                       rounds=rng.choice([1, 3]) if kind == "host" else 1)
    if kind == "batch":
        return dict(kind=kind, curves=_log_int(rng, 3, 64), sectors=rng.choice([1, 3, 6, 13]),
                    n_dur=rng.choice([8, 11, 16]))
    if kind == "propose":
        return dict(kind=kind, curves=_log_int(rng, 8, 128), sectors=rng.choice([3, 6, 13]),
                    n_dur=rng.choice([8, 16]), frac=round(rng.uniform(0.03, 0.2), 3))
    if kind == "forward":
        return dict(kind=kind, curves=_log_int(rng, 1, 256), n_dur=rng.choice([8, 11, 16, 32]))
    if kind == "train":
        return dict(kind=kind, curves=_log_int(rng, 2, 64), n_dur=rng.choice([8, 11, 16, 32]))
    return dict(kind="comb", curves=_log_int(rng, 4, 256), sectors=rng.choice([1, 3, 13]),
                intervals=rng.choice([128, 300, 512]))


# ------------------------------------------------------------------------------- inputs

def _log_grid(lo, hi, n):
    return np.exp(np.linspace(math.log(lo), math.log(hi), int(n)))


def _template(n=4096):
    """A transit from first to last contact: a chord at impact parameter 0.32 across a disk with
    quadratic limb darkening, its ends smoothed over the ingress of a small planet."""
    x = np.linspace(-1.0, 1.0, n)
    r2 = 0.32 ** 2 + (1.0 - 0.32 ** 2) * x * x
    mu = np.sqrt(np.clip(1.0 - r2, 0.0, 1.0))
    prof = (1.0 - 0.4804 * (1.0 - mu) - 0.1867 * (1.0 - mu) ** 2)
    prof = prof * np.clip((1.0 - np.abs(x)) / 0.06, 0.0, 1.0)
    return (prof / prof.max()).astype(np.float32)


def _inject(t, P, t0, D, depth, tmpl):
    ph = t - t0
    ph = ph - np.round(ph / P) * P
    x = (ph + 0.5 * D) / D
    inside = (x >= 0.0) & (x <= 1.0)
    out = np.zeros(t.size)
    out[inside] = depth * np.interp(x[inside] * (tmpl.size - 1), np.arange(tmpl.size), tmpl)
    return out


def _curve(case, rng, tmpl):
    """(time, flux, flux_err) of a single-curve case, on the host."""
    cad = case["cadence_s"] / DAY_S
    n = int(round(case["days"] / cad))
    t = np.arange(n, dtype=np.float64) * cad
    if case["gap"]:
        a = 0.48 * case["days"]
        t = t[(t < a) | (t >= a + case["gap"])]
    if case["drop"]:
        keep = rng.random(t.size) >= case["drop"]
        keep[0] = keep[-1] = True
        t = t[keep]
    sigma = rng.uniform(300e-6, 1000e-6)
    flux = 1.0 + rng.standard_normal(t.size) * sigma
    for frac, snr in ((0.21, 15.0), (0.43, 25.0)):
        P = case["p_lo"] * (case["p_hi"] / case["p_lo"]) ** (frac + 0.4 * rng.random())
        D = 13.0 * HOUR * (P / 365.0) ** (1.0 / 3.0)
        depth = snr * sigma / math.sqrt(max(1.0, case["days"] / P * D / cad))
        flux -= _inject(t, P, rng.uniform(0.0, P), D, depth, tmpl)
    err = np.full(t.size, sigma, np.float32)
    return t + case["offset"], flux.astype(np.float32), err


def _batch_curves(case, rng, tmpl):
    """CSR-packed curves of 1 to `sectors` sectors at 30 min, a planet in three of ten."""
    cad = 1800.0 / DAY_S
    n_s = int(SECTOR / cad)
    times, fluxes, errs = [], [], []
    for _ in range(case["curves"]):
        S = int(rng.integers(1, case["sectors"] + 1))
        t = np.concatenate([(SECTOR + 1.0) * k + np.arange(n_s) * cad for k in range(S)])
        T = t[-1]
        sig_c = 500e-6 * 10.0 ** rng.random()
        sig = sig_c * np.exp(0.2 * rng.standard_normal(t.size))
        flux = 1.0 + rng.standard_normal(t.size) * sig
        if rng.random() < 0.3:
            P = min(100.0, T / 2.0) ** rng.random()
            D = 13.0 * HOUR * (P / 365.0) ** (1.0 / 3.0)
            depth = rng.uniform(5.0, 20.0) * sig_c / math.sqrt(max(1.0, T / P * D / cad))
            flux -= _inject(t, P, rng.uniform(0.0, P), D, depth, tmpl)
        times.append(t)
        fluxes.append(flux.astype(np.float32))
        errs.append(sig.astype(np.float32))
    off = np.zeros(case["curves"] + 1, np.int64)
    off[1:] = np.cumsum([t.size for t in times])
    return off, np.concatenate(times), np.concatenate(fluxes), np.concatenate(errs)


def _features(case, seed):
    """Max-pooled likelihood ratios as the linear search gives them: the best of a few windows
    of noise per bin, wider durations smoother, and transits; labels mark the transits' bins."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    B, J = case["curves"], case["n_dur"]
    z = torch.randn((B, 1, BINS), generator=g, device="cuda")
    z = z + 0.6 * torch.randn((B, J, BINS), generator=g, device="cuda")
    P = 40.0 * 25.0 ** torch.rand((B, 1), generator=g, device="cuda")
    t0 = P * torch.rand((B, 1), generator=g, device="cuda")
    bins = torch.arange(BINS, device="cuda", dtype=torch.float32)[None, :]
    labels = (((bins - t0 + 2.0) % P) < 4.0).float()
    labels = labels * (torch.rand((B, 1), generator=g, device="cuda") < 0.5)
    z = 0.5 + z + 4.0 * labels[:, None, :]
    return (0.5 * z.clamp(min=0.0) ** 2).contiguous(), labels.contiguous()


def _weights(n_dur):
    """Parameters of a proposal network (each layer: weights [out][in][9], biases [out]), spread
    as a trained one's are; a program loads its own."""
    rng = np.random.default_rng(7)
    out = []
    for ci, co in ((n_dur, 32), (32, 32), (32, 32), (32, 1)):
        out.append(rng.standard_normal(co * ci * 9) * math.sqrt(2.0 / (9 * ci)))
        out.append(0.05 * rng.standard_normal(co))
    return np.concatenate(out).astype(np.float32)


def _network(ctx, n_dur, max_batch):
    net = cetra.CNN(ctx, n_dur, n_bins=BINS, max_batch=max_batch)
    net.set_params(_weights(n_dur))
    return net


def _durations(case):
    if "d_lo" in case:
        return _log_grid(case["d_lo"] * HOUR, case["d_hi"] * HOUR, case["n_dur"])
    return _log_grid(1.0 * HOUR, 16.0 * HOUR, case["n_dur"])


def _periods(case):
    return _log_grid(case["p_lo"], case["p_hi"], case["n_per"]) if case["n_per"] else \
        np.empty(0)


def _single(case, seed):
    rng = np.random.default_rng(seed)
    tmpl = _template()
    t, f, e = _curve(case, rng, tmpl)
    kw = dict(cadence=case["cadence_s"] / DAY_S, t0_step=case["step_s"] / DAY_S,
              precision=case["precision"])
    return t, f, e, _durations(case), tmpl, kw


# ------------------------------------------------------------------------------- the passes

def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": dict(case)}
    ctx = s["ctx"] = cetra.Context(0)
    if kind in ("search", "host", "events"):
        t, f, e, d, tmpl, kw = _single(case, seed)
        if kind == "host":
            s.update(t=t, f=f, e=e, d=d, tmpl=tmpl, kw=kw, P=_periods(case))
            return s
        plan = s["plan"] = cetra.Plan(ctx, t, f, e, d, tmpl, **kw)
        s["in"] = tuple(torch.from_numpy(a).cuda() for a in (t, f, e))
        if kind == "search":
            s["ds"] = cetra.DeviceSearch(ctx, plan, _periods(case))
        else:
            nb = int(_native.lib.cetra_monotransit_workspace_bytes(plan.handle, EVENTS))
            s["ws"] = torch.empty(nb, dtype=torch.uint8, device="cuda")
            # one record: dlogl, t0, duration, depth, depth_var (FP64), i (int64), j, padding
            s["ev"] = torch.zeros(EVENTS * 56, dtype=torch.uint8, device="cuda")
            s["n"] = torch.zeros(1, dtype=torch.int32, device="cuda")
            s["values"] = s["ev"].view(torch.float64).view(EVENTS, 7)[:, :5]
            s["index"] = s["ev"].view(torch.int64).view(EVENTS, 7)[:, 5:]
        return s
    if kind in ("batch", "propose"):
        rng = np.random.default_rng(seed)
        tmpl = _template()
        s["batch"] = cetra.Batch(ctx, None, _durations(case), tmpl, 0.5,
                                 csr=_batch_curves(case, rng, tmpl), cadence=1800.0 / DAY_S,
                                 t0_step=600.0 / DAY_S)
        if kind == "propose":
            s["cnn"] = _network(ctx, case["n_dur"], 64)
        return s
    if kind in ("forward", "train"):
        s["cnn"] = _network(ctx, case["n_dur"], case["curves"])
        s["f"], s["y"] = _features(case, seed)
        s["p"] = torch.empty((case["curves"], BINS), dtype=torch.float32, device="cuda")
        return s
    bw, nv, hi = _comb_bins(case, seed)
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    s["map"] = torch.rand((case["curves"], BINS), generator=g, device="cuda") * \
        torch.randn((case["curves"], BINS), generator=g, device="cuda") ** 2
    s["bw"], s["nv"] = torch.from_numpy(bw).cuda(), torch.from_numpy(nv).cuda()
    s["hi"] = hi
    s["scores"] = torch.empty((case["curves"], case["intervals"]), dtype=torch.float32,
                              device="cuda")
    return s


def _comb_bins(case, seed):
    """Bin widths (days), valid bins and the longest trial period of curves of 1 to `sectors`
    sectors on a 10-min t0 grid."""
    S = np.random.default_rng(seed).integers(1, case["sectors"] + 1, case["curves"])
    S[0] = case["sectors"]
    span = S * SECTOR + (S - 1) * 1.0
    I = np.floor((span + 16.0 * HOUR) * 144.0).astype(np.int64)
    width = -(-I // BINS)
    return width / 144.0, (-(-I // width)).astype(np.int32), float(span.max() / 2.0)


def run(s):
    kind, ctx = s["kind"], s["ctx"]
    if kind == "search":
        ds = s["ds"].run(*s["in"])
        return {"depth": ds.depth, "depth_var": ds.depth_var, "dlogl": ds.dlogl, "periodic": ds.out}
    if kind == "host":
        grid, depth, var, lr = cetra.cetra_linear_search(ctx, s["t"], s["f"], s["e"], s["d"],
                                                         s["tmpl"], **s["kw"])
        out = {"depth": depth, "depth_var": var, "dlogl": lr,
               "periodic": cetra.cetra_periodic_search(ctx, grid, s["P"])}
        if s["case"]["rounds"] > 1:
            out["rounds"] = cetra.cetra_search_iterative(ctx, grid, s["P"],
                                                         n_iter=s["case"]["rounds"])
        grid.close()
        return out
    if kind == "events":
        cetra.cetra_resample_device(ctx, s["plan"], *s["in"], s["ws"])
        cetra.cetra_linear_device(ctx, s["plan"], s["ws"])
        cetra.cetra_monotransits_device(ctx, s["plan"], s["ws"], EVENTS, s["ev"], s["n"])
        return {"values": s["values"], "index": s["index"], "n": s["n"]}
    if kind == "batch":
        return s["batch"].run()
    if kind == "propose":
        best, n_items, n_periods = s["batch"].search_proposed(s["cnn"],
                                                              top_frac=s["case"]["frac"])
        return {"best": best, "n_items": n_items, "n_periods": n_periods}
    if kind == "forward":
        s["cnn"].forward(s["f"], s["p"])
        return s["p"]
    if kind == "train":
        loss, grads = s["cnn"].backward(s["f"], s["y"], grads=True)
        return {"loss": loss, "grads": grads}
    cetra.cetra_cnn_comb(ctx, s["map"], s["bw"], 0.5, s["hi"], s["case"]["intervals"], s["scores"],
                         s["nv"])
    return s["scores"]


# ------------------------------------------------------------------------------- the work

def work(case):
    """Bytes: inputs read once, outputs written once. Flops: 4 per window point and t0 of the
    linear search (two multiply-adds), 2 per cell read of the fold (two adds)."""
    kind = case["kind"]
    if kind in ("search", "host", "events"):
        step = case["step_s"] / DAY_S
        d = _durations(case)
        n = case["days"] * DAY_S / case["cadence_s"]
        I = case["days"] / step
        lin = 4.0 * I * float(np.sum(d)) * DAY_S / case["cadence_s"]
        P = _periods(case)
        fold = 2.0 * I * float(sum(int(np.sum(P > x)) for x in d))
        rounds = 1 if kind != "host" else (case["rounds"] + 1 if case["rounds"] > 1 else 1)
        out = EVENTS * 56 if kind == "events" else 12.0 * I * d.size + 52.0 * P.size
        return {"bytes": 16.0 * n + 8.0 * P.size + out,
                "flops": lin * max(1, rounds - 1) + fold * rounds}
    if kind in ("batch", "propose"):
        # mean over S = 1 .. sectors sectors: I = span / 10 min, K = ln(span) / ln(ratio)
        I2 = K2 = pts = 0.0
        for S in range(1, case["sectors"] + 1):
            T = S * SECTOR + S - 1
            K = math.log(T) * 2.0 * T / HOUR
            I2 += T * 144.0 * K * case["n_dur"] / case["sectors"]
            K2 += K / case["sectors"]
            pts += S * SECTOR * 48.0 / case["sectors"]
        frac = case.get("frac", 1.0)
        return {"bytes": case["curves"] * (16.0 * pts + 80.0),
                "flops": 2.0 * case["curves"] * I2 * frac}
    if kind in ("forward", "train"):
        layers = 32 * case["n_dur"] + 32 * 32 * 2 + 32
        fl = 2.0 * 9 * layers * BINS * case["curves"]
        if kind == "train":
            fl = 3.0 * fl - 2.0 * 9 * 32 * case["n_dur"] * BINS * case["curves"]
        per = case["n_dur"] + 1
        return {"bytes": 4.0 * case["curves"] * BINS * per, "flops": fl}
    # comb: trials of one curve ln(hi / lo) V, each V cells (an add per cell)
    adds = 0.0
    for S in range(1, case["sectors"] + 1):
        I = (S * SECTOR + S - 1 + 16.0 * HOUR) * 144.0
        V = I / math.ceil(I / BINS)
        span = S * SECTOR + S - 1
        adds += V * V * math.log(span) / case["sectors"]
    return {"bytes": 4.0 * case["curves"] * (BINS + case["intervals"]),
            "flops": case["curves"] * adds}


# ------------------------------------------------------------------------------- 64-bit values

def _exact_geometry(case, t, d):
    """The resampled grid, the t0 grid and the periods' cells in FP64 (ticks of cadence / q)."""
    c = case["cadence_s"] / DAY_S
    ratio = (case["step_s"] / DAY_S) / c
    for q in range(1, 65):
        p = max(1, math.floor(ratio * q + 0.5))
        if abs(p / q - ratio) / ratio <= 1e-9:
            break
    pad = math.ceil(0.5 * float(d.max()) / c)
    n = 2 * pad + math.floor((t.max() - t.min()) / c + 0.5) + 1
    return c, p, q, pad, n, (n - 1) * q // p + 1


def _exact_linear(case, t, f, e, d, tmpl):
    """(A, B) [J][I] of the window sums A = sum m W y, B = sum m^2 W, as FP64 CUDA tensors."""
    c, p, q, pad, n, I = _exact_geometry(case, t, d)
    tt = torch.from_numpy(t).cuda()
    k = pad + torch.floor((tt - tt.min()) / c + 0.5).long()
    w = 1.0 / torch.from_numpy(e.astype(np.float64)).cuda() ** 2
    y = 1.0 - torch.from_numpy(f.astype(np.float64)).cuda()
    W = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, k, w)
    Wy = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, k, w * y)
    pos = np.arange(1024) * (tmpl.size - 1) / 1023.0
    i0 = np.minimum(np.floor(pos).astype(np.int64), tmpl.size - 2)
    T = tmpl.astype(np.float64)
    T = T[i0] * (1.0 - (pos - i0)) + T[i0 + 1] * (pos - i0)
    T = T / np.abs(T).max()
    J = d.size
    A = torch.zeros((J, I), dtype=torch.float64, device="cuda")
    B = torch.zeros((J, I), dtype=torch.float64, device="cuda")
    for j in range(J):
        Dt = d[j] * q / c
        for r in range(min(q, I)):
            m = np.arange(math.floor((r * p - 0.5 * Dt) / q) - 2,
                          math.ceil((r * p + 0.5 * Dt) / q) + 3)
            x = ((m * q - r * p).astype(np.float64) + 0.5 * Dt) / Dt
            inside = (x >= 0.0) & (x <= 1.0)
            m, x = m[inside], x[inside]
            v = T[np.floor(x * 1023.0 + 0.5).astype(np.int64)]
            U = (I - r + q - 1) // q
            lo, hi = int(m[0]), int(m[-1])
            left, right = max(0, -lo), max(0, hi + p * (U - 1) - (n - 1))
            wy = torch.nn.functional.pad(Wy, (left, right))
            ww = torch.nn.functional.pad(W, (left, right))
            a = torch.zeros(U, dtype=torch.float64, device="cuda")
            b = torch.zeros(U, dtype=torch.float64, device="cuda")
            for mk, vk in zip(m.tolist(), v.tolist()):
                s = mk + left
                a.add_(wy[s:s + p * (U - 1) + 1:p], alpha=vk)
                b.add_(ww[s:s + p * (U - 1) + 1:p], alpha=vk * vk)
            A[j, r::q], B[j, r::q] = a, b
    return A, B, c, p, q, I


def _exact_fold(A, B, d, P, c, p, q, I):
    """Largest (sum A)^2 / (2 sum B) of every period over durations below it and phases."""
    J = d.size
    out = torch.full((P.size,), float("nan"), dtype=torch.float64, device="cuda")
    for k, pk in enumerate(P.tolist()):
        Ps = (pk * q) / (c * p)
        use = int(np.sum(d < pk))  # the durations ascend
        if Ps < 1.0 or use == 0:
            continue
        nph = min(math.ceil(Ps), I)
        o = np.floor(np.arange(int((I + 0.5) / Ps) + 2) * Ps + 0.5).astype(np.int64)
        SA = torch.zeros((use, nph), dtype=torch.float64, device="cuda")
        SB = torch.zeros((use, nph), dtype=torch.float64, device="cuda")
        for x in o[o < I].tolist():
            n = min(nph, I - x)
            SA[:, :n] += A[:use, x:x + n]
            SB[:, :n] += B[:use, x:x + n]
        lr = torch.where(SB > 0, 0.5 * SA * SA / SB, torch.full_like(SA, -1.0))
        m = lr.max()
        out[k] = torch.where(m >= 0, m, torch.full_like(m, float("nan")))
    return out


def _exact_cnn(case, seed, train):
    f, y = _features(case, seed)
    flat = torch.from_numpy(_weights(case["n_dur"]))
    ws, at = [], 0
    for ci, co in ((case["n_dur"], 32), (32, 32), (32, 32), (32, 1)):
        w = flat[at:at + co * ci * 9].view(co, ci, 9).bfloat16().double().cuda()
        at += co * ci * 9
        b = flat[at:at + co].double().cuda()
        at += co
        ws += [w.requires_grad_(train), b.requires_grad_(train)]
    total, probs = 0.0, []
    for a in range(0, case["curves"], 16):  # a few curves at a time
        x = torch.log1p(f[a:a + 16].double())
        for l in range(4):
            x = torch.nn.functional.conv1d(x, ws[2 * l], ws[2 * l + 1], padding=4)
            if l < 3:
                x = torch.relu(x)
        x = x[:, 0]
        if not train:
            probs.append(torch.sigmoid(x))
            continue
        yy = y[a:a + 16].double()
        loss = (20.0 * yy * torch.nn.functional.softplus(-x)
                + (1.0 - yy) * torch.nn.functional.softplus(x)).sum() / (case["curves"] * BINS)
        loss.backward()
        total += float(loss)
    if not train:
        return torch.cat(probs)
    return {"loss": total, "grads": torch.cat([w.grad.reshape(-1) for w in ws]).cpu().numpy()}


def _exact_comb(case, seed):
    bw, nv, hi = _comb_bins(case, seed)
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    m = torch.rand((case["curves"], BINS), generator=g, device="cuda") * \
        torch.randn((case["curves"], BINS), generator=g, device="cuda") ** 2
    m = torch.cat([m.double(), torch.zeros((case["curves"], 1), dtype=torch.float64,
                                           device="cuda")], 1)
    n_int = case["intervals"]
    out = torch.zeros((case["curves"], n_int), dtype=torch.float64, device="cuda")
    for w in np.unique(bw).tolist():  # curves of the same length share their bins
        rows = torch.from_numpy(np.nonzero(bw == w)[0]).cuda()
        V = int(nv[np.nonzero(bw == w)[0][0]])
        for q in range(n_int):
            lo = 0.5 * (hi / 0.5) ** (q / n_int) / w
            up = 0.5 * (hi / 0.5) ** ((q + 1) / n_int) / w
            if up < 1.0 or lo > 0.5 * V:
                continue
            nP = max(1, math.ceil((up - lo) * V / lo))
            Pb = lo + (up - lo) * (np.arange(nP) + 0.5) / nP
            Pb = Pb[(Pb >= 1.0) & (Pb <= 0.5 * V)]
            best = torch.zeros(rows.numel(), dtype=torch.float64, device="cuda")
            sub = m[rows]
            for a in range(0, Pb.size, 32):
                F = torch.from_numpy(np.floor(Pb[a:a + 32] * 2.0 ** 32 + 0.5)
                                     .astype(np.int64)).cuda()
                nph = torch.from_numpy(np.ceil(Pb[a:a + 32]).astype(np.int64)).cuda()
                ph = torch.arange(int(nph.max()), device="cuda")
                e = torch.arange(int(V / Pb[a]) + 2, device="cuda")
                te = ((ph[None, :, None] << 32) + e[None, None, :] * F[:, None, None]
                      + (1 << 31)) >> 32
                ok = (te < V) & (ph[None, :, None] < nph[:, None, None])
                E = ok.sum(2).clamp(min=1).double()
                te = torch.where(ok, te, torch.full_like(te, BINS))
                for c0 in range(0, rows.numel(), 8):
                    s = sub[c0:c0 + 8][:, te].sum(3) / torch.sqrt(E)
                    best[c0:c0 + 8] = torch.maximum(best[c0:c0 + 8], s.flatten(1).max(1).values)
            out[rows, q] = best
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("search", "host"):
        t, f, e, d, tmpl, _ = _single(case, seed)
        A, B, c, p, q, I = _exact_linear(case, t, f, e, d, tmpl)
        good = B > 0
        nan = torch.full_like(A, float("nan"))
        lin = {"depth": torch.where(good, A / B, nan), "depth_var": torch.where(good, 1.0 / B, nan),
               "dlogl": torch.where(good, 0.5 * A * A / B, nan)}
        none = dict.fromkeys(("t0", "duration", "depth", "depth_var"))
        P = _periods(case)
        # the fold in 64 bits takes an operation for every epoch of every period
        epochs = float(np.sum(float(t.max() - t.min()) / P))
        per = _exact_fold(A, B, d, P, c, p, q, I) if epochs < 2e5 else None
        out = dict(lin, periodic=dict(none, dlogl=per))
        if kind == "host":
            out = {k: v.cpu().numpy() for k, v in lin.items()}
            out["periodic"] = dict(none, best_k=None,
                                   dlogl=None if per is None else per.cpu().numpy())
            if case["rounds"] > 1:
                out["rounds"] = None
        return out
    if kind in ("forward", "train"):
        return _exact_cnn(case, seed, kind == "train")
    if kind == "comb":
        return _exact_comb(case, seed)
    return None  # events, batch and propose: chosen models, whose indices have no 64-bit value
