"""Kernel variants at the sizes where they can go wrong, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from oracle import cnn as ocnn
from _parity import compare_linear, gpu_search, oracle_search

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [0.0, 2.45e6])
def test_resample_at_half_points(offset):
    """Times within a few ulps of the midpoint between two grid points: the nearest point is
    decided by the FP64 division, and its reciprocal shortcut must not decide otherwise."""
    c = 120.0 / 86400.0
    k = np.arange(600)
    t = offset + k * c
    half = (k % 3) == 1
    t[half] = offset + (k[half] + 0.5) * c
    for u in range(4):  # 0, 1, 2, 3 ulps either side
        sel = half & (k % 4 == u)
        for _ in range(u):
            t[sel] = np.nextafter(t[sel], np.where(k[sel] % 8 < 4, np.inf, -np.inf))
    rng = np.random.default_rng(3)
    f = (1.0 + rng.normal(0.0, 1e-3, t.size)).astype(np.float32)
    e = np.full(t.size, 1e-3, np.float32)
    d = np.array([0.03, 0.1])
    tm = np.ones(64, np.float32)
    kw = dict(cadence=c, t0_step=c)
    compare_linear(gpu_search(t, f, e, d, tm, **kw), oracle_search(t, f, e, d, tm, **kw), d)


@pytest.mark.parametrize("T,bin_days,valid,lo,hi,n", [
    (256, 0.4, 256, 0.5, 0.56, 2),       # 2 phases: eight trials share a warp
    (256, 0.1, 256, 0.7, 0.74, 2),       # 8 phases: four trials
    (256, 0.1, 231, 1.5, 1.58, 3),       # 16 phases: two trials
    (256, 0.02, 255, 0.6, 0.65, 2),      # 31 to 33 phases: one and two rows
    (1024, 0.01, 1001, 1.27, 1.29, 2),   # 127 to 129 phases: four and five rows
    (1024, 0.01, 1024, 3.5, 3.53, 2),    # 350 phases: 12 rows, of which 11 hold phases
    (1536, 0.01, 1536, 7.6, 7.68, 2),    # 768 phases: two units, two epochs
    (25088, 0.002, 1200, 0.6, 0.61, 1),  # a map that is not staged in shared memory
])
def test_comb_shapes(T, bin_days, valid, lo, hi, n):
    """Scores over the shapes the comb's lanes take; the sums are of at most 256 terms, each
    rounded once (relative error below 256 * 2^-24 = 1.6e-5, far less for random signs)."""
    import torch
    from paper_2503_20875_gb300 import Context, cetra_cnn_comb
    rng = np.random.default_rng(T)
    m = (rng.uniform(size=(3, T)) ** 6).astype(np.float32)
    bw = np.array([bin_days, bin_days * 1.1, bin_days])
    nv = np.array([valid, valid, valid // 2], np.int32)
    scores = torch.empty((3, n), dtype=torch.float32, device="cuda")
    cetra_cnn_comb(Context(0), torch.from_numpy(m).cuda(), torch.from_numpy(bw).cuda(), lo, hi, n,
                   scores, torch.from_numpy(nv).cuda())
    np.testing.assert_allclose(scores.cpu().numpy(), ocnn.comb(m, bw, lo, hi, n, nv), rtol=1.6e-5,
                               atol=1e-7)


@pytest.mark.parametrize("cin,T,B", [(1, 256, 1), (16, 256, 3), (17, 512, 2), (32, 768, 2)])
def test_network_tiles(cin, T, B):
    """Probabilities over channel counts that fill one and two K steps, one to four tiles per
    curve, a ragged last tile, zero padding at both ends and large inputs. Tolerance: 288 products
    per sum and layer, as in the network's parity test."""
    import torch
    from paper_2503_20875_gb300 import CNN, Context
    rng = np.random.default_rng(cin + T)
    f = (rng.chisquare(1, (B, cin, T)) * 3.0).astype(np.float32)
    f[0, 0, :5] = 1e4
    f[-1, -1, -3:] = 3e7
    net = CNN(Context(0), cin, n_bins=T, max_batch=B, seed=cin)
    p = net.get_params()
    p += rng.normal(0.0, 0.01, p.size).astype(np.float32)  # biases too
    net.set_params(p)
    out = torch.empty((B, T), dtype=torch.float32, device="cuda")
    net.forward(torch.from_numpy(f).cuda(), out)
    np.testing.assert_allclose(out.cpu().numpy(), ocnn.probabilities(p, f), rtol=0, atol=2e-5)


@pytest.mark.parametrize("n_dur", [2, 3, 7])
@pytest.mark.parametrize("flat", [False, True])
def test_fold_shapes(n_dur, flat):
    """Periods whose phase counts and epochs sit at the edges of the fold's tiles: several duration
    rows per tile with 1 to 4 rows of lanes at work, the change to whole tiles, ragged last tiles,
    and winners summed over 1 to 70 epochs. Flat data has equal windows everywhere: the first one
    wins. Tolerances are the parity tests' (compare_periodic)."""
    from _parity import compare_periodic
    from synth.lightcurves import custom
    step = 120.0 / 86400.0
    phases = [40, 75, 111, 112, 113, 149, 150, 223, 224, 225, 298, 299, 336, 337, 447, 448, 449, 672,
              673, 896, 897, 1500, 2699, 2750]
    periods = np.sort(np.concatenate([np.array(phases) * step, (np.array(phases) - 0.4) * step]))
    w = custom(seed=n_dur, n_points=2800, cadence_s=120.0,
               durations_h=np.linspace(0.3, 1.2, n_dur), periods=periods,
               planets=[] if flat else [dict(P=0.42, t0=0.1, D=0.02, depth=3e-3)])
    if flat:
        w.flux[:] = 1.0
    args = (w.time, w.flux, w.flux_err, w.durations, w.template, periods)
    kw = dict(cadence=w.cadence, t0_step=w.t0_step)
    g, o = gpu_search(*args, **kw), oracle_search(*args, **kw)
    if flat:
        np.testing.assert_array_equal(g["periodic"]["dlogl"], o["periodic"]["dlogl"])
        np.testing.assert_array_equal(g["periodic"]["i"], o["periodic"]["i"])
        np.testing.assert_array_equal(g["periodic"]["j"], o["periodic"]["j"])
    else:
        compare_periodic(g, o, periods)


@pytest.mark.parametrize("n_points", [40, 300, 5000])
def test_event_segments(n_points):
    """Single-transit events whose hidden cells lie in one segment, cross segments and cover the
    whole grid: the greedy picks of a plain scan over the same linear grid."""
    from paper_2503_20875_gb300 import Context, cetra_linear_search, cetra_monotransit_search
    from synth.lightcurves import custom
    w = custom(seed=n_points, n_points=n_points, cadence_s=120.0, durations_h=(0.4, 1.1, 9.0))
    ctx = Context(0)
    grid, depth, _, lr = cetra_linear_search(ctx, w.time, w.flux, w.flux_err, w.durations,
                                             w.template, cadence=w.cadence, t0_step=w.t0_step)
    ev = cetra_monotransit_search(ctx, grid, 12)
    score = np.where(depth > 0, lr, -1.0).astype(np.float64)
    reach = w.durations / w.t0_step
    i_all = np.arange(lr.shape[1])
    for m in range(len(ev["i"])):
        j, i = np.unravel_index(np.nanargmax(score), score.shape)
        assert (ev["i"][m], ev["j"][m]) == (i, j)
        score[:, np.abs(i_all - i) < reach[j]] = -1.0
    assert len(ev["i"]) == 12 or not np.nanmax(score) > 0


@pytest.mark.parametrize("n_points,max_events", [(2, 1), (40, 1), (5000, 1), (5000, 3)])
def test_event_scratch_limit(n_points, max_events):
    """Events in a workspace with one word per t0 cell and event, and nothing past its end
    written: the first picks of the host form."""
    import ctypes
    import torch
    from paper_2503_20875_gb300 import (Context, Plan, cetra_linear_device, cetra_linear_search,
                                        cetra_monotransit_search, cetra_monotransits_device,
                                        cetra_resample_device)
    from paper_2503_20875_gb300 import _native as N
    from synth.lightcurves import custom
    w = custom(seed=n_points, n_points=n_points, cadence_s=120.0, durations_h=(0.4, 1.1, 9.0))
    ctx = Context(0)
    grid, _, _, _ = cetra_linear_search(ctx, w.time, w.flux, w.flux_err, w.durations, w.template,
                                        cadence=w.cadence, t0_step=w.t0_step)
    ev = cetra_monotransit_search(ctx, grid, max_events)
    plan = Plan(ctx, w.time, w.flux, w.flux_err, w.durations, w.template, cadence=w.cadence,
                t0_step=w.t0_step)
    nb = N.lib.cetra_workspace_bytes(plan.handle, plan.info["n_t0"] + max_events)
    buf = torch.full((nb + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
    ws = buf[:nb]
    t, f, e = (torch.from_numpy(np.ascontiguousarray(x)).cuda()
               for x in (w.time, w.flux, w.flux_err))
    cetra_resample_device(ctx, plan, t, f, e, ws)
    cetra_linear_device(ctx, plan, ws, None, None, None)
    rec = ctypes.sizeof(N.cetra_event)
    d_ev = torch.zeros(max_events * rec, dtype=torch.uint8, device="cuda")
    d_n = torch.zeros(1, dtype=torch.int32, device="cuda")
    cetra_monotransits_device(ctx, plan, ws, max_events, d_ev, d_n)
    torch.cuda.synchronize()
    raw = d_ev.cpu().numpy().tobytes()
    got = [N.cetra_event.from_buffer_copy(raw[rec * m:rec * (m + 1)])
           for m in range(int(d_n.item()))]
    assert [(x.i, x.j) for x in got] == list(zip(ev["i"], ev["j"]))
    assert bool((buf[nb:] == 0xA5).all())


@pytest.mark.parametrize("n_points,n_dur,n_per,steps", [
    (300, 1, 12, (310, 440)),      # epoch slices
    (2000, 1, 12, (2010, 2600)),   # whole tiles
    (20, 4, 4900, (29, 60)),       # several durations per tile
])
def test_null_sum_is_never_a_maximum(n_points, n_dur, n_per, steps):
    """A template whose ends are so small that their squares underflow (m = 1e-23): a window that
    meets the data with such a sample alone has B = 0 and A not 0, and a phase with only such
    windows is null. Periods longer than the curve make it a phase of its own. The winners are
    those of the 64-bit search, in which the end samples weigh nothing."""
    from _parity import compare_periodic
    from synth.lightcurves import custom
    c = 120.0 / 86400.0
    periods = np.linspace(steps[0], steps[1], n_per) * c
    w = custom(seed=n_points, n_points=n_points, cadence_s=120.0,
               planets=[dict(P=1e3, t0=0.5 * n_points * c, D=9.0 * c, depth=2e-2)])
    d = np.array([2.0, 4.0, 6.0, 8.0])[4 - n_dur:] * c
    tmpl = np.ones(1024, np.float32)
    tmpl[0] = tmpl[-1] = 1e-23
    args = (w.time, w.flux, w.flux_err, d, tmpl, periods)
    kw = dict(cadence=c, t0_step=c)
    g, o = gpu_search(*args, **kw), oracle_search(*args, **kw)
    assert np.isnan(g["dlogl"][-1, -1]) and np.isfinite(o["dlogl"][-1, -1])  # B = 0, A not 0
    compare_periodic(g, o, periods)


@pytest.mark.parametrize("n_dur,precision", [(33, "fp32"), (64, "fp32"), (64, "kahan")])
def test_packed_rows_beyond_a_warp(n_dur, precision):
    """Strips of 33 to 64 duration rows (periods of 13 to 26 t0 steps in a launch large enough to
    keep the durations together), so that lanes of the producer warp copy two rows each.
    Tolerances are the parity tests' (compare_periodic)."""
    from _parity import compare_periodic
    from synth.lightcurves import custom
    step = 1800.0 / 86400.0
    periods = np.exp(np.linspace(np.log(12.6 * step), np.log(26.0 * step), 4900))
    w = custom(seed=n_dur, n_points=700, cadence_s=1800.0,
               durations_h=np.linspace(0.6, 6.0, n_dur), periods=periods,
               planets=[dict(P=0.4, t0=0.1, D=0.1, depth=3e-3)])
    args = (w.time, w.flux, w.flux_err, w.durations, w.template, periods)
    kw = dict(cadence=w.cadence, t0_step=w.t0_step)
    compare_periodic(gpu_search(*args, precision=precision, **kw), oracle_search(*args, **kw),
                     periods)


@pytest.mark.parametrize("n_points,n_dur,n_per,steps,gap", [
    (900, 1, 24, (40, 440), 0),      # epoch slices
    (2600, 3, 24, (450, 2700), 700),  # whole tiles
    (700, 12, 4900, (13, 60), 200),  # several durations per tile
    (20, 12, 4900, (13, 60), 0),     # the same, phases without data
])
def test_first_of_zeros(n_points, n_dur, n_per, steps, gap):
    """A curve without any signal has LR 0 at every window with data: the winner is the first of
    them in (duration, phase) order, also where the first phases hold none, with a mask, and for
    a curve of a batch."""
    from paper_2503_20875_gb300 import Batch, Context
    from synth.lightcurves import custom
    c = 120.0 / 86400.0
    periods = np.exp(np.linspace(np.log(steps[0] * c), np.log(steps[1] * c), n_per))
    w = custom(seed=n_points, n_points=n_points, cadence_s=120.0, gaps=[(3 * c, (3 + gap) * c)],
               durations_h=np.linspace(0.1, 0.4, n_dur), periods=periods)
    w.flux[:] = 1.0
    args = (w.time, w.flux, w.flux_err, w.durations, w.template, periods)
    kw = dict(cadence=c, t0_step=c)
    mask = (np.random.default_rng(n_dur).uniform(size=(n_per, n_dur)) < 0.5).astype(np.uint8)
    for m in (None, mask):
        g, o = gpu_search(*args, mask=m, **kw), oracle_search(*args, mask=m, **kw)
        for key in ("dlogl", "i", "j"):
            np.testing.assert_array_equal(g["periodic"][key], o["periodic"][key])
    b = Batch(Context(0), [(w.time, w.flux, w.flux_err)] * 2, w.durations, w.template,
              periods[0], periods[-1], periods[1] / periods[0], cadence=c, t0_step=c)
    best = b.run()
    o = oracle_search(*args, **kw)["periodic"]
    first = int(np.flatnonzero(~np.isnan(o["dlogl"]))[0])
    for x in range(2):
        assert (best["k"][x], best["i"][x], best["j"][x], best["dlogl"][x]) == (
            first, o["i"][first], o["j"][first], 0.0)


@pytest.mark.parametrize("precision", ["fp32", "kahan"])
def test_a_flat_curve_is_no_slower(precision):
    """Windows without any signal are no candidates for a period's maximum: the search of a flat
    curve may not take longer than a noisy one's (1.2 x, for the timer's sake; least of ten)."""
    import torch
    import synth
    from paper_2503_20875_gb300 import Context, DeviceSearch, Plan
    from synth.lightcurves import custom
    w = custom(seed=4, n_points=60000, cadence_s=20.0, durations_h=np.linspace(0.5, 12.0, 20))
    periods = synth.log_grid(0.5, 6.5, 6000)
    ctx = Context(0)
    plan = Plan(ctx, w.time, w.flux, w.flux_err, w.durations, w.template, cadence=w.cadence,
                t0_step=w.t0_step, precision=precision)
    ds = DeviceSearch(ctx, plan, periods)
    t, f, e = (torch.from_numpy(np.ascontiguousarray(x)).cuda()
               for x in (w.time, w.flux, w.flux_err))
    took = {}
    for name, flux in (("noisy", f), ("flat", torch.ones_like(f))):
        ms = []
        for _ in range(13):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            ds.run(t, flux, e)
            b.record()
            torch.cuda.synchronize()
            ms.append(a.elapsed_time(b))
        took[name] = min(ms[3:])
    assert took["flat"] <= 1.2 * took["noisy"], took


@pytest.mark.parametrize("n_points,n_dur,n_per,steps", [
    (900, 1, 24, (40, 440)),      # epoch slices
    (2600, 3, 24, (450, 2700)),   # whole tiles
    (700, 12, 4900, (13, 60)),    # several durations per tile
])
@pytest.mark.parametrize("flat", [False, True])
@pytest.mark.parametrize("power", [40, 48])
def test_winners_do_not_depend_on_the_errors_unit(n_points, n_dur, n_per, steps, flat, power):
    """Flux errors 2^40 and 2^48 times as large scale every window's (A, B) by a power of two, and
    LR with it: the same winners, their LR scaled exactly, although A^2 falls below the smallest
    float. Flat: all windows but those that hold one point have LR 0."""
    from paper_2503_20875_gb300 import Batch, Context
    from synth.lightcurves import custom
    c = 120.0 / 86400.0
    periods = np.exp(np.linspace(np.log(steps[0] * c), np.log(steps[1] * c), n_per))
    w = custom(seed=power + n_points, n_points=n_points, cadence_s=120.0, sigma_spread=0.3,
               durations_h=np.linspace(0.1, 0.4, n_dur), periods=periods)
    if flat:
        w.flux[:] = 1.0
        w.flux[2 * n_points // 3] = np.float32(0.999)
    scale = np.float32(2.0 ** power)
    out = []
    for err in (w.flux_err, w.flux_err * scale):
        g = gpu_search(w.time, w.flux, err, w.durations, w.template, periods, cadence=c,
                       t0_step=c)["periodic"]
        b = Batch(Context(0), [(w.time, w.flux, err)], w.durations, w.template, periods[0],
                  periods[-1], periods[1] / periods[0], cadence=c, t0_step=c).run()
        out.append((g, b))
    (g0, b0), (g1, b1) = out
    for key in ("i", "j"):
        np.testing.assert_array_equal(g1[key], g0[key])
        np.testing.assert_array_equal(b1[key], b0[key])
    np.testing.assert_array_equal(g1["dlogl"] * 4.0 ** power, g0["dlogl"])
    np.testing.assert_array_equal(b1["dlogl"] * 4.0 ** power, b0["dlogl"])
    np.testing.assert_array_equal(b1["k"], b0["k"])
