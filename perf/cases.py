"""What is timed when this framework's speed is compared between two versions.

Each case is one call (or the short sequence of calls) that a program built on
the library makes for one window, one batch or one step, through the public
entry points of ``paper_2603_08386_gb300.ddhf``. The sizes are those of the
repository's own configurations, benchmark and tests (48x40 and 320x240 test
scenes, 640x360 and 640x480 sensors, the 1280x720 sensor; 100, 333, 750, 2000
and 10,000 bins), and ``draw`` spreads over the ranges between them.

Events are drawn on the GPU with the distributions of ``synth``: heavy-tailed
(Pareto 1.5) per-pixel counts with 30 % of the events bunched in time, drones
whose rotor pixels see periodic bursts, or the lognormal edge texture of the
ego-motion scenes; a share of events that do not belong to the window where
that is stated. ``exact`` evaluates the same definitions in FP64 with torch.
"""
import math

import numpy as np
import torch

from paper_2603_08386_gb300 import ddhf, synth

CAP = 4096   # boxes a caller makes room for
D9 = 1_000_000_000

# Table 2's comb (and thresholds) unless a case says otherwise
COMB = dict(M=4, d=3, h_min=4)


def listed():
    return [
        # the smallest call: a region of interest around one drone, 100 bins
        dict(name="detect_48x40", kind="detect", W=48, H=40, window_us=20_000, mean=9.9,
             bins=100, step_mhz=10_000),
        # an odd region with another comb, a 0/1 polarity sensor and packets
        # that overlap the window's edges; 333 bins
        dict(name="detect_347x261_odd", kind="detect", W=347, H=261, window_us=25_000, mean=6.3,
             bins=333, step_mhz=5_000, M=6, d=2, h_min=3, pol01=True, outside=0.05),
        # a sparse full-sensor window replayed as a graph: the latency that a
        # live detector sees most of the time
        dict(name="detect_hd_sparse", kind="detect", W=1280, H=720, window_us=30_000, mean=1.0,
             bins=750, step_mhz=2_000, graph=True),
        # a dense full-sensor window (about 20 million events), default tuning
        dict(name="detect_hd", kind="detect", W=1280, H=720, window_us=30_000, mean=21.7,
             bins=750, step_mhz=2_000),
        # throughput: consecutive dense windows in one graph, with the tuning
        # that the autotuner picks there (overlapped windows, hybrid spectra)
        dict(name="batch_hd", kind="batch", W=1280, H=720, window_us=30_000, mean=21.7,
             bins=750, step_mhz=2_000, windows=4, overlap=1, hybrid_min=128, wpb=8),
        # events that arrive in pinned host memory, results back on the host
        dict(name="host_320x240", kind="host", W=320, H=240, window_us=30_000, mean=21.7,
             bins=750, step_mhz=2_000, windows=8),
        # spectra alone on the edge-texture scene: binning and 2000 bins per pixel
        dict(name="spectra_640x480", kind="spectra", W=640, H=480, window_us=50_000, mean=17.0,
             bins=2000, step_mhz=1_000, scene="texture"),
        # spectra alone on the finest grid: 10,000 bins, 200 ms, timestamps near 2^40 us
        dict(name="spectra_fine_320x180", kind="spectra", W=320, H=180, window_us=200_000,
             mean=65.0, bins=10_000, step_mhz=500, t0=(1 << 40) - 200_000),
        # scoring alone: given spectra, 750 bins
        dict(name="scores_640x360", kind="scores", W=640, H=360, bins=750, step_mhz=2_000),
        # scoring alone on the 2000-bin grid
        dict(name="scores_2000_320x240", kind="scores", W=320, H=240, bins=2000, step_mhz=1_000),
        # the differentiable soft comb, forward and backward, on one ego-motion window
        dict(name="softcomb_640x480", kind="softcomb", W=640, H=480, window_us=40_000, mean=16.0,
             bins=750, step_mhz=2_000, scene="texture", harmonics=6, Q=3),
        # a sliding window: one push (the events of 3.75 ms in, as many out) and a detection
        dict(name="slide_640x360", kind="slide", W=640, H=360, window_us=30_000, mean=21.7,
             bins=750, step_mhz=2_000, hops=8),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _sensor(rng, lo, hi):
    """A W x H of about lo..hi pixels (log-uniform), odd sizes among them."""
    px = _log(rng, lo, hi)
    aspect = rng.uniform(1.0, 1.9)
    return max(8, round(math.sqrt(px * aspect))), max(8, round(math.sqrt(px / aspect)))


def draw(rng):
    kind = rng.choice(["detect", "detect", "detect", "batch", "host", "spectra", "spectra",
                       "scores", "scores", "softcomb", "slide"])
    if kind == "detect":
        W, H = _sensor(rng, 1_500, 900_000)
        c = dict(kind=kind, W=W, H=H, window_us=rng.randint(15_000, 40_000),
                 mean=round(_log(rng, 1.0, 21.0), 2), graph=rng.random() < 0.5)
        c.update(rng.choice([dict(bins=100, step_mhz=10_000), dict(bins=750, step_mhz=2_000),
                             dict(bins=rng.randint(40, 1000), step_mhz=2_000),
                             dict(bins=333, step_mhz=5_000, M=6, d=2, h_min=3)]))
        if rng.random() < 0.3:
            c.update(pol01=True, outside=0.05)
        return c
    if kind == "batch":
        W, H = _sensor(rng, 20_000, 900_000)
        return dict(kind=kind, W=W, H=H, window_us=30_000, mean=round(rng.uniform(2, 20), 2),
                    bins=750, step_mhz=2_000, windows=rng.randint(2, 4),
                    overlap=rng.randint(0, 1), hybrid_min=rng.choice([0, 64, 128]),
                    wpb=rng.choice([4, 8]))
    if kind == "host":
        W, H = _sensor(rng, 10_000, 77_000)
        return dict(kind=kind, W=W, H=H, window_us=30_000, mean=round(_log(rng, 2, 20), 2),
                    bins=750, step_mhz=2_000, windows=rng.randint(2, 8))
    if kind == "spectra":
        W, H = _sensor(rng, 2_000, 300_000)
        bins, step = rng.choice([(100, 10_000), (750, 2_000), (rng.randint(30, 2_000), 1_000),
                                 (2_000, 1_000)])
        if W * H < 58_000 and rng.random() < 0.3:
            bins, step = rng.randint(4_000, 10_000), 500
        return dict(kind=kind, W=W, H=H, window_us=rng.randint(20_000, 200_000),
                    mean=round(_log(rng, 2, 40), 2), bins=bins, step_mhz=step,
                    scene=rng.choice(["noise", "texture"]),
                    t0=rng.choice([0, rng.randint(0, 1 << 40)]))
    if kind == "scores":
        W, H = _sensor(rng, 1_500, 230_000)
        c = dict(kind=kind, W=W, H=H, bins=rng.choice([100, 750, rng.randint(200, 1_000)]),
                 step_mhz=2_000)
        if W * H < 77_000 and rng.random() < 0.4:
            c["bins"] = rng.randint(1_025, 2_000)
        if rng.random() < 0.3:
            c.update(M=6, d=2, h_min=3)
        return c
    if kind == "softcomb":
        W, H = _sensor(rng, 2_000, 300_000)
        return dict(kind=kind, W=W, H=H, window_us=rng.randint(20_000, 40_000),
                    mean=round(_log(rng, 6, 16), 2), bins=750, step_mhz=2_000,
                    scene=rng.choice(["noise", "texture"]), harmonics=rng.randint(1, 8),
                    Q=rng.randint(1, 8))
    W, H = _sensor(rng, 10_000, 230_000)
    return dict(kind="slide", W=W, H=H, window_us=30_000, mean=round(_log(rng, 3, 21), 2),
                bins=rng.choice([750, rng.randint(300, 1_000)]), step_mhz=2_000,
                hops=rng.choice([4, 8, 16]))


# ------------------------------------------------------------------ inputs

def _gen(seed, salt):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 1009 + salt)


def _x_m(mean):
    """Scale of the Pareto(1.5) counts floor(x_m U^(-2/3)) with this mean (below a mean of
    one, the scale is proportional to the mean)."""
    return synth.pareto_x_m(mean) if mean >= 1.0 else mean * synth.pareto_x_m(1.0)


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _signs(g, n):
    return (torch.randint(0, 2, (n,), generator=g, device="cuda", dtype=torch.int8) * 2 - 1)


def _drone_events(case, seed, salt):
    """Rotor pixels of up to three drones (as the batched configuration places them) and
    their events over the window: numpy keys, times, polarities."""
    W, H = case["W"], case["H"]
    rng = np.random.default_rng([int(seed), salt, 7])
    sizes = (10, 300, 2000) if W * H >= 200_000 else (min(120, max(4, W * H // 16)),)
    parts = []
    for n_px, f0 in zip(sizes, (100.0, 200.0, 300.0) if len(sizes) == 3 else (150.0,)):
        cx = int(rng.integers(W // 8, max(W // 8 + 1, 7 * W // 8)))
        cy = int(rng.integers(H // 8, max(H // 8 + 1, 7 * H // 8)))
        for rk in synth.drone_keys(W, H, cx, cy, n_px):
            parts.append(synth.rotor_events(rng, rk, f0 * rng.uniform(0.995, 1.005), 0.0,
                                            float(case["window_us"]), per_edge=4))
    return [np.concatenate([p[i] for p in parts]) for i in range(3)]


def _events(case, seed, salt=0):
    """One window's events on the GPU, in time order: x, y int16, t int64 (absolute), p int8."""
    W, H, win = case["W"], case["H"], case["window_us"]
    npx = W * H
    g = _gen(seed, salt)
    if case.get("scene") == "texture":
        # lognormal counts (median set by the mean), bursts at one to three crossing instants
        mu = math.log(case["mean"]) - 1.16 ** 2 / 2
        z = torch.randn(npx, generator=g, device="cuda", dtype=torch.float64)
        counts = torch.exp(mu + 1.16 * z).floor().clamp_(max=2000).long()
        keys = torch.repeat_interleave(torch.arange(npx, device="cuda"), counts)
        n = keys.numel()
        cross = 1 + torch.randint(0, 3, (npx,), generator=g, device="cuda")
        which = (_rand(g, n) * cross[keys]).long()
        inst = _rand(g, npx, 3) * win
        t = inst[keys, which]
        t += -torch.log1p(-_rand(g, n)) * 250.0 * _signs(g, n)
        pol = _signs(g, npx * 3).view(npx, 3)[keys, which]
        pol = torch.where(_rand(g, n) < 0.1, -pol, pol)
        keep = (t >= 0) & (t < win)
        keys, t, pol = keys[keep], t[keep].round_(), pol[keep]
    else:
        u = _rand(g, npx).clamp_(min=1e-300)
        counts = (_x_m(case["mean"]) * u.pow_(-1.0 / 1.5)).floor_().clamp_(max=20_000).long()
        dk, dt, dp = _drone_events(case, seed, salt)
        counts[torch.from_numpy(np.unique(dk)).cuda()] = 0
        keys = torch.repeat_interleave(torch.arange(npx, device="cuda"), counts)
        n = keys.numel()
        t = (_rand(g, n) * win).floor_()
        centre = _rand(g, npx) * win
        near = centre[keys] + 300.0 * torch.randn(n, generator=g, device="cuda",
                                                  dtype=torch.float64)
        t = torch.where(_rand(g, n) < 0.3, near.round_(), t)
        pol = _signs(g, n)
        keys = torch.cat([keys, torch.from_numpy(dk).cuda()])
        t = torch.cat([t, torch.from_numpy(dt).cuda().round_()])
        pol = torch.cat([pol, torch.from_numpy(dp).cuda()])
    t = t.long().clamp_(0, win - 1)
    if case.get("outside"):
        # packets that begin before the window or end after it
        m = max(1, int(case["outside"] * t.numel()))
        keys = torch.cat([keys, torch.randint(0, npx, (m,), generator=g, device="cuda")])
        early = torch.randint(-win // 10, 0, (m,), generator=g, device="cuda")
        late = torch.randint(win, win + win // 10, (m,), generator=g, device="cuda")
        t = torch.cat([t, torch.where(_rand(g, m) < 0.5, early, late)])
        pol = torch.cat([pol, _signs(g, m)])
    order = torch.argsort(t, stable=True)
    keys, t, pol = keys[order], t[order], pol[order]
    if case.get("pol01"):
        pol = (pol + 1) // 2
    y = torch.div(keys, W, rounding_mode="floor")
    return ((keys - y * W).to(torch.int16), y.to(torch.int16), t + int(case.get("t0", 0)),
            pol.to(torch.int8))


def _params(case):
    over = {k: case.get(k, v) for k, v in COMB.items()}
    return ddhf.default_params(polarity_01=int(bool(case.get("pol01"))), **over)


def _grid(case):
    return ddhf.make_grid(0, case["step_mhz"], D9, case["bins"])


def _spectra_rows(case, seed):
    """Power spectra for scoring, [pixels, bins]: random-phase spectra (exponential powers,
    scaled by the pixel's event count), a tenth of them with a harmonic comb on top."""
    g = _gen(seed, 3)
    npx, N = case["W"] * case["H"], case["bins"]
    P = torch.empty(npx, N, device="cuda").exponential_(1.0, generator=g)
    P *= (5.0 * (1 - _rand(g, npx)).pow_(-2.0 / 3.0)).float()[:, None]
    rows = torch.nonzero(_rand(g, npx) < 0.1).flatten()
    w = torch.randint(8, max(9, N // 5), (rows.numel(),), generator=g, device="cuda")
    for m in range(1, 5):
        amp = 2.0 + 38.0 * torch.rand(rows.numel(), generator=g, device="cuda")
        P[rows, (m * w).clamp_(max=N - 1)] *= 1.0 + amp
    return P


class _State:
    pass


def _zeros(n, dtype):
    return torch.zeros(n, dtype=dtype, device="cuda")


def _outputs(s, npx, windows=1):
    s.boxes = torch.zeros((windows * CAP, 5), dtype=torch.int32, device="cuda")
    s.nbox = _zeros(windows, torch.int32)
    s.mask = torch.zeros((windows, npx), dtype=torch.uint8, device="cuda")
    s.log_sf, s.snr = _zeros(npx, torch.float32), _zeros(npx, torch.float32)
    s.box_f0, s.box_snr, s.box_hz = (_zeros(CAP, torch.int32), _zeros(CAP, torch.float32),
                                     _zeros(CAP, torch.float32))


def prepare(case, seed):
    s = _State()
    s.case, s.kind = case, case["kind"]
    W, H = case["W"], case["H"]
    npx = W * H
    params, grid = _params(case), _grid(case)
    if s.kind in ("detect", "batch", "host"):
        nw = case.get("windows", 1)
        win = case["window_us"]
        t0 = int(case.get("t0", 0))
        s.ev = [_events(case, seed, 100 + w) for w in range(nw)]
        s.ctx = ddhf.Context(W, H, grid, params, max_events=max(e[0].numel() for e in s.ev),
                             max_windows=nw)
        if s.kind == "batch":
            s.ctx.set_tuning(overlap=case["overlap"], hybrid_min=case["hybrid_min"],
                             warps_per_block=case["wpb"])
        if s.kind == "host":
            s.ev = [tuple(a.cpu().pin_memory() for a in e) for e in s.ev]
            s.boxes = torch.zeros((nw * CAP, 5), dtype=torch.int32).pin_memory()
            s.nbox = torch.zeros(nw, dtype=torch.int32).pin_memory()
            s.mask = torch.zeros((nw, npx), dtype=torch.uint8).pin_memory()
        else:
            _outputs(s, npx, nw)
        s.windows = [(*e, e[0].numel(), t0, win) for e in s.ev]
    elif s.kind == "spectra":
        s.ev = _events(case, seed)
        s.ctx = ddhf.Context(W, H, grid, params, max_events=s.ev[0].numel())
        # room for every pixel; rows from the active count on stay zero
        s.P = torch.zeros((npx, case["bins"]), device="cuda")
    elif s.kind == "scores":
        # one event per pixel, so that every pixel is listed and row a is pixel a
        params.n_min = 1
        s.ctx = ddhf.Context(W, H, grid, params, max_events=npx)
        k = torch.arange(npx, device="cuda")
        s.ctx.bin_events((k % W).to(torch.int16), (k // W).to(torch.int16), torch.zeros_like(k),
                         torch.ones(npx, dtype=torch.int8, device="cuda"), 0, 1000)
        s.P = _spectra_rows(case, seed)
        s.log_sf, s.snr = _zeros(npx, torch.float32), _zeros(npx, torch.float32)
        s.f0, s.mask = _zeros(npx, torch.int32), _zeros(npx, torch.uint8)
    elif s.kind == "softcomb":
        s.ev = _events(case, seed)
        s.ctx = ddhf.Context(W, H, grid, params, max_events=s.ev[0].numel())
        s.ctx.bin_events(*s.ev, 0, case["window_us"])
        act = s.ctx.csr()["active"].clone()
        s.pixels = act[_soft_pick(case, seed, act.numel())].contiguous()
        s.f0, s.w, s.sigma, s.B, s.gS = _soft_inputs(case, seed)
        for v in (s.f0, s.w, s.sigma):
            v.requires_grad_(True)
    elif s.kind == "slide":
        T, hops = case["window_us"], case["hops"]
        x, y, t, p = _events(case, seed)
        edge = [T * i // hops for i in range(hops + 1)]
        at = torch.searchsorted(t, torch.tensor(edge, device="cuda")).tolist()
        s.hop = [(x[a:b].clone(), y[a:b].clone(), t[a:b].clone(), p[a:b].clone())
                 for a, b in zip(at, at[1:])]
        most = max(b - a for a, b in zip(at, at[1:]))
        s.edge, s.k = edge, 0
        s.ctx = ddhf.Context(W, H, grid, params, max_events=t.numel() + 2 * most + 1)
        s.ctx.slide_begin(T, 0, rebuild_every=64)
        for _ in range(hops):
            _push(s)
        _outputs(s, npx)
    else:
        raise ValueError(s.kind)
    return s


def _soft_pick(case, seed, n_active):
    """Which active pixels are scored: half as many as the sensor has pixels, in order."""
    n = case["W"] * case["H"] // 2
    pick = torch.randperm(max(n, n_active), generator=_gen(seed, 4), device="cuda")[:n]
    return (pick % max(n_active, 1)).sort().values


def _soft_inputs(case, seed):
    g = _gen(seed, 5)
    n, nh = case["W"] * case["H"] // 2, case["harmonics"]
    f0 = 50.0 + 150.0 * torch.rand(n, generator=g, device="cuda")
    w = 0.5 + torch.rand(nh, generator=g, device="cuda")
    sigma = 1.5 + torch.rand(nh, generator=g, device="cuda")
    B = 2.0 + 20.0 * torch.rand(n, generator=g, device="cuda")
    gS = torch.rand(n, generator=g, device="cuda")
    return f0, w, sigma, B, gS


# ------------------------------------------------------------------ one pass

def _push(s):
    """The next hop of the stream: the window's pattern repeats every window_us, so its
    sensor times are offset to absolute ones."""
    hops = len(s.hop)
    x, y, t, p = s.hop[s.k % hops]
    base = (s.k // hops) * s.case["window_us"]
    ddhf.ddhf_slide_push(s.ctx.h, x, y, t + base, p, x.numel(), base + s.edge[s.k % hops + 1])
    s.k += 1


def run(s):
    h = s.ctx.h
    if s.kind == "detect":
        if s.case.get("graph"):
            ddhf.ddhf_detect_batch(h, s.windows, s.boxes, CAP, s.nbox, s.mask, use_graph=True)
        else:
            ddhf.ddhf_detect(h, *s.windows[0], s.boxes, CAP, s.nbox, s.mask)
        ddhf.ddhf_box_frequencies(h, 0, s.boxes, s.nbox, CAP, s.box_f0, s.box_snr, s.box_hz)
        ddhf.ddhf_export_scores(h, 0, None, s.log_sf, s.snr, None, None)
        return [s.boxes, s.nbox, s.mask, s.box_f0, s.box_snr, s.box_hz, s.log_sf, s.snr]
    if s.kind == "batch":
        ddhf.ddhf_detect_batch(h, s.windows, s.boxes, CAP, s.nbox, s.mask, use_graph=True)
        ddhf.ddhf_export_scores(h, len(s.windows) - 1, None, s.log_sf, s.snr, None, None)
        return [s.boxes, s.nbox, s.mask, s.log_sf, s.snr]
    if s.kind == "host":
        ddhf.ddhf_detect_batch_host(h, s.windows, s.boxes, CAP, s.nbox, s.mask)
        return [s.boxes, s.nbox, s.mask]
    if s.kind == "spectra":
        s.ctx.bin_events(*s.ev, int(s.case.get("t0", 0)), s.case["window_us"])
        ddhf.ddhf_power_spectrum(h, ddhf.FORM["blocked"], s.P, s.P.shape[0])
        return [s.P]
    if s.kind == "scores":
        ddhf.ddhf_comb_score(h, s.P, s.P.shape[0], s.log_sf, s.snr, s.f0, s.mask)
        return [s.log_sf, s.snr, s.f0, s.mask]
    if s.kind == "softcomb":
        S = ddhf.SoftComb.apply(s.f0, s.w, s.sigma, h, s.pixels, s.B, s.case["Q"], 2.0,
                                s.case["window_us"] / 2)
        return [S.detach(), *torch.autograd.grad(S, (s.f0, s.w, s.sigma), s.gS)]
    _push(s)
    ddhf.ddhf_slide_detect(h, s.boxes, CAP, s.nbox, s.mask)
    ddhf.ddhf_export_scores(h, 0, None, s.log_sf, s.snr, None, None)
    return [s.boxes, s.nbox, s.mask, s.log_sf, s.snr]


# ------------------------------------------------------------------ work

def _expected(case, n_min=6):
    """Expected active pixels and their events, per window."""
    npx = case["W"] * case["H"]
    if case.get("scene") == "texture":
        mu, sg = math.log(case["mean"]) - 1.16 ** 2 / 2, 1.16
        z = (math.log(n_min) - mu) / sg
        share = 0.5 * math.erfc(z / math.sqrt(2))
        return npx * share, npx * case["mean"] * 0.5 * math.erfc((z - sg) / math.sqrt(2))
    xm = _x_m(case["mean"])
    c = np.arange(n_min, 20_001, dtype=np.float64)
    p = np.minimum(1.0, (xm / c) ** 1.5)
    return npx * float(p[0]), npx * float(n_min * p[0] + p[1:].sum())


def work(case):
    """Bytes: events (13 B each) and inputs once, outputs once. Operations: two multiply-adds
    per event and bin (the cosine and the sine sum of Eq. 6); the scores a few per bin."""
    npx, N = case["W"] * case["H"], case.get("bins", 0)
    k = case["kind"]
    if k == "scores":
        return dict(bytes=npx * (4 * N + 13), flops=npx * N * 10)
    act, ev = _expected(case)
    raw = 13 * npx * case["mean"] * (1 + case.get("outside", 0))
    if k in ("detect", "batch", "host"):
        nw = case.get("windows", 1)
        return dict(bytes=nw * (raw + npx) + (0 if k == "host" else 16 * act),
                    flops=nw * (4 * ev * N + 10 * act * N))
    if k == "spectra":
        return dict(bytes=raw + 4 * act * N, flops=4 * ev * N)
    if k == "softcomb":
        n = npx // 2
        terms = n * ev / act * case["harmonics"] * (2 * case["Q"] + 1)
        return dict(bytes=2 * 4 * n * ev / act + 6 * 4 * n, flops=(4 + 8) * terms)
    # slide: the hop's events in, as many out; the touched pixels' sums read and written
    hop = ev / case["hops"]
    touched = npx * (1 - math.exp(-2 * case["mean"] / case["hops"]))
    return dict(bytes=raw / case["hops"] * 2 + touched * N * 16 + act * N * 8 + npx + 8 * act,
                flops=2 * 4 * hop * N + 10 * act * N)


# ------------------------------------------------------------------ 64 bits

def _csr(case, ev, t_lo, t_hi):
    """Kept events of [t_lo, t_hi) grouped by pixel (input order inside a pixel): keys of the
    active pixels, their first event and count, and the grouped tau and sign (FP64)."""
    x, y, t, p = ev
    keep = (t >= t_lo) & (t < t_hi)
    key = (y.long() * case["W"] + x.long())[keep]
    order = torch.argsort(key, stable=True)
    tau = (t[keep] - t_lo)[order]
    sgn = p[keep][order].double()
    if case.get("pol01"):
        sgn = 2 * sgn - 1
    cnt = torch.bincount(key, minlength=case["W"] * case["H"])
    first = torch.cumsum(cnt, 0) - cnt
    act = torch.nonzero(cnt >= 6).flatten()
    return act, first[act], cnt[act], tau, sgn


def _power64(case, first, cnt, tau, sgn, sink, room=1 << 27):
    """Eq. 6 in FP64, a few pixels of similar count at a time: sink(rows, P[rows, bins])."""
    N, da = case["bins"], case["step_mhz"]
    nb = (N + 31) // 32
    ja = torch.arange(nb, device="cuda") * (32 * da)
    jr = torch.arange(32, device="cuda") * da
    by_count = torch.argsort(cnt)
    sizes = cnt[by_count].tolist()
    i = 0
    while i < len(sizes):
        j = i + 1
        top = max(32, int(1.25 * sizes[i]))
        most = max(1, room // (max(N, top * (nb + 32)) * 4))
        j = min(len(sizes), i + most)
        hi = int(np.searchsorted(np.asarray(sizes[i:j]), top, side="right"))
        j = i + max(1, hi)
        rows = by_count[i:j]
        c = int(sizes[j - 1])
        at = torch.arange(c, device="cuda")[None, :]
        ok = at < cnt[rows][:, None]
        idx = torch.where(ok, first[rows][:, None] + at, torch.zeros_like(at))
        tt = tau[idx]
        s = torch.where(ok, sgn[idx], torch.zeros((), dtype=torch.float64, device="cuda"))

        def phasor(a):  # e^{-2 pi i a tau / D}, exact residues
            r = ((a % D9) * (tt[..., None] % D9)) % D9
            ph = r.double() * (-2.0 * math.pi / D9)
            return torch.complex(torch.cos(ph), torch.sin(ph))

        A = phasor(ja) * s[..., None]
        F = torch.bmm(A.transpose(1, 2), phasor(jr)).reshape(rows.numel(), nb * 32)[:, :N]
        sink(rows, F.real ** 2 + F.imag ** 2)
        i = j


def _scores64(P, case):
    """Eq. 7-10 in FP64 on rows of P: ln SF and, where SF <= tau_sf, the best SNR (else 0)."""
    N = P.shape[1]
    M, d, h_min = (case.get(k, v) for k, v in COMB.items())
    lsf = P.clamp(min=1e-30).log().mean(1) - P.mean(1).log()
    srt, order = P.sort(dim=1)
    rank = torch.empty_like(order)
    rank.scatter_(1, order, torch.arange(N, device="cuda").expand_as(order))
    wmax = torch.nn.functional.max_pool1d(P[:, None], 2 * d + 1, 1)[:, 0]  # centre c at c - d
    best = torch.zeros(P.shape[0], dtype=torch.float64, device="cuda")
    for w in range(max(1, d), N):
        mv = min(M, (N - 1 - d) // w)
        if mv < h_min:
            break
        H = sorted({m * w + q for m in range(1, mv + 1) for q in range(-d, d + 1)})
        c = N - len(H)
        if c <= 0:
            continue
        nw = wmax[:, [m * w - d for m in range(1, mv + 1)]].mean(1)
        gone = rank[:, H].sort(dim=1).values
        pos = [torch.full_like(gone[:, 0], (c - 1) // 2), torch.full_like(gone[:, 0], c // 2)]
        for q in range(len(H)):
            for k in (0, 1):
                pos[k] += (gone[:, q] <= pos[k]).long()
        B = 0.5 * (srt.gather(1, pos[0][:, None]) + srt.gather(1, pos[1][:, None]))[:, 0]
        snr = torch.where(B > 0, nw / B, torch.where(nw > 0, math.inf, 0.0))
        best = torch.maximum(best, snr)
    return lsf, torch.where(lsf <= math.log(float(np.float32(0.89))), best, 0.0)


# FP64 scoring ranks every bin per candidate: up to this many (row, candidate) pairs
SCORED = 12_000_000


def _window64(case, ev, t_lo, t_hi, npx):
    act, first, cnt, tau, sgn = _csr(case, ev, t_lo, t_hi)
    lsf = torch.zeros(npx, dtype=torch.float64, device="cuda")
    cand = case["bins"] // case.get("h_min", COMB["h_min"])
    want_snr = act.numel() * cand <= SCORED
    snr = torch.zeros(npx, dtype=torch.float64, device="cuda") if want_snr else None

    def sink(rows, P):
        if want_snr:
            lsf[rows], snr[rows] = _scores64(P, case)
        else:
            lsf[rows] = P.clamp(min=1e-30).log().mean(1) - P.mean(1).log()

    _power64(case, first, cnt, tau, sgn, sink)
    return lsf, snr


def exact(case, seed):
    k = case["kind"]
    npx = case["W"] * case["H"]
    t0 = int(case.get("t0", 0))
    if k in ("detect", "batch"):
        if k == "batch":
            ev = _events(case, seed, 100 + case["windows"] - 1)
            return [None, None, None, *_window64(case, ev, t0, t0 + case["window_us"], npx)]
        ev = _events(case, seed, 100)
        return [None] * 6 + list(_window64(case, ev, t0, t0 + case["window_us"], npx))
    if k == "host":
        return None  # boxes, counts and masks: no computed numbers
    if k == "spectra":
        ev = _events(case, seed)
        act, first, cnt, tau, sgn = _csr(case, ev, t0, t0 + case["window_us"])
        P = torch.zeros((npx, case["bins"]), dtype=torch.float64, device="cuda")

        def sink(rows, p):
            P[rows] = p

        _power64(case, first, cnt, tau, sgn, sink)
        return [P]
    if k == "scores":
        P = _spectra_rows(case, seed)
        cand = case["bins"] // case.get("h_min", COMB["h_min"])
        step = max(1, (1 << 25) // case["bins"])
        parts = [P[i:i + step].double() for i in range(0, npx, step)]
        if npx * cand > 3 * SCORED:
            return [torch.cat([p.clamp(min=1e-30).log().mean(1) - p.mean(1).log()
                               for p in parts]), None, None, None]
        both = [_scores64(p, case) for p in parts]
        return [torch.cat([b[0] for b in both]), torch.cat([b[1] for b in both]), None, None]
    if k == "softcomb":
        return _soft64(case, seed)
    # slide: the window after the first timed push holds one whole period of the pattern
    x, y, t, p = _events(case, seed)
    T, first_edge = case["window_us"], case["window_us"] // case["hops"]
    t = torch.where(t < first_edge, t + T, t)
    return [None, None, None,
            *_window64(case, (x, y, t, p), first_edge, first_edge + T, npx)]


def _soft64(case, seed):
    act, first, cnt, tau, sgn = _csr(case, _events(case, seed), 0, case["window_us"])
    pick = _soft_pick(case, seed, act.numel())
    first, cnt = first[pick], cnt[pick]
    n, nh, Q, delta = pick.numel(), case["harmonics"], case["Q"], 2.0
    f0, w, sigma, B, gS = (v.double() for v in _soft_inputs(case, seed))
    f0 = (f0 * 1e6).round() * 1e-6
    px = torch.repeat_interleave(torch.arange(n, device="cuda"), cnt)
    # the scored pixels' events, in order
    idx = torch.repeat_interleave(first, cnt) + (
        torch.arange(px.numel(), device="cuda")
        - torch.repeat_interleave(torch.cumsum(cnt, 0) - cnt, cnt))
    tt = (tau[idx].double() - case["window_us"] / 2) * 1e-6
    s = sgn[idx]
    S = torch.zeros(n, dtype=torch.float64, device="cuda")
    gf = torch.zeros_like(S)
    gw, gsg = torch.zeros_like(w), torch.zeros_like(sigma)
    for h in range(1, nh + 1):
        Z = Ac = Ad = Cc = Ec = 0.0
        for q in range(-Q, Q + 1):
            ph = -2 * math.pi * torch.remainder((h * f0[px] + q * delta) * tt, 1.0)
            re, im = s * torch.cos(ph), s * torch.sin(ph)
            col = torch.zeros(n, 4, dtype=torch.float64, device="cuda")
            wt = 2 * math.pi * tt
            col.index_add_(0, px, torch.stack([re, im, wt * im, -wt * re], 1))
            P = col[:, 0] ** 2 + col[:, 1] ** 2
            Pd = 2 * (col[:, 0] * col[:, 2] + col[:, 1] * col[:, 3])
            qd = q * delta
            G = torch.exp(-qd * qd / (2 * sigma[h - 1] ** 2))
            Z, Ac, Ad = Z + G, Ac + G * P, Ad + G * Pd
            Cc, Ec = Cc + G * P * qd * qd, Ec + G * qd * qd
        S += w[h - 1] * Ac / Z / B
        gf += w[h - 1] * h * Ad / Z / B
        gw[h - 1] = (gS * Ac / Z / B).sum()
        gsg[h - 1] = (gS * w[h - 1] / (B * sigma[h - 1] ** 3) * (Cc / Z - Ac / Z * Ec / Z)).sum()
    return [S, gS * gf, gw, gsg]
