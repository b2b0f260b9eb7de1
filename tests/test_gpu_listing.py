"""ddhf_power_spectrum lists the long pixels of slot 0 itself: every row is
written, once, and right, whatever tuning the window was binned under and
whatever other windows a batched detection queued before."""
import numpy as np
import pytest
import torch

from paper_2603_08386_gb300 import build, ddhf, synth

pytestmark = pytest.mark.gpu

COUNTS = [3, 31, 32, 40, 63, 64, 100, 127, 128, 200, 255, 256, 300, 900, 1024, 1500, 2047, 2048,
          3000, 5000]


def _scene(seed, counts):
    rng = np.random.default_rng(seed)
    key = np.repeat(np.arange(len(counts)), counts)
    t = np.sort(rng.integers(0, 30_000, key.size)).astype(np.int64)
    key = rng.permutation(key)
    return synth.Scene(W=len(counts), H=1, t0=0, window_us=30_000, x=key.astype(np.int16),
                       y=np.zeros(key.size, np.int16), t=t,
                       p=rng.choice(np.array([-1, 1], np.int8), key.size),
                       grid=synth.hz_grid(0, 2, 750))


def _spectra(c, form, n):
    P = torch.full((n, 750), float("nan"), device="cuda")
    ddhf.ddhf_power_spectrum(c.h, ddhf.FORM[form], P, n)
    c.stats()
    return P


def _fresh(s, ev, form, **tuning):
    c = ddhf.Context(s.W, s.H, s.grid, ddhf.default_params(n_min=1), max_events=s.n)
    c.set_tuning(**tuning)
    c.bin_events(*ev, s.t0, s.window_us)
    P = _spectra(c, form, s.W)
    c.close()
    return P


@pytest.mark.parametrize("form", ["blocked", "hybrid"])
@pytest.mark.parametrize("binned,run", [(1024, 64), (64, 1024), (32, 4096), (4096, 32)])
def test_tuning_changed_after_binning(binned, run, form):
    build.build()
    s = _scene(1, COUNTS)
    ev = ddhf.events_to_device(s)
    c = ddhf.Context(s.W, s.H, s.grid, ddhf.default_params(n_min=1), max_events=s.n)
    c.set_tuning(heavy_min=binned)
    c.bin_events(*ev, s.t0, s.window_us)
    c.set_tuning(heavy_min=run)
    P = _spectra(c, form, s.W)
    c.close()
    assert torch.equal(P, _fresh(s, ev, form, heavy_min=run))


@pytest.mark.parametrize("fuse", [0, 1])
def test_spectra_of_slot_0_after_a_batch(fuse):
    build.build()
    scenes = [_scene(2, COUNTS), _scene(3, COUNTS[::-1])]
    dev = [ddhf.events_to_device(s) for s in scenes]
    s = scenes[0]
    c = ddhf.Context(s.W, s.H, s.grid, ddhf.default_params(n_min=1), max_events=s.n,
                     max_windows=2)
    c.set_tuning(fuse=fuse)
    wins = [(d[0], d[1], d[2], d[3], q.n, q.t0, q.window_us) for d, q in zip(dev, scenes)]
    boxes = torch.empty((2 * 8, 5), dtype=torch.int32, device="cuda")
    nb = torch.zeros(2, dtype=torch.int32, device="cuda")
    ddhf.ddhf_detect_batch(c.h, wins, boxes, 8, nb)
    P = _spectra(c, "blocked", s.W)
    c.close()
    assert torch.equal(P, _fresh(s, dev[0], "blocked"))


def _context(scenes, **tuning):
    c = ddhf.Context(scenes[0].W, scenes[0].H, scenes[0].grid, ddhf.default_params(n_min=1),
                     max_events=max(s.n for s in scenes), max_windows=2)
    c.set_tuning(**tuning)
    return c


def _batch(c, scenes, dev, graph=False):
    wins = [(d[0], d[1], d[2], d[3], q.n, q.t0, q.window_us) for d, q in zip(dev, scenes)]
    boxes = torch.empty((2 * 8, 5), dtype=torch.int32, device="cuda")
    nb = torch.zeros(2, dtype=torch.int32, device="cuda")
    ddhf.ddhf_detect_batch(c.h, wins, boxes, 8, nb, use_graph=graph)
    return boxes, nb


def test_list_follows_every_change():
    # one context through binnings, tunings, batches (with and without a graph) and
    # detections of one window, spectra after each
    build.build()
    a, b = _scene(4, COUNTS), _scene(5, COUNTS[::-1])
    da, db = ddhf.events_to_device(a), ddhf.events_to_device(b)
    want = {(k, hm): _fresh(s, d, "blocked", heavy_min=hm)
            for k, s, d in (("a", a, da), ("b", b, db)) for hm in (1024, 64)}
    c = _context([a, b], heavy_min=1024)
    keep, hm = [], 1024
    for step in ("bin a", "again", 64, "again", "batch ba", 1024, "bin a", "batch ba", "graph ab",
                 "again", "graph ab", "graph b", 64, "graph ba", "detect a", "bin b", 1024):
        if isinstance(step, int):
            c.set_tuning(heavy_min=step)
            hm = step
        elif step != "again":
            how, what = step.split()
            sc, dv = zip(*[(a, da) if k == "a" else (b, db) for k in what])
            if how == "bin":
                c.bin_events(*dv[0], sc[0].t0, sc[0].window_us)
            elif how == "detect":
                c.detect(*dv[0], sc[0].t0, sc[0].window_us)
            else:
                keep.append(_batch(c, sc, dv, graph=how == "graph"))
            slot0 = what[0]
        assert torch.equal(_spectra(c, "blocked", a.W), want[slot0, hm]), step
    c.close()


def test_captured_calls_and_their_replays():
    build.build()
    a, b = _scene(6, COUNTS), _scene(7, COUNTS[::-1])
    da, db = ddhf.events_to_device(a), ddhf.events_to_device(b)
    wa, wb = _fresh(a, da, "blocked"), _fresh(b, db, "blocked")
    c = _context([a, b])
    c.bin_events(*da, a.t0, a.window_us)
    _spectra(c, "blocked", a.W)
    keep = [_batch(c, [a, b], [da, db])]
    c.bin_events(*da, a.t0, a.window_us)
    # a captured spectrum call, replayed after other windows took the list
    P = torch.full((a.W, 750), float("nan"), device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ddhf.ddhf_power_spectrum(c.h, ddhf.FORM["blocked"], P, a.W)
    for scenes, dev, want in (([a], [da], wa), ([b, a], [db, da], wb), ([a, b], [da, db], wa)):
        if len(scenes) == 1:
            c.bin_events(*dev[0], scenes[0].t0, scenes[0].window_us)
        else:
            keep.append(_batch(c, scenes, dev))
        P.fill_(float("nan"))
        g.replay()
        c.stats()
        assert torch.equal(P, want)
    # a captured batch, replayed behind the host's back
    g2 = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g2):
        keep.append(_batch(c, [b, a], [db, da]))
    c.bin_events(*da, a.t0, a.window_us)
    g2.replay()
    assert torch.equal(_spectra(c, "blocked", a.W), wb)
    c.close()
