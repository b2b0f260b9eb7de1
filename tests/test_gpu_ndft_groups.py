"""The tensor-core NDFT where its work changes hands: event counts at the edges
of its 8-event groups, 32-event chunks, four-warp teams (256) and clusters
(2048), bins at the edges of its 32-bin rows and of its 8-row tiles, one and
several passes; against the oracle, and the same bits from every launch shape
and entry point that must agree."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_08386_gb300 import build, ddhf, synth

pytestmark = pytest.mark.gpu

COUNTS = [1, 2, 7, 8, 9, 31, 32, 33, 63, 64, 65, 255, 256, 257, 300, 2047, 2048, 2049, 6100]
# against the peak power of the pixel; the FP32 sums of 6100 terms and the
# factors' 9 rotation steps of 2^-24 each stay below a few 1e-6
TOL = 1e-5


def _scene(nb, a0=0, da=2000, denom=synth.HZ_DENOM):
    rng = np.random.default_rng(nb)
    win = 30_000
    key = np.repeat(np.arange(len(COUNTS)), COUNTS)
    t = rng.integers(0, win, key.size)
    p = rng.choice(np.array([-1, 1], np.int8), key.size)
    # pixels whose polarities cancel: the power at 0 Hz is exactly zero
    for k, n in enumerate(COUNTS):
        if n % 2 == 0:
            p[np.flatnonzero(key == k)] = np.tile(np.array([-1, 1], np.int8), n // 2)
    order = np.argsort(t, kind="stable")
    return synth.Scene(W=len(COUNTS), H=1, t0=0, window_us=win,
                       x=key[order].astype(np.int16), y=np.zeros(key.size, np.int16),
                       t=t[order].astype(np.int64), p=p[order], grid=(a0, da, denom, nb))


def _spectra(s, ev, **tuning):
    c = ddhf.Context(s.W, s.H, s.grid, ddhf.default_params(n_min=1), max_events=s.n)
    if tuning:
        c.set_tuning(**tuning)
    c.bin_events(*ev, s.t0, s.window_us)
    P, csr = c.power_spectrum("blocked").clone(), c.csr()
    c.stats()
    c.close()
    return P, csr


@pytest.mark.parametrize("nb,a0,da,denom", [
    (1, 0, 2000, synth.HZ_DENOM), (31, 0, 2000, synth.HZ_DENOM), (33, 500, 2000, synth.HZ_DENOM),
    (256, 0, 1, 30_000), (257, 0, 2000, synth.HZ_DENOM), (750, 0, 2000, synth.HZ_DENOM),
    (1025, 7, 1500, synth.HZ_DENOM), (2000, 0, 1000, synth.HZ_DENOM), (100, 0, 1, 40)])
def test_blocked_spectra_at_every_edge(nb, a0, da, denom):
    build.build()
    oracle.build()
    s = _scene(nb, a0, da, denom)
    ev = ddhf.events_to_device(s)
    P, csr = _spectra(s, ev)
    o = oracle.bin_events(s.W, s.H, s.x, s.y, s.t, s.p, s.t0, s.window_us)
    Pn = P.cpu().numpy().astype(np.float64)
    for k in range(s.W):
        o0, o1 = o["offsets"][k], o["offsets"][k + 1]
        ref = oracle.ndft(o["tau"][o0:o1], o["pol"][o0:o1], *s.grid)
        assert np.abs(Pn[k] - ref).max() <= TOL * ref.max(), (k, COUNTS[k])
        # bins whose frequency is a multiple of denom: the squared polarity sum
        zero = np.flatnonzero((a0 + da * np.arange(nb)) % denom == 0)
        want = float(o["pol"][o0:o1].astype(np.int64).sum()) ** 2
        assert (Pn[k][zero] == np.float32(want)).all(), (k, zero[:4])
    # the same bits without a context, and (below the cluster's 2048 events)
    # from blocks of two, four and eight warps
    Q = torch.full_like(P, -1.0)
    ddhf.ddhf_power_spectrum_noalloc(ddhf.make_grid(*s.grid), csr["offsets"], csr["ev"],
                                     csr["n_valid"], csr["active"], P.shape[0], Q, P.shape[0])
    assert torch.equal(P, Q)
    small = torch.tensor([n < 2048 for n in COUNTS], device="cuda")
    for w in (2, 8):
        R, _ = _spectra(s, ev, warps_per_block=w)
        assert torch.equal(P[small], R[small]), w
    A, _ = _spectra(s, ev, heavy_min=1 << 30)
    B, _ = _spectra(s, ev, heavy_min=1 << 30, warps_per_block=2, blocks_per_sm=1)
    assert torch.equal(A, B) and torch.equal(A[small], P[small])


@pytest.mark.parametrize("nb,rows,wpb", [(630, 1, 8), (640, 1, 8), (640, 2, 4), (96, 1, 2),
                                         (300, 0, 8)])
def test_fused_spectra_fill_their_shared_rows(nb, rows, wpb):
    # a comb of 35 bins takes the generic scoring, whose scratch leaves eight
    # warps of a block just the 20 rows of 640 bins
    build.build()
    s = _scene(nb)
    ev = ddhf.events_to_device(s)
    out = []
    for fuse in (1, 0):
        c = ddhf.Context(s.W, s.H, s.grid, ddhf.default_params(n_min=1, M=5, d=3, tau_sf=1.0),
                         max_events=s.n)
        c.set_tuning(fuse=fuse, rows_per_lane=rows, warps_per_block=wpb)
        mask = c.detect(*ev, s.t0, s.window_us, want_mask=True)[2].clone()
        sc = {k: c.scores()[k].clone() for k in ("f0_bin", "snr", "log_sf")}
        c.stats()
        c.close()
        out.append((mask, sc))
    assert torch.equal(out[0][0], out[1][0])
    for k in out[0][1]:
        assert torch.equal(out[0][1][k].view(torch.int32), out[1][1][k].view(torch.int32)), k
