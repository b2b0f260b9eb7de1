"""Dominant frequencies of boxes of every size: the work is cut into units of
each box's rows, so boxes from one pixel to the whole sensor, clipped,
overlapping, empty and inverted ones, and more boxes than the workspace has
records for, must all give the oracle's strongest pixel and lower median."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_08386_gb300 import build, ddhf, synth

pytestmark = pytest.mark.gpu


# (W, H, bins, step Hz): rows of several 256-pixel segments; a small sensor
# whose workspace holds fewer records (37) than there are boxes; a grid above
# the shared-memory histogram's 4096 bins
@pytest.mark.parametrize("W,H,nb,step", [(531, 40, 333, 5), (48, 40, 750, 2), (64, 50, 5000, 0.5)])
def test_box_frequencies_of_any_boxes(W, H, nb, step):
    build.build()
    oracle.build()
    s = synth.small_scene(17, W=W, H=H, n_noise=12 * W * H, drone_px=100,
                          grid=synth.hz_grid(0, step, nb))
    c = ddhf.Context(W, H, s.grid, max_events=s.n)
    _, _, mask = c.detect(*ddhf.events_to_device(s), s.t0, s.window_us, want_mask=True)
    sc = {k: v.cpu().numpy() if torch.is_tensor(v) else v for k, v in c.scores().items()}
    rng = np.random.default_rng(W)
    bx = [[0, 0, W - 1, H - 1], [-5, -5, W + 5, H + 5], [W // 2, 0, W // 2, H - 1],
          [0, H // 2, W - 1, H // 2], [3, 4, 3, 4], [10, 10, 5, 5], [W + 2, 0, W + 9, 5]]
    while len(bx) < 60:
        x, y = sorted(rng.integers(0, W, 2)), sorted(rng.integers(0, H, 2))
        bx.append([x[0], y[0], x[1], y[1]])
    bx = np.array([b + [1] for b in bx], np.int32)
    cap, n = 70, len(bx)
    boxes = torch.zeros((cap, 5), dtype=torch.int32, device="cuda")
    boxes[:n] = torch.from_numpy(bx).cuda()
    count = torch.tensor([n], dtype=torch.int32, device="cuda")
    f0 = torch.full((cap,), -7, dtype=torch.int32, device="cuda")
    snr = torch.full((cap,), -7.0, device="cuda")
    hz = torch.full((cap,), -7.0, device="cuda")
    ddhf.ddhf_box_frequencies(c.h, 0, boxes, count, cap, f0, snr, hz)
    only = torch.full((cap,), -7, dtype=torch.int32, device="cuda")
    ddhf.ddhf_box_frequencies(c.h, 0, boxes, count, cap, only)
    c.stats()
    c.close()
    m = mask.cpu().numpy()
    act = sc["active"].astype(np.int64)
    assert m.sum() > W * H // 4
    rf, rs = oracle.box_frequencies(bx, act, m, sc["snr"], sc["f0_bin"], W)
    np.testing.assert_array_equal(f0[:n].cpu().numpy(), rf)
    np.testing.assert_array_equal(only[:n].cpu().numpy(), rf)
    np.testing.assert_array_equal(snr[:n].cpu().numpy().view(np.int32), rs.view(np.int32))
    np.testing.assert_array_equal(hz[:n].cpu().numpy(),
                                  oracle.box_median_hz(bx, act, m, sc["f0_bin"], W, s.grid))
    assert (f0[n:] == -7).all() and (snr[n:] == -7).all() and (hz[n:] == -7).all()
