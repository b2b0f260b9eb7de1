"""Box frequencies where boxes of one unit (4096 pixels) and of several meet, on
grids below, at and above the shared-memory histogram's 4096 bins; more boxes of
several units than there are records, and more boxes than the workspace has
entries for."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_08386_gb300 import build, ddhf, synth
from test_gpu_box_f0 import test_box_frequencies_of_any_boxes as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,nb,step", [(200, 100, 5000, 0.5), (256, 32, 4096, 0.5),
                                         (310, 130, 100, 10)])
def test_units_and_whole_boxes(W, H, nb, step):
    check(W, H, nb, step)


@pytest.mark.parametrize("W,H,nb,step,n,large", [
    (128, 64, 5000, 0.5, 60, 0.8),  # 24 records
    (8, 4, 100, 10, 300, 0.5)])     # 120 entries
def test_more_boxes_than_the_workspace_holds(W, H, nb, step, n, large):
    build.build()
    oracle.build()
    s = synth.small_scene(17, W=W, H=H, n_noise=12 * W * H, drone_px=min(100, W * H // 2),
                          grid=synth.hz_grid(0, step, nb))
    c = ddhf.Context(W, H, s.grid, max_events=s.n)
    _, _, mask = c.detect(*ddhf.events_to_device(s), s.t0, s.window_us, want_mask=True)
    sc = {k: v.cpu().numpy() if torch.is_tensor(v) else v for k, v in c.scores().items()}
    rng = np.random.default_rng(n)
    bx = []
    for _ in range(n):
        if rng.random() < large:  # nearly the whole sensor
            bx.append([rng.integers(0, 3), rng.integers(0, 3), W - 1 - rng.integers(0, 3), H - 1])
        else:
            x, y = sorted(rng.integers(0, W, 2)), sorted(rng.integers(0, H, 2))
            bx.append([x[0], y[0], x[1], y[1]])
    bx = np.array([list(b) + [1] for b in bx], np.int32)
    count = torch.tensor([n], dtype=torch.int32, device="cuda")
    f0 = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    snr, hz = torch.full((n,), -7.0, device="cuda"), torch.full((n,), -7.0, device="cuda")
    ddhf.ddhf_box_frequencies(c.h, 0, torch.from_numpy(bx).cuda(), count, n, f0, snr, hz)
    c.stats()
    c.close()
    m, act = mask.cpu().numpy(), sc["active"].astype(np.int64)
    rf, rs = oracle.box_frequencies(bx, act, m, sc["snr"], sc["f0_bin"], W)
    np.testing.assert_array_equal(f0.cpu().numpy(), rf)
    np.testing.assert_array_equal(snr.cpu().numpy().view(np.int32), rs.view(np.int32))
    np.testing.assert_array_equal(hz.cpu().numpy(),
                                  oracle.box_median_hz(bx, act, m, sc["f0_bin"], W, s.grid))
