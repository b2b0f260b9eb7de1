"""Fused scores of pixels of 2048 events and more do not depend on how many blocks
their cluster has (four shares are added in the same order by four, two or one),
and are those of the unfused path."""
import pytest
import torch

from paper_2603_08386_gb300 import build, ddhf, synth
from test_gpu_listing import _scene

pytestmark = pytest.mark.gpu

COUNTS = [10, 300, 2047, 2048, 2049, 2080, 2175, 2176, 2177, 4095, 4097, 6100, 20_000]


@pytest.mark.parametrize("nb,M", [(100, 4), (400, 4), (640, 5), (750, 4), (1100, 4), (2100, 4)])
@pytest.mark.parametrize("wpb", [2, 4, 8])
def test_fused_cluster_size_does_not_change_the_bits(nb, M, wpb):
    build.build()
    s = _scene(9, COUNTS)
    ev = ddhf.events_to_device(s)

    def scores(**tuning):
        c = ddhf.Context(s.W, s.H, synth.hz_grid(0, 2, nb),
                         ddhf.default_params(n_min=1, M=M, tau_sf=1.0), max_events=s.n)
        c.set_tuning(warps_per_block=wpb, **tuning)
        mask = c.detect(*ev, s.t0, s.window_us, want_mask=True)[2].clone()
        sc = c.scores()
        c.stats()
        c.close()
        return [mask] + [sc[k].contiguous().view(torch.int32) for k in ("log_sf", "snr", "f0_bin")]

    try:
        want = scores(fuse=1)
    except ddhf.DDHFError:
        assert wpb == 8 and nb >= 640
        pytest.skip("the scratch of eight fused warps does not fit an SM")
    for tuning in [dict(fuse=0)] + [dict(fuse=1, blocks_per_sm=b) for b in (1, 2, 3, 4)]:
        for a, b in zip(want, scores(**tuning)):
            assert torch.equal(a, b), tuning
