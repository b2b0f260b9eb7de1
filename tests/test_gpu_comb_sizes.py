"""The fast comb at the sizes where it changes: a bin index of one more bit in
its sort keys (1024, 2048, 4096, 8192 bins), more histogram buckets above 4096,
Table 2's comb shape and others. Bit for bit the oracle's FP32 comb."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2603_08386_gb300 import build, ddhf, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,n_px,M,d,h_min", [
    (1024, 40, 4, 3, 4), (1026, 40, 4, 3, 3), (2047, 32, 4, 3, 4), (2049, 32, 6, 2, 3),
    (2300, 24, 2, 1, 1), (4096, 12, 4, 3, 4), (4097, 12, 4, 3, 4), (4099, 8, 5, 2, 4),
    (8193, 4, 4, 3, 4)])
def test_comb_bit_exact_where_its_layout_changes(N, n_px, M, d, h_min):
    build.build()
    oracle.build()
    params = ddhf.default_params(M=M, d=d, h_min=h_min, n_min=1)
    c = ddhf.Context(n_px, 1, synth.hz_grid(0, 1, N), params, max_events=n_px)
    one = torch.ones(n_px, dtype=torch.int8, device="cuda")
    c.bin_events(torch.arange(n_px, device="cuda").to(torch.int16), (one - 1).to(torch.int16),
                 (one - 1).long(), one, 0, 100)
    half = n_px // 2
    Pn = np.concatenate([synth.synthetic_spectra(half, N, seed=N),
                         synth.clustered_spectra(n_px - half, N, seed=N + 1)])
    out = {k: v.cpu().numpy() for k, v in c.comb_score(torch.from_numpy(Pn).cuda()).items()}
    c.stats()
    c.close()
    scored = 0
    for a in range(n_px):
        lo = oracle.log_sf(Pn[a].astype(np.float64))
        assert abs(out["log_sf"][a] - lo) <= 1e-4 * max(1.0, abs(lo))
        if out["log_sf"][a] <= np.float32(math.log(0.89)):
            s32, w32 = oracle.comb_f32(Pn[a], M=M, d=d, h_min=h_min)
            assert w32 == out["f0_bin"][a], (a, w32, out["f0_bin"][a])
            assert np.float32(s32).view(np.uint32) == out["snr"][a].view(np.uint32), a
            scored += 1
        else:
            assert out["f0_bin"][a] == -1 and out["snr"][a] == 0 and out["mask"][a] == 0
    assert scored > n_px // 3
