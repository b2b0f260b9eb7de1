"""ddhf_comb_score on rows with negative values, which no power is but a caller's
buffer may hold: the call stays inside its scratch (every other row's bits are
unchanged, at sizes whose scratch is smaller than a histogram's index range too)
and reports them."""
import numpy as np
import pytest
import torch

from paper_2603_08386_gb300 import build, ddhf, synth

pytestmark = pytest.mark.gpu

N_PX = 67


def _context(N, M, d, h_min, **kw):
    build.build()
    c = ddhf.Context(N_PX, 1, synth.hz_grid(0, 1, N),
                     ddhf.default_params(M=M, d=d, h_min=h_min, n_min=1, tau_sf=1.0, **kw),
                     max_events=N_PX)
    one = torch.ones(N_PX, dtype=torch.int8, device="cuda")
    c.bin_events(torch.arange(N_PX, device="cuda").to(torch.int16), (one - 1).to(torch.int16),
                 (one - 1).long(), one, 0, 100)
    return c


def _bits(out, rows):
    return [out[k][rows].contiguous().view(torch.uint8) for k in ("log_sf", "snr", "f0_bin")] + \
        [out["mask"][:N_PX][rows]]


@pytest.mark.parametrize("N,M,d,h_min", [
    (40, 2, 1, 1), (100, 4, 3, 4), (250, 4, 3, 4), (257, 6, 2, 3), (750, 4, 3, 4),
    (1000, 4, 3, 4), (2000, 4, 3, 4), (5000, 4, 3, 4)])
def test_negative_values_touch_no_other_row(N, M, d, h_min):
    c = _context(N, M, d, h_min)
    rng = np.random.default_rng(N)
    P = synth.synthetic_spectra(N_PX, N, seed=N).astype(np.float32)
    good = torch.from_numpy(np.flatnonzero(np.arange(N_PX) % 3 != 1)).cuda()
    want = _bits(c.comb_score(torch.from_numpy(P).cuda()), good)
    c.stats()
    B = P.copy()
    for a in range(1, N_PX, 3):
        B[a] = rng.exponential(1.0, N)
        at = rng.choice(N, max(2, N // 20), replace=False)
        B[a, at] = -np.exp(rng.uniform(-12, 1, at.size))  # from far below the mean to above it
    got = _bits(c.comb_score(torch.from_numpy(B).cuda()), good)
    with pytest.raises(ddhf.DDHFError) as e:
        c.stats()
    assert e.value.status == 2
    again = _bits(c.comb_score(torch.from_numpy(P).cuda()), good)
    c.stats()  # the flag was cleared
    c.close()
    for w, g, r in zip(want, got, again):
        assert torch.equal(w, g) and torch.equal(w, r)


@pytest.mark.parametrize("N", [100, 750, 2000])
def test_rows_of_negative_zero_score_as_zero(N):
    c = _context(N, 4, 3, 4, tau_comb=0.0)
    Z = torch.zeros((N_PX, N), device="cuda")
    zero, neg = c.comb_score(Z), c.comb_score(-Z)
    c.stats()
    c.close()
    assert (zero["f0_bin"] == 3).all() and (zero["mask"][:N_PX] == 1).all()
    for k in ("log_sf", "snr", "f0_bin", "mask"):
        assert torch.equal(zero[k], neg[k]), k
