"""The fixed heavy-pixel list of ddhf_power_spectrum_noalloc (32,768 entries, filled
from both ends): keys listed more often than it holds are flagged, the entries
that did not fit have NaN rows, and every other row is right. Beyond that many
active pixels those of 256 to 1023 events are in no list."""
import numpy as np
import pytest
import torch

from paper_2603_08386_gb300 import build, ddhf, synth

pytestmark = pytest.mark.gpu

ROOM, NB = 32768, 33


def _inputs(counts, rng):
    offsets = torch.tensor(np.concatenate([[0], np.cumsum(counts)]), dtype=torch.int32).cuda()
    n = sum(counts)
    ev = rng.integers(0, 30_000, n).astype(np.uint32) | (rng.integers(0, 2, n) << 31).astype(np.uint32)
    return offsets, torch.from_numpy(ev.view(np.int32)).cuda(), n


@pytest.mark.parametrize("n_active", [ROOM, ROOM + 1, 60_001])
@pytest.mark.parametrize("counts,nb", [([10, 255, 256, 300, 1023, 1024, 2048], NB), ([256], NB),
                                       ([3, 12], NB), ([20, 700], 1100)])
def test_many_active_pixels_around_the_team_threshold(n_active, counts, nb):
    build.build()
    rng = np.random.default_rng(8)
    offsets, ev, n = _inputs(counts, rng)
    g = ddhf.make_grid(0, 2000, synth.HZ_DENOM, nb)
    flags = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    rows = []
    for keys in (np.arange(len(counts)), rng.integers(0, len(counts), n_active)):
        act = torch.from_numpy(keys.astype(np.int32)).cuda()
        P = torch.full((keys.size, nb), -1.0, device="cuda")
        ddhf.ddhf_power_spectrum_noalloc(g, offsets, ev, n, act, keys.size, P, keys.size,
                                         flags=flags)
        torch.cuda.synchronize()
        assert int(flags.item()) == 0
        rows.append((act.long(), P))
    assert torch.equal(rows[1][1], rows[0][1][rows[1][0]])


@pytest.mark.parametrize("n_heavy,n_big", [(20_000, 20_000), (30_000, 2_768), (30_000, 2_769),
                                           (100, 40_000), (40_000, 100)])
def test_repeated_heavy_keys_of_both_classes(n_heavy, n_big):
    build.build()
    rng = np.random.default_rng(5)
    offsets, ev, n = _inputs([1024, 2048, 10], rng)
    g = ddhf.make_grid(0, 2000, synth.HZ_DENOM, NB)
    flags = torch.full((1,), -1, dtype=torch.int32, device="cuda")

    def spectra(keys):
        act = torch.from_numpy(keys.astype(np.int32)).cuda()
        P = torch.full((keys.size, NB), -1.0, device="cuda")
        ddhf.ddhf_power_spectrum_noalloc(g, offsets, ev, n, act, keys.size, P, keys.size,
                                         flags=flags)
        torch.cuda.synchronize()
        return P

    ref = spectra(np.arange(3))
    assert int(flags.item()) == 0
    keys = rng.permutation(np.repeat([0, 1, 2], [n_heavy, n_big, 50]))
    P = spectra(keys)
    lost = torch.isnan(P).all(dim=1)
    over = max(0, n_heavy + n_big - ROOM)
    assert int(lost.sum()) == over
    assert int(flags.item()) == (1 if over else 0)
    want = ref[torch.from_numpy(keys).cuda()]
    assert torch.equal(P[~lost], want[~lost])
    assert not lost[torch.from_numpy(keys).cuda() == 2].any()  # no light pixel is lost
