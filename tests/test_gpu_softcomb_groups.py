"""The soft comb over its lane groups (one, two or four harmonics at a time) and
frequency blocks (up to 8, 16 and 17 frequencies), with pixels of a few and of
many events and more pixels than one block of the gradient sums takes, against
the oracle's analytic FP64 values with the bars of test_gpu_softcomb."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_08386_gb300 import build, ddhf, synth
from test_gpu_softcomb import TOL_GRAD, TOL_S, oracle_all, worst

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def window():
    build.build()
    oracle.build()
    s = synth.small_scene(72, W=40, H=36, n_noise=24_000, drone_px=60, f0_hz=150.0,
                          window_us=40_000, grid=synth.hz_grid(0, 2, 750))
    c = ddhf.Context(s.W, s.H, s.grid, max_events=s.n)
    c.bin_events(*ddhf.events_to_device(s), s.t0, s.window_us)
    o = oracle.bin_events(s.W, s.H, s.x, s.y, s.t, s.p, s.t0, s.window_us)
    yield s, c, o
    c.close()


@pytest.mark.parametrize("nh,Q,delta", [(1, 3, 2.0), (2, 4, 1.5), (3, 1, 2.0), (5, 7, 0.5),
                                        (8, 8, 1.0), (4, 0, 2.0)])
def test_softcomb_groups_match_oracle(window, nh, Q, delta):
    s, c, o = window
    rng = np.random.default_rng(nh * 100 + Q)
    act = np.flatnonzero(o["counts"] >= 6)
    top = act[np.argsort(-o["counts"][act], kind="stable")[:20]]
    keys = np.concatenate([top, rng.choice(act, 560)])
    n = keys.size
    assert n > 512 and o["counts"][top].max() > 64
    d = dict(s=s, c=c, o=o, keys=keys, f0=rng.uniform(60, 200, n).astype(np.float32),
             w=rng.uniform(0.5, 1.5, nh).astype(np.float32),
             sg=rng.uniform(1.0, 4.0, nh).astype(np.float32),
             B=rng.uniform(2.0, 20.0, n).astype(np.float32),
             g=rng.uniform(-1.0, 1.0, n).astype(np.float32))
    cu = lambda a, dt=torch.float32: torch.as_tensor(a, dtype=dt).cuda()
    pix = cu(keys, torch.int32)
    args = (c.h, pix, cu(d["f0"]), nh, Q, delta, s.window_us / 2, cu(d["w"]), cu(d["sg"]),
            cu(d["B"]))
    S, gf0 = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
    gw, gs = torch.empty(nh, device="cuda"), torch.empty(nh, device="cuda")
    gf = torch.full((n, nh, 2 * Q + 1), float("nan"), device="cuda")
    ddhf.ddhf_softcomb(*args, S=S)
    ddhf.ddhf_softcomb(*args, grad_S=cu(d["g"]), grad_f0=gf0, grad_w=gw, grad_sigma=gs,
                       grad_f=gf)
    c.stats()
    ref = oracle_all(d, Q, delta)
    col = lambda k: np.stack([np.asarray(r[k]) for r in ref])
    g, gabs = d["g"].astype(np.float64), np.abs(d["g"]).astype(np.float64)
    assert worst(S.cpu().numpy() - col("S"), TOL_S * col("scale_S")) <= 1.0
    assert worst(gf0.cpu().numpy() - g * col("dS_df0"), TOL_GRAD * gabs * col("scale_df0")) <= 1.0
    assert worst(gf.cpu().numpy() - g[:, None, None] * col("dS_df"),
                 TOL_GRAD * gabs[:, None, None] * col("scale_df")) <= 1.0
    for got, k in ((gw, "dS_dw"), (gs, "dS_dsigma")):
        bar = TOL_GRAD * (gabs[:, None] * col("scale_" + k[3:])).sum(0)
        assert worst(got.cpu().numpy() - (g[:, None] * col(k)).sum(0), bar) <= 1.0
