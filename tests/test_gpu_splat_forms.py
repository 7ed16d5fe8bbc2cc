"""The splat's moment form at each number of rows a bin, and the per-tap form
beyond it, against the FP64 oracle: forward and adjoint at the smallest and
largest standard deviations of each, with pairs beyond both ends of the
window."""
import math

import numpy as np
import pytest
import torch

import oracle
import scenes
from tests import gpu_helpers as H

pytestmark = pytest.mark.gpu

# sigma in bins: 16, 8, 4 and 2 rows a bin, one row a bin (the last: 6 sigma + 1 =
# 60 bins of reach), taps
SIGMAS = [0.26, 0.39, 0.4, 0.78, 0.79, 1.56, 1.57, 2.49, 2.5, 9.8, 9.9]


def _case(sigma, bins, scan_mode, cos_mode):
    dt = 8e-12
    params = scenes.default_params(scan_nx=7, scan_ny=5, wall_half_x=0.4, wall_half_y=0.3, bin_width_s=dt,
                                   num_bins=bins, bin_mode="splat", scan_mode=scan_mode, cos_mode=cos_mode,
                                   laser_xy=(0.1, 0.05), window_start_m=0.9,
                                   jitter_fwhm_s=sigma * dt * 2 * math.sqrt(2 * math.log(2)))
    pts = scenes.random_points(np.random.default_rng(bins), 701, half=0.3, z_lo=0.4, z_hi=0.8)
    return params, pts


def _tolerance(sigma):
    # u in FP32 is within about 1e-4 bins of its FP64 value here (u below 400), and the kernel
    # moves by 0.61 / sigma of its peak a bin; 1e-5 covers the truncation (1.3e-6) and the sums
    return 1e-5 + 1e-4 / sigma


@pytest.mark.parametrize("bins,scan_mode,cos_mode", [(300, "confocal", "object"),
                                                     (77, "nonconfocal", "object_wall"),
                                                     (258, "confocal", "none")])
@pytest.mark.parametrize("sigma", SIGMAS)
def test_splat_forms_match_oracle(sigma, bins, scan_mode, cos_mode):
    from paper_2506_03747_gb300 import nlos
    params, pts = _case(sigma, bins, scan_mode, cos_mode)
    g = H.gpu_forward(params, pts, energy=False)
    o = oracle.forward_splat(params, pts)
    assert (o > 0).any()
    # a transient's own peak, or the cube's where only cut tails reach its window
    peak = np.maximum(o.max(axis=1, keepdims=True), 1e-2 * o.max())
    assert (np.abs(g["tau"] - o) <= _tolerance(sigma) * peak).all(), (np.abs(g["tau"] - o) / peak).max()
    S, B = g["tau"].shape
    gt = np.random.default_rng(1).normal(size=(S, B)).astype(np.float32)
    sc = g["scene"]
    ga = torch.empty(sc.num_points, device="cuda")
    gd = torch.empty(sc.num_points, device="cuda")
    nlos.simulate_backward(sc, torch.from_numpy(gt).cuda(), ga, gd)
    torch.cuda.synchronize()
    oa, od = oracle.backward_splat(params, pts, gt.astype(np.float64))
    for a, b in ((ga, oa), (gd, od)):
        assert np.abs(a.cpu().numpy() - b).max() <= 1e-3 * np.abs(b).max()
