"""Ordering and staging at their edges: point counts around warps, groups,
blocks and grids, points without weight (dark, or facing away from the laser),
a scene's points replaced twice, and the same calls captured in a CUDA graph,
against the FP64 oracle."""
import numpy as np
import pytest
import torch

import scenes
from tests import gpu_helpers as H

pytestmark = pytest.mark.gpu


def _params(scan_mode, **kw):
    return scenes.default_params(scan_nx=9, scan_ny=7, wall_half_x=0.5, wall_half_y=0.5, bin_width_s=16e-12,
                                 num_bins=203, window_start_m=0.3, scan_mode=scan_mode,
                                 laser_xy=(0.2, -0.1), jitter_fwhm_s=60e-12, **kw)


def _points(n, seed):
    pts = scenes.random_points(np.random.default_rng(seed), n)
    pts[::3, 6] = 0.0  # dark
    pts[1::5, 3:6] *= -1.0  # most of these face away from every spot
    return pts


def _check(params, pts, tau):
    o = H.oracle_with_allowance(params, pts)
    H.check_bins(tau.cpu().numpy().astype(np.float64), o["tau_g"], allow=o["flip_g"], what=f"{len(pts)} points")


@pytest.mark.parametrize("scan_mode", ["confocal", "nonconfocal"])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 64, 513, 1023, 1025, 4097, 20001])
def test_replaced_points_match_oracle(n, scan_mode):
    from paper_2506_03747_gb300 import nlos
    H.lib()
    params = _params(scan_mode)
    sc = nlos.scene_create(nlos.params(params), _points(n, 1))
    tau = torch.empty(sc.num_scan, sc.num_bins, device="cuda")
    nlos.forward(sc, tau)
    _check(params, _points(n, 1), tau)
    for seed in (2, 3):
        nlos.scene_set_points(sc, torch.from_numpy(_points(n, seed)).cuda())
        nlos.forward(sc, tau)
    nlos.scene_check(sc)
    _check(params, _points(n, 3), tau)


def test_points_without_weight_give_nothing():
    from paper_2506_03747_gb300 import nlos
    H.lib()
    pts = _points(3000, 4)
    pts[:, 6] = 0.0
    sc = nlos.scene_create(nlos.params(_params("confocal")), pts)
    tau = torch.full((sc.num_scan, sc.num_bins), 3.0, device="cuda")
    nlos.forward(sc, tau)
    assert not tau.any()


def test_pass_captured_in_a_graph():
    from paper_2506_03747_gb300 import nlos
    H.lib()
    params = _params("nonconfocal", noise_mode="peak")
    sc = nlos.scene_create(nlos.params(params), _points(4097, 5))
    pts = torch.from_numpy(_points(4097, 6)).cuda()
    tau = torch.empty(sc.num_scan, sc.num_bins, device="cuda")
    counts = torch.empty(tau.shape, device="cuda", dtype=torch.int32)
    energy = torch.empty(sc.num_scan, device="cuda", dtype=torch.float64)

    def step():
        nlos.scene_set_points(sc, pts)
        nlos.forward(sc, tau)
        nlos.detect(sc, tau, counts, energy)

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step()
    pts.copy_(torch.from_numpy(_points(4097, 7)))
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    nlos.scene_check(sc)
    _check(params, _points(4097, 7), tau)
    assert int(counts.sum()) > 0 and torch.allclose(energy, tau.double().sum(dim=1), rtol=1e-9)
