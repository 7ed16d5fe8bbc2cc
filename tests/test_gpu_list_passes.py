"""Scenes whose live-unit list takes several passes: the same transients as the
scan's rows rendered a few at a time (one pass each) and as the oracle on
sampled scan points; and the memory that such a scene holds."""
import numpy as np
import pytest
import torch

import oracle
import scenes
from tests import gpu_helpers as H

pytestmark = pytest.mark.gpu


def _params(**kw):
    return scenes.default_params(scan_nx=512, scan_ny=256, wall_half_x=0.5, wall_half_y=0.5, bin_width_s=40e-12,
                                 window_start_m=0.5, **kw)


# 4,096 tiles of 32 scan points and 1,075 blocks of points (592 for each of two windows of the splat)
@pytest.mark.parametrize("scan_mode", ["confocal", "nonconfocal"])
@pytest.mark.parametrize("kind", ["nearest", "occluded", "splat"])
def test_passes_match_rows_and_oracle(kind, scan_mode):
    from paper_2506_03747_gb300 import nlos
    H.lib()
    bins, extra = (40, dict(jitter_fwhm_s=60e-12)) if kind != "splat" else \
        (300, dict(jitter_fwhm_s=400e-12, bin_mode="splat"))
    params = _params(num_bins=bins, scan_mode=scan_mode, laser_xy=(0.1, 0.0), **extra)
    pts = scenes.random_points(np.random.default_rng(2), 1100001 if kind != "splat" else 303001, half=0.5,
                               z_lo=0.3, z_hi=0.6)
    occ = np.array([[0, 0.1, 0.0, 0.2, 0.08, 0, 0, 0]], np.float32)
    prm = nlos.params(params)
    sc = nlos.scene_create(prm, pts)
    if kind == "occluded":
        nlos.scene_set_occluders(sc, occ)
    tau = torch.full((sc.num_scan, bins), 7.0, device="cuda")
    for _ in range(2):  # the passes' counters are ready for a second call
        nlos.forward(sc, tau)
    nlos.scene_check(sc)
    whole = tau.view(256, 512, bins)
    for row in (0, 100, 252):
        part = nlos.scene_create_rows(prm, pts, row, 4)
        if kind == "occluded":
            nlos.scene_set_occluders(part, occ)
        t = torch.empty(part.num_scan, bins, device="cuda")
        nlos.forward(part, t)
        a, b = whole[row:row + 4].reshape(-1, bins).double(), t.double()
        # the same FP32 terms in another order: at most a few 1e-7 of a transient's peak for each
        # of the partial sums
        assert ((a - b).abs() <= 1e-5 * b.amax(dim=1, keepdim=True) + 1e-30).all(), row
        part.destroy()
    if kind == "nearest":
        for s in (0, 66000, 131071):
            o = oracle.forward_binned(params, pts, s, 1, eps=H.U_EPS)
            taps = oracle.jitter_taps(params["jitter_fwhm_s"], params["bin_width_s"])
            H.check_bins(tau[s:s + 1].double().cpu().numpy(), oracle.jitter(o["tau"], taps),
                         allow=oracle.jitter(o["flip_mass"], taps), what=f"s={s}")
    sc.destroy()


def test_pass_in_a_graph():
    from paper_2506_03747_gb300 import nlos
    H.lib()
    sc = nlos.scene_create(nlos.params(_params(num_bins=20)),
                           scenes.random_points(np.random.default_rng(2), 1100001, half=0.5, z_lo=0.3, z_hi=0.6))
    tau, ref = (torch.empty(sc.num_scan, 20, device="cuda") for _ in range(2))
    nlos.forward(sc, ref)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        nlos.forward(sc, tau)
    graph.replay()
    torch.cuda.synchronize()
    assert ((tau - ref).abs() <= 1e-5 * ref.amax(dim=1, keepdim=True)).all()
    sc.destroy()


def test_list_memory_is_bounded():
    """512 x 512 scan points and 2,000,000 surface points have 16 million units: the scene
    holds its points (75 bytes each), its scan tables and at most 64 MiB for the list."""
    from paper_2506_03747_gb300 import nlos
    H.lib()
    n = 2000000
    pts = torch.from_numpy(scenes.random_points(np.random.default_rng(1), n)).cuda()
    prm = nlos.params(dict(_params(num_bins=256), scan_ny=512))
    nlos.scene_create(prm, pts[:1000]).destroy()  # what a first scene loads
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    sc = nlos.scene_create(prm, pts)
    held = before - torch.cuda.mem_get_info()[0]
    sc.destroy()
    assert held <= 75 * n + 64 * 512 * 512 + (64 << 20) + (24 << 20), held  # (2 MiB pages, 12 arrays)
