"""The depth-map model on rough maps: blocks of pixels that span many windows of
rows have their pixels tested one by one. Maps with blocks just below and above
that rule, blocks with missing pixels and an odd number of such blocks against
the FP64 oracle, and a random map against a smooth one in time."""
import numpy as np
import pytest
import torch

from oracle import lct
from tests import gpu_helpers as H

pytestmark = pytest.mark.gpu


def _map(n, m, span, rng):
    """Depths whose squared-time rows span `span` within each 4 x 4 block."""
    row = rng.integers(0, max(1, m - span), (n // 4, n // 4))
    rows = np.repeat(np.repeat(row, 4, 0), 4, 1) + rng.integers(0, span + 1, (n, n))
    rows[::4, ::4] = np.repeat(np.repeat(row, 4, 0), 4, 1)[::4, ::4]
    rows[3::4, 3::4] = rows[::4, ::4] + span
    z = np.floor(np.sqrt((np.minimum(rows, m - 1) + 1.0) * m)).astype(np.int32) - 1
    z[rng.random((n, n)) < 0.1] = -1  # no surface
    return z


# windows of 32 rows (n <= 64, rule at 80) and of 64 (rule at 160)
@pytest.mark.parametrize("n,m,span", [(4, 512, 400), (8, 256, 79), (8, 256, 83), (32, 512, 78), (32, 512, 84),
                                      (64, 256, 200), (128, 256, 158), (128, 256, 164), (128, 64, 63)])
def test_rough_maps_match_oracle(n, m, span):
    from paper_2506_03747_gb300 import nlos
    H.lib()
    rng = np.random.default_rng(n + span)
    dt = 16e-12
    w = 0.3 * m * lct.C_LIGHT * dt
    depth = _map(n, m, span, rng)
    if n >= 8:
        depth[:4, :4] = m // 2  # one smooth block among the others
    albedo = (rng.random((n, n)) - 0.25).astype(np.float32)
    tau = torch.empty(n * n * m, device="cuda")
    plan = nlos.Lct(n, m, w, dt)
    plan.forward(torch.from_numpy(depth).cuda(), torch.from_numpy(albedo).cuda(), tau)
    torch.cuda.synchronize()
    plan.destroy()
    g = tau.cpu().numpy().reshape(n, n, m).astype(np.float64)
    f = lct.forward_direct_conv if n <= 32 else lct.forward
    o = f(depth, albedo.astype(np.float64), m, w, dt)
    # FP64 sums rounded to FP32 (6e-8 relative); the oracle's transforms scale with the largest value
    assert (np.abs(g - o) <= 1e-6 * np.abs(o).max() + 1e-6 * np.abs(o)).all()


def test_random_map_costs_a_few_smooth_ones():
    """128 x 128 pixels, 1024 bins: 3.0 ms against 1.3 (8.3 with every block taken whole)."""
    from paper_2506_03747_gb300 import nlos
    H.lib()
    n, m = 128, 1024
    y, x = np.mgrid[0:n, 0:n] / n
    smooth = 0.35 + 0.2 * np.exp(-((x - 0.5) ** 2 + (y - 0.4) ** 2) / 0.05) + 0.05 * x
    plan = nlos.Lct(n, m, 1.0, 32e-12)
    tau = torch.empty(n * n * m, device="cuda")
    ms = []
    for z in (smooth, np.random.default_rng(0).random((n, n))):
        d = torch.from_numpy((z * m).astype(np.int32)).cuda()
        times = []
        for k in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            plan.forward(d, None, tau)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        ms.append(sorted(times[2:])[3])
    plan.destroy()
    assert ms[1] <= 4.0 * ms[0], ms
