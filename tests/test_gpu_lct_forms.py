"""The depth-map model's two forms (the convolution summed over its nonzeros,
and the padded FFTs for short time axes under wide maps) against the FP64
oracle, at the edges of blocks, windows and of the rule between them."""
import numpy as np
import pytest
import torch

from oracle import lct
from tests import gpu_helpers as H

pytestmark = pytest.mark.gpu


# direct: the smallest map (2 x 2), maps below a block and a patch of columns,
# one window and many, the largest time axis; on both sides of n^2 = 900 m:
# (64, 8) and (128, 32) direct, (64, 4) and (128, 16) by FFT
@pytest.mark.parametrize("n,m,offset", [(2, 2, 0), (2, 64, 1), (4, 4096, 0), (8, 16, 0), (16, 1024, 1),
                                        (32, 32, 0), (64, 8, 0), (64, 4, 0), (128, 32, 1), (128, 16, 0)])
def test_lct_forms_match_oracle(n, m, offset):
    from paper_2506_03747_gb300 import nlos
    H.lib()
    rng = np.random.default_rng(n + m)
    dt = 16e-12
    w = 0.3 * m * lct.C_LIGHT * dt
    depth = rng.integers(-2, m + 2, size=(n, n)).astype(np.int32)
    if n * n < 100:
        depth[0, 0] = m // 2  # at least one surface
    albedo = (rng.random((n, n)) - 0.25).astype(np.float32)  # signs and magnitudes as given
    buf = torch.empty(n * n * m + 4, device="cuda")
    tau = buf[offset:offset + n * n * m]  # offset 1: stores that are not 16-byte aligned
    plan = nlos.Lct(n, m, w, dt)
    for _ in range(2):  # a plan is used again
        tau.fill_(-1.0)
        plan.forward(torch.from_numpy(depth).cuda(), torch.from_numpy(albedo).cuda(), tau)
    torch.cuda.synchronize()
    plan.destroy()
    g = tau.cpu().numpy().reshape(n, n, m).astype(np.float64)
    o = lct.forward_direct_conv(depth, albedo.astype(np.float64), m, w, dt) if n <= 32 else \
        lct.forward(depth, albedo.astype(np.float64), m, w, dt)
    # FP64 sums rounded to FP32 (6e-8 relative); the transforms' round-off and
    # cancellation between signs scale with the largest value
    err = np.abs(g - o)
    assert (err <= 1e-6 * np.abs(o).max() + 1e-6 * np.abs(o)).all(), (err.max(), np.abs(o).max())
