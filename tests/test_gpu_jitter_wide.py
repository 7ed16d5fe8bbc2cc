"""The standalone jitter at radii above the unrolled ones, where four taps are
taken at a time: every remainder of the radius by four, rows shorter than the
radius, odd rows and unaligned buffers, against the oracle; and its time."""
import math

import numpy as np
import pytest
import torch

import oracle
from tests import gpu_helpers as H

pytestmark = pytest.mark.gpu

DT = 4e-12


def _fwhm(sigma):
    return sigma * DT * 2.0 * math.sqrt(2.0 * math.log(2.0))


@pytest.mark.parametrize("padding", ["zero", "replicate"])
@pytest.mark.parametrize("bins,offset", [(1, 0), (5, 1), (64, 0), (1024, 0), (1027, 3), (2500, 0)])
@pytest.mark.parametrize("radius", [17, 18, 19, 20, 63, 200, 1024])
def test_wide_radii_match_oracle(radius, bins, offset, padding):
    from paper_2506_03747_gb300 import nlos
    H.lib()
    traces, sigma = 3, radius / 2.0 - 0.1  # R = ceil(2 sigma)
    x = np.random.default_rng(bins).random((traces, bins)).astype(np.float32)
    xin = torch.empty(traces * bins + 4, device="cuda")[offset:offset + traces * bins].view(traces, bins)
    xin.copy_(torch.from_numpy(x))
    out = torch.full((traces * bins + 8,), -7.0, device="cuda")
    nlos.jitter(xin, out[4:], traces, bins, _fwhm(sigma), DT, padding=padding)
    torch.cuda.synchronize()
    o = out.cpu().numpy()
    assert (o[:4] == -7.0).all() and (o[4 + traces * bins:] == -7.0).all()
    taps = oracle.jitter_taps(_fwhm(sigma), DT)
    assert len(taps) == 2 * radius + 1
    ref = oracle.jitter(x.astype(np.float64), taps, padding)
    # each of the 2 R + 1 FP32 additions rounds a partial sum of at most 1; each tap is rounded once
    bound = (2 * radius + 1) * 2.0 ** -25 + 2.0 ** -24
    assert np.abs(o[4:4 + traces * bins].reshape(traces, bins) - ref).max() <= bound


def test_wide_radius_time():
    """401 taps against 13 on 16,384 x 1,024 bins: 16 times as long (29 with one word a tap)."""
    from paper_2506_03747_gb300 import nlos
    H.lib()
    x = torch.rand(16384, 1024, device="cuda")
    out = torch.empty_like(x)
    us = []
    for sigma in (3.0, 100.0):
        times = []
        for _ in range(9):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(4):
                nlos.jitter(x, out, 16384, 1024, _fwhm(sigma), DT)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) * 250.0)
        us.append(sorted(times[2:])[3])
    assert us[1] <= 23.0 * us[0], us
