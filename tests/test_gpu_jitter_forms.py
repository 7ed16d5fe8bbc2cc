"""The standalone jitter's forms (rows read as 16-byte words, staged rows, radii
above the unrolled ones) against the FP64 oracle at the edges of rows, words
and runs."""
import numpy as np
import pytest
import torch

import oracle
from tests import gpu_helpers as H

pytestmark = pytest.mark.gpu


# bins: below a word, odd, a multiple of 4 but not of 8, one run and more
# (1024 staged, 2048 direct); sigma 0 (a copy), radii 1, 8, 16 (the last
# unrolled) and 17; offset 1: rows that are not 16-byte aligned
@pytest.mark.parametrize("padding", ["zero", "replicate"])
@pytest.mark.parametrize("bins", [1, 4, 12, 31, 1024, 1025, 2052, 4100])
@pytest.mark.parametrize("sigma,offset", [(0.0, 0), (0.4, 0), (3.9, 0), (7.9, 0), (7.9, 1), (8.3, 0)])
def test_jitter_forms_match_oracle(bins, sigma, offset, padding):
    from paper_2506_03747_gb300 import nlos
    H.lib()
    traces = 5
    rng = np.random.default_rng(bins)
    x = rng.random((traces, bins)).astype(np.float32)
    xin = torch.empty(traces * bins + 4, device="cuda")[offset:offset + traces * bins].view(traces, bins)
    xin.copy_(torch.from_numpy(x))
    out = torch.full((traces * bins + 8,), -7.0, device="cuda")
    dt = 4e-12
    fwhm = sigma * dt * 2.0 * np.sqrt(2.0 * np.log(2.0))
    nlos.jitter(xin, out[4 + offset:], traces, bins, fwhm, dt, padding=padding)
    torch.cuda.synchronize()
    o = out.cpu().numpy()
    end = 4 + offset + traces * bins
    assert (o[:4 + offset] == -7.0).all() and (o[end:] == -7.0).all()  # nothing outside the rows
    ref = oracle.jitter(x.astype(np.float64), oracle.jitter_taps(fwhm, dt), padding)
    # at most 35 FP32 products of values up to 1 with taps that sum to 1
    assert np.abs(o[4 + offset:end].reshape(traces, bins) - ref).max() <= 40 * 2.0 ** -24
