"""The sampler's listing of bright bins (expected counts of 30 and more) at the
ends of a part, where a warp's last step holds fewer than 32 groups of four
bins, beside bins whose searches end after very different numbers of steps,
against the oracle's sampler on the same expected counts."""
import numpy as np
import pytest
import torch

import oracle
from tests import gpu_helpers as H

pytestmark = pytest.mark.gpu


# groups of the last step: 1, 31, 32, 33 (aligned), and parts that start inside a group
@pytest.mark.parametrize("n,index_base", [(1, 0), (4, 3), (124, 0), (125, 2), (128, 0), (129, 1), (132, 0),
                                          (7168 * 3 + 61, 5)])
@pytest.mark.parametrize("bright", [0.02, 0.5, 1.0])  # share of bright bins: 1.0 overflows the list
def test_bright_bins_at_the_ends_of_a_part(n, index_base, bright):
    from paper_2506_03747_gb300 import nlos
    H.lib()
    rng = np.random.default_rng(n)
    tau = (rng.random(n) * rng.choice([0.001, 0.05, 0.29], n)).astype(np.float32)
    tau[rng.random(n) < bright] = np.float32(0.3) + rng.random(1).astype(np.float32)[0]
    tau[[0, -1]] = 1.0  # the first and the last bin of the part are listed
    t = torch.from_numpy(tau).cuda()
    c = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    nlos.noise(t, n, 100.0, 1e-3, seed=77, stream_tag=3, index_base=index_base, counts=c)
    torch.cuda.synchronize()
    got = c.cpu().numpy().view(np.uint32)
    lam = oracle.lam_from(tau.astype(np.float64), np.float32(100.0), np.float32(1e-3))
    ref = oracle.poisson(lam, index_base, 77, 3)
    # a search may end one step apart where the device's and the host's exp round apart:
    # at most a few of the bins, by one count
    off = got.astype(np.int64) - ref.astype(np.int64)
    assert (off != 0).sum() <= 3 and np.abs(off).max() <= 1
