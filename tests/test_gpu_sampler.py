"""The GPU sampler over (nearly) its whole argument grid.

Each Box-Muller pair takes a radius argument and an angle argument from
grids of 2^23 values; 2^26 normals are 2^25 pairs, which meet each value of
either grid with probability 1 - exp(-4) = 98 %.  The branch-free quotient,
root and argument reductions of the kernel equal the specification's IEEE
operations bit for bit (the oracle's, in plain C).
"""
import numpy as np
import pytest
import torch

from paper_1904_06680_gb300 import npp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,n_theta", [(0, 1 << 26), (7, (1 << 26) + 2), (123456789, 450), (3, 1)])
def test_normals_equal_the_oracle(orc, n, n_theta):
    seed, t, stream = 0x5EED0000 + n, 11, n % 5
    out = torch.empty(n_theta, dtype=torch.float32, device="cuda")
    npp.npp_sample_params(seed, t, stream, n, 1, n_theta, out)
    want = orc.theta(seed, t, n, n_theta, stream)
    got = out.cpu().numpy()
    bad = np.flatnonzero(got.view(np.uint32) != want.view(np.uint32))
    assert bad.size == 0, (bad.size, bad[:4], got[bad[:4]], want[bad[:4]])
