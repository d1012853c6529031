"""The scene encoding's two 32-bit sums per bin against whole numbers: point
counts around a block's threads and the points a thread has in flight, and
on both sides of the count from which the sums carry into a third word."""
import numpy as np
import pytest
import torch

from paper_1904_06680_gb300 import inputs, npp, proposal

pytestmark = pytest.mark.gpu


# px: at the vehicle (weight 1, upper sum largest), and just inside the
# histogram's radius (weight 255 / 2^24, lower sum largest)
@pytest.mark.parametrize("px", [0.0, 20.0 * (1.0 - 255.0 * 2.0 ** -24)])
@pytest.mark.parametrize("M", [1, 511, 513, 2047, 2049, 65535, 65536, 131073, 200001])
def test_sums_of_equal_points(M, px):
    sc = inputs.tiny_scene(3, N=64, T=10, M=16, width=16)
    pl = npp.Planner(sc["preset"], max_N=64, max_T=10, max_M=M)
    obs = torch.zeros(M, 4, device="cuda")
    obs[:, 0] = px
    one = dict(state=(0, 0, 0, 5, 0, 0), goal=sc["goal"], N=64, T=10, M=M, width=16, obs_offset=0, seed=1)
    x = proposal.encode(pl, [one], obs)[0, :64].double().cpu().numpy()
    w = np.float32(1.0) - np.float32(px) / np.float32(20.0)
    h = float(M) * float(w)
    k = 32                                     # heading 0
    want = np.zeros(64)
    want[k] = h / (1 + h)
    # w is off by half an ulp of px / 20 at most (2^-25 of 255 / 2^24: 0.2 %),
    # dx = dh / (1 + h)^2, and x is rounded to FP32 after two operations; a
    # lost carry is 1 or 65536 of h
    tol = 0.004 * h / (1 + h) ** 2 + 2 * 2.0 ** -24
    assert np.max(np.abs(x - want)) <= tol
    lost = h - (65536.0 if px == 0.0 else 1.0)
    if M > 65536:
        assert abs(max(lost, 0) / (1 + max(lost, 0)) - want[k]) > 2 * tol
    pl.close()
