"""The 20-warp trajectory shape of width 16 against the register kernels, bit
for bit, on both sides of its rule in samples (16 and 20 warps of eight
samples on every SM): sampled and explicit parameters, with and without the
rollout variants."""
import numpy as np
import pytest
import torch

from paper_1904_06680_gb300 import inputs, npp

pytestmark = pytest.mark.gpu


def _sizes():
    per = 8 * torch.cuda.get_device_properties(0).multi_processor_count
    return (16 * per, 16 * per + 1, 18 * per + 13, 20 * per, 20 * per + 1)


@pytest.mark.parametrize("variant", [{}, dict(v_limits=1, v_min=-2.0, v_max=3.0), dict(feature_frame=1)])
@pytest.mark.parametrize("k", range(5))
def test_sampled(k, variant):
    N, T = _sizes()[k], 7
    sc = inputs.tiny_scene(k, N=N, T=T, M=30, width=16)
    sc["preset"] = dict(sc["preset"], **variant)
    obs = torch.tensor(sc["obs"], dtype=torch.float32, device="cuda")
    out = []
    for shape in (0, 3 if not variant else 2):
        pl = npp.Planner(sc["preset"], max_N=N, max_T=T, max_M=30)
        npp.npp_set_option(pl.h, "traj_variant", shape)
        pl.plan(sc["state"], sc["goal"], obs, N, T, sc["seed"], sc["t_index"])
        out.append(pl.result(N, T))
        pl.close()
    for key in ("costs", "first_hit", "params", "controls", "trajectory"):
        a, b = (np.ascontiguousarray(r[key]).view(np.uint32) for r in out)
        assert np.array_equal(a, b), key


def test_explicit():
    K, T, nt = _sizes()[1], 5, 450
    sc = inputs.tiny_scene(1, N=K, T=T, M=30, width=16)
    obs = torch.tensor(sc["obs"], dtype=torch.float32, device="cuda")
    theta = torch.randn(K * nt, generator=torch.Generator(device="cuda").manual_seed(3), device="cuda")
    out = []
    for shape in (0, 3):
        pl = npp.Planner(sc["preset"], max_N=K, max_T=T, max_M=30)
        npp.npp_set_option(pl.h, "traj_variant", shape)
        r = [torch.zeros(K, device="cuda"), torch.zeros(K, dtype=torch.int32, device="cuda"),
             torch.zeros(T + 1, K, 4, device="cuda"), torch.zeros(T, K, 2, device="cuda")]
        npp.npp_rollout_params(pl.h, sc["state"], sc["goal"], obs, 30, theta, K, T, *r)
        out.append([x.cpu().numpy().view(np.uint32) for x in r])
        pl.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
