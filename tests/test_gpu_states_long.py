"""The state-parallel check of a few points with two samples a warp (8192
samples and more) at the edges of its 16-step rounds, and at the horizon from
which it takes one sample a warp: same first collisions, costs and winner as
the brute-force variants, bit for bit."""
import numpy as np
import pytest
import torch

from paper_1904_06680_gb300 import inputs, npp

pytestmark = pytest.mark.gpu


def _plan(sc, variant):
    pl = npp.Planner(sc["preset"], max_N=sc["N"], max_T=sc["T"], max_M=len(sc["obs"]))
    npp.npp_set_option(pl.h, "collide_variant", variant)
    obs = torch.tensor(sc["obs"], dtype=torch.float32, device="cuda")
    pl.plan(sc["state"], sc["goal"], obs, sc["N"], sc["T"], sc["seed"], sc["t_index"])
    r = pl.result(sc["N"], sc["T"])
    pl.close()
    return r


@pytest.mark.parametrize("limits", [False, True])
@pytest.mark.parametrize("N,T,M", [(8193, 14, 63), (8193, 15, 20), (8193, 16, 21), (8192, 31, 63), (8194, 47, 1),
                                   (8193, 127, 20), (8193, 128, 20)])
def test_equals_brute_force(N, T, M, limits):
    sc = inputs.tiny_scene(N + T + M, N=N, T=T, M=M, box=14.0)
    if limits:
        sc["preset"] = dict(sc["preset"], v_limits=1, v_min=-2.0, v_max=4.0)
    auto = _plan(sc, -1)
    for variant in (2, 3):
        b = _plan(sc, variant)
        for k in ("first_hit", "best_idx", "status"):
            assert np.array_equal(auto[k], b[k]), (k, variant)
        for k in ("costs", "params", "controls", "trajectory"):
            assert np.array_equal(np.asarray(auto[k]).view(np.uint32), np.asarray(b[k]).view(np.uint32)), (k, variant)
