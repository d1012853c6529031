"""The state-parallel check of a few points (the automatic choice below 160
points) against the brute-force variants: same first collisions, costs and
winner, bit for bit, at the edges of its warps' rounds (T + 1 states a
multiple of 16 or 32, one more, one less), odd and even point counts, sample
counts that leave lanes empty, on both sides of its launch rule, with speed
limits."""
import numpy as np
import pytest

from paper_1904_06680_gb300 import inputs, npp

pytestmark = pytest.mark.gpu

CASES = [(16, 1, 1, 0), (16, 7, 15, 1), (16, 33, 16, 2), (32, 129, 30, 3), (16, 300, 31, 20), (64, 65, 32, 33),
         (16, 2049, 63, 64), (16, 8191, 20, 63), (16, 8193, 33, 63), (16, 8200, 33, 64), (32, 1024, 40, 159),
         (16, 1024, 20, 256), (16, 1025, 20, 159)]


def _plan(sc, variant):
    import torch
    N, T, M = sc["N"], sc["T"], len(sc["obs"])
    pl = npp.Planner(sc["preset"], max_N=N, max_T=T, max_M=max(M, 1))
    npp.npp_set_option(pl.h, "collide_variant", variant)
    obs = torch.tensor(sc["obs"], dtype=torch.float32, device="cuda") if M else None
    pl.plan(sc["state"], sc["goal"], obs, N, T, sc["seed"], sc["t_index"])
    r = pl.result(N, T)
    pl.close()
    return r


@pytest.mark.parametrize("limits", [False, True])
@pytest.mark.parametrize("width,N,T,M", CASES)
def test_equals_brute_force(width, N, T, M, limits):
    sc = inputs.tiny_scene(N + T + M, N=N, T=T, M=M, width=width, box=14.0)
    if limits:
        sc["preset"] = dict(sc["preset"], v_limits=1, v_min=-2.0, v_max=4.0)
    auto = _plan(sc, -1)
    for variant in (2, 3):
        b = _plan(sc, variant)
        for k in ("first_hit", "best_idx", "status"):
            assert np.array_equal(auto[k], b[k]), (k, variant)
        for k in ("costs", "params", "controls", "trajectory"):
            assert np.array_equal(np.asarray(auto[k]).view(np.uint32), np.asarray(b[k]).view(np.uint32)), (k, variant)
