"""The check with a step's grid in shared memory (the automatic choice from
1024 samples on) against brute force: same first collisions, costs and
winner, bit for bit, on both sides of its rule in samples and points, at
sample counts that leave a block one state, at a chunk's edge, with odd
numbers of points, without any, and with speed limits; first collisions start
afresh on every call."""
import numpy as np
import pytest

from paper_1904_06680_gb300 import inputs, npp

pytestmark = pytest.mark.gpu


def _plans(sc, variant, calls=1):
    import torch
    N, T, M = sc["N"], sc["T"], len(sc["obs"])
    pl = npp.Planner(sc["preset"], max_N=N, max_T=T, max_M=max(M, 1))
    npp.npp_set_option(pl.h, "collide_variant", variant)
    npp.npp_set_option(pl.h, "fuse", 0)
    obs = torch.tensor(sc["obs"], dtype=torch.float32, device="cuda") if M else None
    out = []
    for k in range(calls):
        pl.plan(sc["state"], sc["goal"], obs, N, T, sc["seed"], sc["t_index"] + k)
        out.append(pl.result(N, T))
    pl.close()
    return out


@pytest.mark.parametrize("limits", [False, True])
@pytest.mark.parametrize("width,N,T,M", [(16, 1023, 9, 300), (16, 1024, 1, 301), (16, 1025, 40, 999), (32, 1537, 20, 161),
                                         (32, 5003, 61, 800), (16, 2049, 30, 8702), (16, 2049, 30, 8703), (64, 1500, 7, 500),
                                         (16, 20001, 455, 400)])
def test_equals_brute_force(width, N, T, M, limits):
    sc = inputs.tiny_scene(N + T + M, N=N, T=T, M=M, width=width, box=25.0, vmax=5.0)
    if limits:
        sc["preset"] = dict(sc["preset"], v_limits=1, v_min=-2.0, v_max=4.0)
    for got, want in zip(_plans(sc, 5, 2), _plans(sc, 2, 2)):
        for k in ("first_hit", "best_idx", "status"):
            assert np.array_equal(got[k], want[k]), k
        for k in ("costs", "params", "controls", "trajectory"):
            assert np.array_equal(np.asarray(got[k]).view(np.uint32), np.asarray(want[k]).view(np.uint32)), k


def test_without_points():
    sc = inputs.tiny_scene(4, N=2000, T=9, M=0, width=16)
    (got,), (want,) = _plans(sc, 5), _plans(sc, 2)
    assert np.all(got["first_hit"] == -1)
    assert np.array_equal(got["costs"].view(np.uint32), want["costs"].view(np.uint32))
