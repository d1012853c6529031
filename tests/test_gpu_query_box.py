"""The bounding-box queries of the binned check against brute force over
vehicle shapes where the box differs most from a disk (long and thin, wide
and short, reference point at the rear) and, with polygons, a box far off the
reference point: first collisions, costs and winner bit for bit, with points
dense enough that collisions begin at every step."""
import numpy as np
import pytest

from paper_1904_06680_gb300 import inputs, npp

pytestmark = pytest.mark.gpu

SHAPES = dict(thin=dict(half_len=6.0, half_wid=0.1), wide=dict(half_len=0.2, half_wid=3.0),
              rear=dict(half_len=2.25, half_wid=0.9, c_off=4.0),
              ahead=dict(footprint=[[[4.0, -0.5], [6.0, -0.5], [6.0, 0.5], [4.0, 0.5]]]),
              bar=dict(footprint=[[[-5.0, -0.05], [5.0, -0.05], [5.0, 0.05], [-5.0, 0.05]],
                                  [[-0.1, -2.0], [0.1, -2.0], [0.1, 2.0], [-0.1, 2.0]]]))


def _plan(sc, variant, fuse):
    import torch
    N, T, M = sc["N"], sc["T"], len(sc["obs"])
    pl = npp.Planner(sc["preset"], max_N=N, max_T=T, max_M=M)
    npp.npp_set_option(pl.h, "collide_variant", variant)
    npp.npp_set_option(pl.h, "fuse", fuse)
    obs = torch.tensor(sc["obs"], dtype=torch.float32, device="cuda")
    pl.plan(sc["state"], sc["goal"], obs, N, T, sc["seed"], sc["t_index"])
    r = pl.result(N, T)
    pl.close()
    return r


@pytest.mark.parametrize("width,N,T,M", [(16, 1500, 15, 900), (32, 700, 33, 400), (64, 300, 20, 2000)])
@pytest.mark.parametrize("shape", sorted(SHAPES))
def test_equals_brute_force(shape, width, N, T, M):
    sc = inputs.tiny_scene(N + M, N=N, T=T, M=M, width=width, box=30.0, clear=7.0, vmax=6.0)
    sc["preset"] = dict(sc["preset"], **SHAPES[shape])
    want = _plan(sc, 2, -1)
    assert 0 < np.count_nonzero(want["first_hit"] > 0)
    for fuse in ((0, 1) if "footprint" not in SHAPES[shape] else (-1,)):
        got = _plan(sc, 5 if "footprint" not in SHAPES[shape] else -1, fuse)
        for k in ("first_hit", "best_idx", "status"):
            assert np.array_equal(got[k], want[k]), (k, fuse)
        for k in ("costs", "params", "controls", "trajectory"):
            assert np.array_equal(np.asarray(got[k]).view(np.uint32), np.asarray(want[k]).view(np.uint32)), (k, fuse)
