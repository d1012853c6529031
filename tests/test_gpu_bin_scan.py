"""The grid build's scan: first collisions of the binned check equal brute
force with every point in one cell, in a warp's first and last cells, and
spread so that each of the scan's rounds and warps carries a sum on."""
import numpy as np
import pytest
import torch

from paper_1904_06680_gb300 import inputs, npp

pytestmark = pytest.mark.gpu


def _hits(sc, variant):
    N, T, M = sc["N"], sc["T"], len(sc["obs"])
    pl = npp.Planner(sc["preset"], max_N=N, max_T=T, max_M=M)
    npp.npp_set_option(pl.h, "collide_variant", variant)
    obs = torch.tensor(sc["obs"], dtype=torch.float32, device="cuda")
    pl.plan(sc["state"], sc["goal"], obs, N, T, sc["seed"], sc["t_index"])
    r = pl.result(N, T)["first_hit"].copy()
    pl.close()
    return r


@pytest.mark.parametrize("layout", ["one", "rows", "spread"])
@pytest.mark.parametrize("N", [200, 1500])
def test_first_collisions(layout, N):
    sc = inputs.tiny_scene(11, N=N, T=20, M=3000, width=16, box=90.0, clear=4.0)
    o = sc["obs"]
    if layout == "one":
        o[:, :2] = sc["state"][:2] + np.array([6.0, 0.3])
        o[:, 2:] = 0.0
    elif layout == "rows":
        # along lines through the grid: the first and last cells of rows
        o[:1500, 1] = sc["state"][1] + 5.0
        o[1500:, 0] = sc["state"][0] - 5.0
    got, want = _hits(sc, 5), _hits(sc, 2)
    assert np.array_equal(got, want)
    assert layout == "one" or np.count_nonzero(want >= 0) > 0
