"""Points advanced in the vehicle's launch (up to 4096) or in their own:
the same loop, bit for bit, when a point too far away to matter takes the
count over the line, and without points."""
import numpy as np
import pytest
import torch

from paper_1904_06680_gb300 import inputs, npp

pytestmark = pytest.mark.gpu


def _run(sc, obs, steps):
    M = len(obs)
    pl = npp.Planner(sc["preset"], max_N=sc["N"], max_T=sc["T"], max_M=max(M, 1))
    npp.npp_set_option(pl.h, "collide_variant", 5)
    o = torch.tensor(obs, dtype=torch.float32, device="cuda") if M else None
    L = npp.npp_loop_create(pl.h, sc["state"], [sc["goal"]], inputs.EPS, o, M, sc["N"], sc["T"], sc["seed"])
    npp.npp_loop_run(L, steps)
    log, st = npp.npp_loop_log(L), npp.npp_loop_read(L)
    npp.npp_loop_destroy(L)
    pl.close()
    return np.asarray(log), st


@pytest.mark.parametrize("M", [1, 2, 1023, 1025, 4095, 4096])
def test_same_loop(M):
    sc = inputs.tiny_scene(M, N=600, T=12, M=M, width=16, box=30.0, dyn_frac=0.7, clear=5.0)
    far = np.tile([[9.0e3, 9.0e3, 0.0, 0.0]], (4097 - M, 1))
    a, sa = _run(sc, sc["obs"], 5)
    b, sb = _run(sc, np.concatenate([sc["obs"], far]), 5)
    assert np.array_equal(a, b)
    assert all(sa[k] == sb[k] for k in ("x", "y", "phi", "v", "t"))
