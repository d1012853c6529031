"""Launches of the same kernels with different shared-memory sizes: threads
that plan at the same time on handles of their own, with few and with many
points, and batches that live side by side.  Every call succeeds, and every
result is the one the call gets alone."""
import threading

import numpy as np
import pytest
import torch

from paper_1904_06680_gb300 import inputs, npp

pytestmark = pytest.mark.gpu


def _same(a, b):
    return all(np.array_equal(np.asarray(a[k]).view(np.uint32), np.asarray(b[k]).view(np.uint32))
               for k in ("costs", "first_hit", "params", "controls", "trajectory"))


def _plan_in_threads(scenes, options, rounds=400, calls=6):
    """Hill climbs of many rounds (so that the threads spend their time in
    the library, launching) on each scene, alone and then at once."""
    planners = []
    for sc in scenes:
        pl = npp.Planner(sc["preset"], max_N=sc["N"], max_T=sc["T"], max_M=len(sc["obs"]))
        for name, value in options.items():
            npp.npp_set_option(pl.h, name, value)
        planners.append((sc, pl, torch.tensor(sc["obs"], dtype=torch.float32, device="cuda"), torch.cuda.Stream()))

    def climb(sc, pl, obs, stream):
        npp.npp_plan_tshc(pl.h, sc["state"], sc["goal"], obs, obs.shape[0], sc["N"], sc["T"], sc["seed"],
                          sc["t_index"], None, rounds, 0.1, pl.outputs(), stream)
        stream.synchronize()

    alone = []
    torch.cuda.synchronize()
    for p in planners:
        climb(*p)
        alone.append(p[1].result(p[0]["N"], p[0]["T"]))
    start, errors = threading.Barrier(len(planners)), []

    def work(p):
        start.wait()
        try:
            for _ in range(calls):
                climb(*p)
        except Exception as e:
            errors.append(e)

    threads = [threading.Thread(target=work, args=(p,)) for p in planners]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for (sc, pl, _, _), want in zip(planners, alone):
        assert _same(pl.result(sc["N"], sc["T"]), want), len(sc["obs"])
        pl.close()


def test_grid_check():
    """The automatic check of 1024 samples and more, 33 to 100 KB a block."""
    _plan_in_threads([inputs.tiny_scene(80 + i, N=1024, T=2, M=M, box=25.0)
                      for i, M in enumerate((200, 8702, 3000, 5001))], {})


@pytest.mark.parametrize("variant", range(5))
def test_brute_force_checks(variant):
    """64 to 208 KB a block."""
    _plan_in_threads([inputs.tiny_scene(85 + i, N=64, T=2, M=M, box=25.0) for i, M in enumerate((4000, 13000, 6000, 9001))],
                     {"collide_variant": variant})


def test_batches_side_by_side():
    """A brute-force batch planned after another one's set-up (80 and 144 KB)."""
    big, small = (inputs.tiny_scene(90 + i, N=200, T=3, M=M, box=25.0) for i, M in enumerate((9000, 5000)))
    pl = npp.Planner(big["preset"], max_N=200, max_T=3, max_M=9000)
    obs = torch.tensor(big["obs"], dtype=torch.float32, device="cuda")
    pl.plan(big["state"], big["goal"], obs, 200, 3, big["seed"], big["t_index"])
    want = pl.result(200, 3)
    batches = []
    for sc in (big, small):
        B = npp.npp_batch_create(pl.h, npp.make_scenes([dict(
            state=sc["state"], goal=sc["goal"], N=200, T=3, M=len(sc["obs"]), width=16, obs_offset=0, seed=sc["seed"],
            t_index=sc["t_index"])]))
        npp.npp_batch_set_option(B, "collide", 0)
        batches.append(B)
    best = torch.zeros(8, dtype=torch.int32, device="cuda")
    costs, fh = torch.zeros(200, device="cuda"), torch.zeros(200, dtype=torch.int32, device="cuda")
    out = npp.npp_batch_outputs()
    out.best, out.costs, out.first_hit = best.data_ptr(), costs.data_ptr(), fh.data_ptr()
    npp.npp_plan_batch(batches[0], obs, out)
    torch.cuda.synchronize()
    assert np.array_equal(fh.cpu().numpy(), want["first_hit"])
    assert np.array_equal(costs.cpu().numpy().view(np.uint32), want["costs"].view(np.uint32))
    for B in batches:
        npp.npp_batch_destroy(B)
    pl.close()
