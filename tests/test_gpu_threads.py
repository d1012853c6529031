"""Threads that plan at the same time on handles of their own, with few and
with many points (launches of different shared-memory sizes of the same
kernels): every call succeeds, and every thread's result is the one it gets
alone."""
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
