"""Batches whose trajectory queues hold more items than warps start with, at
each width: costs, first collisions and winners bit for bit those of a plan
step on the scene alone, for both block sizes, both checks, with speed limits
and with the stages one after another (timing on) or side by side."""
import numpy as np
import pytest
import torch

from paper_1904_06680_gb300 import inputs, npp

pytestmark = pytest.mark.gpu


def _single(sc):
    N, T, M = sc["N"], sc["T"], len(sc["obs"])
    pl = npp.Planner(sc["preset"], max_N=N, max_T=T, max_M=M)
    obs = torch.tensor(sc["obs"], dtype=torch.float32, device="cuda")
    pl.plan(sc["state"], sc["goal"], obs, N, T, sc["seed"], sc["t_index"])
    r = pl.result(N, T)
    pl.close()
    return r


@pytest.mark.parametrize("limits", [False, True])
def test_queues(limits):
    scs = []
    for i, (w, N, T) in enumerate([(64, 3101, 5), (16, 20003, 4), (32, 9803, 6), (64, 1, 9), (16, 7, 1), (32, 31, 3)]):
        sc = inputs.tiny_scene(70 + i, N=N, T=T, M=60 + i, width=w, box=12.0)
        if limits:
            sc["preset"] = dict(sc["preset"], v_limits=1, v_min=-2.0, v_max=3.0)
        scs.append(sc)
    want = [_single(sc) for sc in scs]
    offs = np.cumsum([0] + [len(sc["obs"]) for sc in scs])
    descs = [dict(state=sc["state"], goal=sc["goal"], N=sc["N"], T=sc["T"], M=len(sc["obs"]),
                  width=sc["preset"]["widths"][1], obs_offset=int(offs[i]), seed=sc["seed"],
                  t_index=sc["t_index"]) for i, sc in enumerate(scs)]
    obs = torch.tensor(np.concatenate([sc["obs"] for sc in scs]), dtype=torch.float32, device="cuda")
    pl = npp.Planner(scs[0]["preset"], max_N=1, max_T=1, max_M=1)
    B = npp.npp_batch_create(pl.h, npp.make_scenes(descs))
    S = len(descs)
    off = npp.npp_batch_offsets(B, S)
    best = torch.zeros(S * 8, dtype=torch.int32, device="cuda")
    costs = torch.zeros(int(off[S, 3]), device="cuda")
    fh = torch.zeros(int(off[S, 3]), dtype=torch.int32, device="cuda")
    traj = torch.zeros(int(off[S, 2]) * 4, device="cuda")
    out = npp.npp_batch_outputs()
    out.best, out.costs, out.first_hit, out.trajectory = (x.data_ptr() for x in (best, costs, fh, traj))
    for warps, check, timing in ((8, 1, 0), (4, 1, 0), (8, 1, 1), (8, 0, 0), (4, 0, 1)):
        npp.npp_set_timing(pl.h, bool(timing))
        npp.npp_batch_set_option(B, "traj_warps", warps)
        npp.npp_batch_set_option(B, "collide", check)
        for x in (best, costs, fh, traj):
            x.fill_(-7)
        npp.npp_plan_batch(B, obs, out)
        torch.cuda.synchronize()
        for i, r in enumerate(want):
            a, b = int(off[i, 3]), int(off[i, 3]) + scs[i]["N"]
            what = (warps, check, timing, i)
            assert np.array_equal(fh[a:b].cpu().numpy(), r["first_hit"]), what
            assert np.array_equal(costs[a:b].cpu().numpy().view(np.uint32), r["costs"].view(np.uint32)), what
            t = traj[4 * int(off[i, 2]):4 * int(off[i, 2]) + r["trajectory"].size].cpu().numpy()
            assert np.array_equal(t.view(np.uint32), r["trajectory"].ravel().view(np.uint32)), what
    npp.npp_batch_destroy(B)
    pl.close()
