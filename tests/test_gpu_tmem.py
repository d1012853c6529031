"""The trajectory kernels that keep layer-2 weights in tensor memory against
the ones that keep them in registers (launch shapes 0, 1, 2 against 3): every
output the same bits, at sample counts on both sides of the launch rules and
of blocks, warps and lane groups, with and without the rollout variants, with
a sampling proposal, a warm start and explicit parameters."""
import numpy as np
import pytest

from paper_1904_06680_gb300 import inputs, npp

pytestmark = pytest.mark.gpu

VARIANTS = dict(plain={}, limits=dict(v_limits=1, v_min=-2.0, v_max=3.0), body=dict(feature_frame=1))


def _bits(r):
    return {k: np.ascontiguousarray(v).view(np.uint32) for k, v in r.items() if isinstance(v, np.ndarray)}


def _plan(sc, shape, fuse, records, n_prop=0, warm=False):
    import torch
    N, T, M = sc["N"], sc["T"], len(sc["obs"])
    pl = npp.Planner(sc["preset"], max_N=N, max_T=T, max_M=M, record_samples=records)
    npp.npp_set_option(pl.h, "traj_variant", shape)
    npp.npp_set_option(pl.h, "fuse", fuse)
    obs = torch.tensor(sc["obs"], dtype=torch.float32, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(1)
    vec = torch.randn(3, pl.n_theta, generator=g, device="cuda")
    w = vec[2].contiguous() if warm else None
    if n_prop:
        npp.npp_plan_step_proposal(pl.h, sc["state"], sc["goal"], obs, M, N, T, sc["seed"], sc["t_index"], w,
                                   vec[0].contiguous(), (0.3 * vec[1].abs()).contiguous(), n_prop, pl.outputs())
    else:
        pl.plan(sc["state"], sc["goal"], obs, N, T, sc["seed"], sc["t_index"], warm=w)
    r = pl.result(N, T)
    pl.close()
    return r


@pytest.mark.parametrize("variant", sorted(VARIANTS))
@pytest.mark.parametrize("width,N,T", [(16, 1, 1), (16, 33, 9), (16, 2128, 5), (16, 2129, 5), (32, 17, 9),
                                       (32, 1064, 4), (32, 1081, 4), (64, 7, 9), (64, 2431, 13), (64, 2433, 13),
                                       (64, 16383, 3), (64, 16389, 3)])
def test_shapes_equal_registers(width, N, T, variant):
    sc = inputs.tiny_scene(N + width, N=N, T=T, M=300, width=width, box=15.0)
    sc["preset"] = dict(sc["preset"], **VARIANTS[variant])
    for fuse in ((0, 1) if width == 64 else (0,)):
        want = _bits(_plan(sc, 3, fuse, fuse == 0))
        for shape in (0, 1, 2):
            got = _bits(_plan(sc, shape, fuse, fuse == 0))
            assert got.keys() == want.keys()
            for k in want:
                assert np.array_equal(got[k], want[k]), (shape, fuse, k)


@pytest.mark.parametrize("width", [16, 32, 64])
def test_proposal_and_warm_start(width):
    sc = inputs.tiny_scene(5, N=401, T=11, M=300, width=width, box=15.0)
    for n_prop, warm in ((0, True), (150, False), (401, True)):
        want = _bits(_plan(sc, 3, -1, False, n_prop, warm))
        for shape in (0, 1, 2):
            got = _bits(_plan(sc, shape, -1, False, n_prop, warm))
            for k in want:
                assert np.array_equal(got[k], want[k]), (shape, n_prop, k)


@pytest.mark.parametrize("width,K", [(16, 37), (32, 5), (64, 3)])
def test_explicit_parameters(width, K):
    """rows of explicit parameters start at any 4-byte boundary"""
    import torch
    sc = inputs.tiny_scene(9, N=K, T=12, M=40, width=width)
    nt = 12 * width + width * width + 2
    buf = torch.randn(K * nt + 3, generator=torch.Generator().manual_seed(2)).cuda()
    out = []
    for shape in (3, 0, 1, 2):
        for shift in (0, 1):
            pl = npp.Planner(sc["preset"], max_N=K, max_T=12, max_M=40)
            npp.npp_set_option(pl.h, "traj_variant", shape)
            theta = buf[shift:shift + K * nt]
            theta.copy_(buf[:K * nt].clone()) if shift else None
            costs = torch.zeros(K, device="cuda")
            fh = torch.zeros(K, dtype=torch.int32, device="cuda")
            tr, ct = torch.zeros(13, K, 4, device="cuda"), torch.zeros(12, K, 2, device="cuda")
            obs = torch.tensor(sc["obs"], dtype=torch.float32, device="cuda")
            npp.npp_rollout_params(pl.h, sc["state"], sc["goal"], obs, 40, theta, K, 12, costs, fh, tr, ct)
            out.append([x.cpu().numpy().view(np.uint32) for x in (costs, fh, tr, ct)])
            if shift:
                buf[:K * nt].copy_(theta.clone())
            pl.close()
    for o in out[1:]:
        for a, b in zip(o, out[0]):
            assert np.array_equal(a, b)
