"""The work that users of this library have it do, as cases that can be timed
and checked: plan steps of every network width over the range of samples,
horizons and obstacle points, the paper's hill climb, explicit parameters,
polygon footprints, a closed-loop mission, a batch of scenes, and the learned
proposal's training, evaluation and GEMM.  Each pass goes through the public
binding (paper_1904_06680_gb300.npp, .proposal); scenes come from the
library's seeded generators (paper_1904_06680_gb300.inputs).

`exact` restates the paths in 64-bit torch from the paper's equations and the
sampler's published definition, without the library's code.
"""
import math

import numpy as np
import torch

from paper_1904_06680_gb300 import inputs, npp, proposal

DEV = "cuda"


# ------------------------------------------------------------------ cases
def listed():
    return [
        # one small planning instance (the library's single-scene setting):
        # a call whose latency and launches count
        dict(name="plan_small", kind="plan", scene="single", width=16, N=256, T=20, M=200),
        # the forward/reverse waypoint course: the ordinary sampling time
        dict(name="plan_course", kind="plan", scene="course", width=32, N=16384, T=40, M=2000),
        # the 80 x 80 m area with 8192 points: the largest single plan step
        dict(name="plan_large", kind="plan", scene="large", width=64, N=65536, T=100, M=8192),
        # the paper's Step 5: 15 hill-climb rounds of 20480 samples over
        # H = 200 steps on a road with 20 points
        dict(name="climb_road", kind="climb", width=16, N=20480, T=200, rounds=15),
        # a mixed plan step: half of the samples from a learned proposal
        dict(name="plan_mixed", kind="plan", scene="course", width=16, N=4096, T=40, M=2000, n_prop=2048),
        # explicit parameter vectors judged with every sample's records kept
        # (an odd number of them): analysis and tests of stored controllers
        dict(name="rollout_records", kind="rollout", width=32, K=5003, T=60, M=1111),
        # a car with a tow bar (two convex pieces) under speed limits
        dict(name="plan_footprint", kind="plan", scene="course", width=32, N=16384, T=40, M=2000, footprint=True,
             v_limits=True),
        # a road mission driven in closed loop: 40 sampling times
        dict(name="mission", kind="mission", width=32, N=8192, T=40, steps=40),
        # uneven reverse-parking scenes of all three widths planned at once
        dict(name="batch", kind="batch", scenes=48, sizes=0),
        # the proposal's training at the benchmark's batch: 16 steps, then
        # the weights and gradients are read
        dict(name="train", kind="train", batch=8192, steps=16),
        # scenes encoded and evaluated by a proposal of the recipe's batch
        # (1024), fewer scenes than the batch
        dict(name="evaluate", kind="evaluate", batch=1024, scenes=300),
        # the BF16 tensor-core GEMM on its own
        dict(name="gemm", kind="gemm", M=8192, N=8192, K=8192),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A further case: the kinds of `listed`, sizes log-uniform over their
    ranges, odd ones among them."""
    kind = rng.choice(["plan", "plan", "plan", "climb", "rollout", "mission", "batch", "train", "evaluate", "gemm"])
    if kind == "plan":
        width = rng.choice([16, 32, 64])
        scene = rng.choice(["single", "course", "large"])
        c = dict(kind=kind, scene=scene, width=width, N=_log_int(rng, 200, 65536 if width < 64 else 50000),
                 T=rng.randint(10, 100), M=_log_int(rng, *{"single": (1, 600), "course": (100, 4000),
                                                           "large": (600, 8192)}[scene]))
        extra = rng.choice(["", "", "", "v_limits", "body_frame", "footprint", "n_prop"])
        if extra == "n_prop":
            c["n_prop"] = rng.randint(1, c["N"])
        elif extra:
            c[extra] = True
        return c
    if kind == "climb":
        return dict(kind=kind, width=rng.choice([16, 32]), N=_log_int(rng, 1000, 20480), T=rng.randint(40, 150),
                    rounds=rng.randint(2, 10))
    if kind == "rollout":
        return dict(kind=kind, width=rng.choice([16, 32, 64]), K=_log_int(rng, 1, 16000), T=rng.randint(10, 100),
                    M=_log_int(rng, 1, 4000))
    if kind == "mission":
        return dict(kind=kind, width=rng.choice([16, 32, 64]), N=_log_int(rng, 1000, 12000), T=rng.randint(20, 60),
                    steps=rng.randint(5, 40))
    if kind == "batch":
        return dict(kind=kind, scenes=rng.randint(2, 24), sizes=rng.randint(1, 1000))
    if kind == "train":
        return dict(kind=kind, batch=128 * _log_int(rng, 1, 60), steps=rng.randint(4, 16))
    if kind == "evaluate":
        batch = 128 * _log_int(rng, 1, 64)
        return dict(kind=kind, batch=batch, scenes=rng.randint(1, min(batch, 2048)))
    return dict(kind=kind, M=128 * _log_int(rng, 1, 60), N=128 * _log_int(rng, 1, 60), K=64 * _log_int(rng, 1, 120))


# ------------------------------------------------------------------ inputs
def _course(seed, N, T, width, M):
    n_wall, n_island = M // 2, M // 4
    return inputs.scene_course(seed, N=N, T=T, width=width, n_wall=n_wall, n_island=n_island,
                               n_dyn=M - n_wall - n_island)


def _scene(case, seed):
    """The planning instance of a case: a scene of the library's generators
    with the case's sizes and options."""
    N, T, width = case.get("N", case.get("K")), case["T"], case["width"]
    kind = case.get("scene", "road" if case["kind"] == "climb" else "course")
    if kind == "single":
        sc = inputs.scene_single(seed, N=N, T=T, M=case["M"], width=width)
    elif kind == "course":
        sc = _course(seed, N, T, width, case["M"])
    elif kind == "large":
        sc = inputs.scene_large(seed, N=N, T=T, width=width, M=case["M"])
    else:
        sc = inputs.scene_paper_road(True, seed, N=N, T=T)
        sc["preset"] = dict(sc["preset"], widths=(8, width, width, 2))
        rng = np.random.default_rng(seed)
        sc["state"][:4] += rng.uniform(-1, 1, 4) * [0.5, 0.3, 0.02, 1.0]
        sc["obs"][:, :2] += rng.uniform(-0.2, 0.2, (len(sc["obs"]), 2))
    sc["preset"] = dict(sc["preset"])
    if case.get("body_frame"):
        sc["preset"]["feature_frame"] = 1
    if case.get("v_limits"):
        sc["preset"].update(v_limits=1, v_min=-3.0, v_max=6.0)
    if case.get("footprint"):
        sc["preset"]["footprint"] = inputs.CAR_FOOTPRINT
    sc["t_index"] = seed % 1000
    return sc


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _proposal_of(case, seed, n_theta):
    """Mean and standard deviation of a sampling proposal, as the trained
    network gives them: a basis with scene-dependent shifts, std about 0.3."""
    g = _gen(seed + 17)
    mean = torch.randn(n_theta, generator=g, device=DEV)
    std = 0.3 * torch.exp(0.2 * torch.randn(n_theta, generator=g, device=DEV))
    return mean, std


def _theta(case, seed):
    return torch.randn(case["K"], 12 * case["width"] + case["width"] ** 2 + 2, generator=_gen(seed + 29), device=DEV)


def _net_params(seed):
    """Parameters of a proposal network in the middle of its training, in
    the library's packed order."""
    rng = np.random.default_rng(seed)
    H, I, O = 256, proposal.N_IN, 2 * proposal.N_THETA
    b3 = np.concatenate([rng.standard_normal(O // 2), np.full(O // 2, math.log(0.3))])
    parts = [rng.standard_normal((H, I)) * math.sqrt(2.0 / I), 0.05 * rng.standard_normal(H),
             rng.standard_normal((H, H)) * math.sqrt(2.0 / H), 0.05 * rng.standard_normal(H),
             rng.standard_normal((O, H)) * 0.3 * math.sqrt(1.0 / H), b3]
    return np.concatenate([p.ravel() for p in parts]).astype(np.float32)


def _pairs(case, seed):
    """Training pairs: encodings in [0, 1) with the 8 inputs in [-1, 1], and
    parameters around a basis."""
    g = _gen(seed + 5)
    n = case["batch"] * min(case["steps"], 4)
    x = torch.rand(n, proposal.N_IN, generator=g, device=DEV)
    x[:, 64:] = 2 * x[:, 64:] - 1
    base = torch.randn(1, proposal.N_THETA, generator=g, device=DEV)
    return x, base + 0.4 * torch.randn(n, proposal.N_THETA, generator=g, device=DEV)


def _gemm_operands(case, seed):
    g = _gen(seed)
    A = torch.randn(case["M"], case["K"], generator=g, device=DEV).to(torch.bfloat16)
    B = torch.randn(case["N"], case["K"], generator=g, device=DEV).to(torch.bfloat16)
    return A, B


def _points(obs):
    return torch.tensor(np.asarray(obs), dtype=torch.float32, device=DEV)


def _batch_scenes(case, seed):
    """Scenes whose sizes (N, T, M, widths) are the case's, with start
    states, points and sampler seeds of the seed's own."""
    b = inputs.scene_batch(case["sizes"], S=case["scenes"])
    rng = np.random.default_rng(seed)
    for sc in b["scenes"]:
        sc["state"][:4] += rng.uniform(-1, 1, 4) * [0.3, 0.3, 0.1, 0.5]
        sc["seed"] = inputs.philox_seed(int(rng.integers(0, 1 << 30)))
    b["obs"][:, :2] += rng.uniform(-0.05, 0.05, (len(b["obs"]), 2))
    return b


def _encode_scenes(case, seed):
    return inputs.scene_proposal_batch(seed, S=case["scenes"])


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind in ("plan", "climb", "rollout"):
        sc = _scene(case, seed)
        s.update(sc=sc, obs=_points(sc["obs"]))
        s["pl"] = npp.Planner(sc["preset"], max_N=sc["N"], max_T=sc["T"], max_M=len(sc["obs"]))
        if case.get("n_prop"):
            s["mean"], s["std"] = _proposal_of(case, seed, s["pl"].n_theta)
        if kind == "rollout":
            K, T = case["K"], case["T"]
            s["theta"] = _theta(case, seed)
            s["costs"] = torch.zeros(K, dtype=torch.float32, device=DEV)
            s["first_hit"] = torch.zeros(K, dtype=torch.int32, device=DEV)
            s["traj"] = torch.zeros(T + 1, K, 4, dtype=torch.float32, device=DEV)
            s["ctrl"] = torch.zeros(T, K, 2, dtype=torch.float32, device=DEV)
    elif kind == "mission":
        sc = inputs.scene_mission(seed, N=case["N"], T=case["T"], width=case["width"])
        s.update(sc=sc, obs=_points(sc["obs"]))
        s["pl"] = npp.Planner(sc["preset"], max_N=sc["N"], max_T=sc["T"], max_M=len(sc["obs"]))
    elif kind == "batch":
        b = _batch_scenes(case, seed)
        s["obs"] = _points(b["obs"])
        S = case["scenes"]
        s["own"] = _Batch(b)
        off = npp.npp_batch_offsets(s["own"].B, S)
        s["out"] = dict(best=torch.zeros(S, 8, dtype=torch.int32, device=DEV),
                        params=torch.zeros(int(off[S, 0]), device=DEV),
                        controls=torch.zeros(int(off[S, 1]), 2, device=DEV),
                        trajectory=torch.zeros(int(off[S, 2]), 4, device=DEV),
                        costs=torch.zeros(int(off[S, 3]), device=DEV),
                        first_hit=torch.zeros(int(off[S, 3]), dtype=torch.int32, device=DEV))
        o = npp.npp_batch_outputs()
        for k, t in s["out"].items():
            setattr(o, k, t.data_ptr())
        s["o"] = o
    elif kind == "train":
        s["net"] = proposal.ProposalNet(batch=case["batch"])
        s["net"].set_params(_net_params(seed))
        s["x"], s["theta"] = _pairs(case, seed)
    elif kind == "evaluate":
        b = _encode_scenes(case, seed)
        s["pl"] = npp.Planner(b["preset"], max_N=32, max_T=40, max_M=1)
        s["obs"] = _points(b["obs"])
        s["scenes"] = npp.scenes_to_device(npp.make_scenes(b["scenes"]))
        s["net"] = proposal.ProposalNet(batch=case["batch"])
        s["net"].set_params(_net_params(seed))
        s["x"] = torch.empty(case["scenes"], proposal.N_IN, dtype=torch.float32, device=DEV)
    else:
        s["A"], s["B"] = _gemm_operands(case, seed)
        s["C"] = torch.empty(case["M"], case["N"], dtype=torch.float32, device=DEV)
    return s


class _Batch:
    """A batch and the planner it lives on, freed in that order."""

    def __init__(self, b):
        self.pl = npp.Planner(b["preset"], max_N=32, max_T=1, max_M=1)
        self.B = npp.npp_batch_create(self.pl.h, npp.make_scenes(b["scenes"]))

    def __del__(self):
        npp.npp_batch_destroy(self.B)
        self.pl.close()


# ------------------------------------------------------------------ passes
def _plan_outputs(pl, N, T):
    return dict(best=pl.best, params=pl.params, controls=pl.controls[:T], trajectory=pl.trajectory[:T + 1],
                costs=pl.costs[:N], first_hit=pl.first_hit[:N])


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "plan":
        sc, pl = s["sc"], s["pl"]
        if case.get("n_prop"):
            npp.npp_plan_step_proposal(pl.h, sc["state"], sc["goal"], s["obs"], s["obs"].shape[0], sc["N"], sc["T"],
                                       sc["seed"], sc["t_index"], None, s["mean"], s["std"], case["n_prop"],
                                       pl.outputs())
        else:
            pl.plan(sc["state"], sc["goal"], s["obs"], sc["N"], sc["T"], sc["seed"], sc["t_index"])
        return _plan_outputs(pl, sc["N"], sc["T"])
    if kind == "climb":
        sc, pl = s["sc"], s["pl"]
        npp.npp_plan_tshc(pl.h, sc["state"], sc["goal"], s["obs"], s["obs"].shape[0], sc["N"], sc["T"], sc["seed"],
                          sc["t_index"], None, case["rounds"], 0.1, pl.outputs())
        return _plan_outputs(pl, sc["N"], sc["T"])
    if kind == "rollout":
        sc = s["sc"]
        npp.npp_rollout_params(s["pl"].h, sc["state"], sc["goal"], s["obs"], s["obs"].shape[0], s["theta"], case["K"],
                               case["T"], s["costs"], s["first_hit"], s["traj"], s["ctrl"])
        return dict(costs=s["costs"], first_hit=s["first_hit"], traj=s["traj"], ctrl=s["ctrl"])
    if kind == "mission":
        # a loop is a mission: created, driven, its log read, destroyed
        sc, n = s["sc"], case["steps"]
        L = npp.npp_loop_create_mission(s["pl"].h, sc["state"], sc["ref"], sc["field"], sc["window"], True,
                                        inputs.EPS, s["obs"], s["obs"].shape[0], sc["N"], sc["T"], sc["seed"], n)
        npp.npp_loop_run(L, n)
        state, log = npp.npp_loop_read(L), npp.npp_loop_log(L, n)
        npp.npp_loop_destroy(L)
        return dict(log=log, state={k: v for k, v in state.items() if k != "reserved"})
    if kind == "batch":
        npp.npp_plan_batch(s["own"].B, s["obs"], s["o"])
        return s["out"]
    if kind == "train":
        net, b = s["net"], case["batch"]
        losses = []
        for k in range(case["steps"]):
            i = k % (s["x"].shape[0] // b) * b
            losses.append(net.train_step(s["x"][i:i + b], s["theta"][i:i + b], 1e-3).clone())
        return dict(loss=torch.cat(losses), params=net.params(), grads=net.grads())
    if kind == "evaluate":
        npp.npp_proposal_encode(s["pl"].h, s["scenes"], case["scenes"], s["obs"], s["x"])
        mean, std = s["net"].forward(s["x"])
        return dict(x=s["x"], mean=mean, std=std)
    npp.npp_gemm_bf16(s["A"], s["B"], s["C"], case["M"], case["N"], case["K"])
    return s["C"]


# ------------------------------------------------------------------ work
def _rollout_flops(width, samples, steps, drawn=True):
    """The 8-W-W-2 network's products of `steps` control steps, and about 20
    operations per sampled parameter."""
    n_theta = 12 * width + width * width + 2
    return 2.0 * (width * width + 10 * width) * steps + (20.0 * samples * n_theta if drawn else 0.0)


# share of the N T control steps that lie before a sample's first collision,
# as these scenes give it (a sample needs none after it); the drives' and the
# batch's are rounded down from theirs
LIVE = dict(single=0.95, course=0.7, large=0.55, road=0.57, mission=0.5, batch=0.5)


def work(case):
    kind = case["kind"]
    if kind in ("plan", "climb"):
        N, T, W = case["N"], case["T"], case["width"]
        r = case.get("rounds", 1)
        live = LIVE[case.get("scene", "road")]
        n_theta = 12 * W + W * W + 2
        return dict(bytes=16.0 * case.get("M", 20) + 8.0 * N + 4.0 * n_theta + 24.0 * T,
                    flops=r * _rollout_flops(W, N, live * N * T))
    if kind == "rollout":
        K, T, W = case["K"], case["T"], case["width"]
        n_theta = 12 * W + W * W + 2
        return dict(bytes=K * (4.0 * n_theta + 8 + 16 * (T + 1) + 8 * T) + 16.0 * case["M"],
                    flops=_rollout_flops(W, K, K * T, drawn=False))
    if kind == "mission":
        N, T, W = case["N"], case["T"], case["width"]
        return dict(bytes=case["steps"] * (16.0 * 855 + 8.0 * N),
                    flops=case["steps"] * _rollout_flops(W, N, LIVE["mission"] * N * T))
    if kind == "batch":
        # means of the generator's ranges: N log-uniform in 1024..65536, T
        # uniform in 20..80, M log-uniform in 100..20000, the widths evenly
        S = case["scenes"]
        N, M = (65536 - 1024) / math.log(64), 19900 / math.log(200)
        return dict(bytes=S * (16.0 * M + 8.0 * N),
                    flops=S * sum(_rollout_flops(w, N, LIVE["batch"] * N * 50) for w in (16, 32, 64)) / 3)
    H, I, O = 256, proposal.N_IN, 2 * proposal.N_THETA
    params = H * I + H * H + O * H
    if kind == "train":
        b, k = case["batch"], case["steps"]
        return dict(bytes=k * (4.0 * b * (I + proposal.N_THETA) + 24.0 * params),
                    flops=k * 2.0 * b * (2 * H * I + 3 * H * H + 3 * O * H))
    if kind == "evaluate":
        n = case["scenes"]
        return dict(bytes=4.0 * n * (I + O) + 4.0 * params + 16.0 * 2000 * min(n, 16),
                    flops=2.0 * n * params + 30.0 * 2000 * n)
    M, N, K = case["M"], case["N"], case["K"]
    return dict(bytes=2.0 * (M * K + N * K) + 4.0 * M * N, flops=2.0 * M * N * K)


# ------------------------------------------------------------------ exact
def _philox(n, i, t_index, stream, seed):
    """The four words of Philox4x32-10 (Salmon et al., SC'11) at counter
    (i, n, t_index, stream), key = seed; n [N, 1], i [1, Q] int64 tensors."""
    m32 = 0xFFFFFFFF
    c0, c1 = torch.broadcast_tensors(i, n)
    c2, c3 = torch.full_like(c0, t_index), torch.full_like(c0, stream)
    k0, k1 = seed & m32, (seed >> 32) & m32
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
        p0, p1 = 0xD2511F53 * c0, 0xCD9E8D57 * c2
        c0, c1, c2, c3 = ((p1 >> 32) & m32) ^ c1 ^ k0, p1 & m32, ((p0 >> 32) & m32) ^ c3 ^ k1, p0 & m32
    return c0, c1, c2, c3


def _normals(samples, n_theta, t_index, stream, seed):
    """theta [samples, n_theta] ~ N(0, 1) by Box-Muller on a 23-bit grid."""
    q = torch.arange((n_theta + 3) // 4, device=DEV)[None]
    w = _philox(samples[:, None], q, t_index, stream, seed)
    u = [(2.0 * (x >> 9).double() + 1.0) * 2.0 ** -24 for x in w]
    out = []
    for a, b in ((u[0], u[1]), (u[2], u[3])):
        r = torch.sqrt(-2.0 * torch.log(a))
        out += [r * torch.cos(2 * math.pi * b), r * torch.sin(2 * math.pi * b)]
    return torch.stack(out, -1).reshape(len(samples), -1)[:, :n_theta]


def _wrap(a):
    return a - 2 * math.pi * torch.floor((a + math.pi) / (2 * math.pi))


def _f32(v):
    return np.asarray(v, np.float32).astype(np.float64)


def _rollout64(sc, theta):
    """States [n, T+1, 4] (EV frame), controls [n, T, 2] and the cost without
    collisions of parameter rows theta (64 bits): the paper's features,
    network, rate limit and Euler bicycle, the library's cost."""
    p = {k: (float(np.float32(v)) if isinstance(v, float) else v) for k, v in sc["preset"].items()}
    T, W, n = sc["T"], p["widths"][1], len(theta)
    x0, y0, phi0, v0, a0, a1 = _f32(sc["state"])
    gx, gy, gphi, gv = _f32(sc["goal"])
    c0, s0 = math.cos(phi0), math.sin(phi0)
    g = (c0 * (gx - x0) + s0 * (gy - y0), -s0 * (gx - x0) + c0 * (gy - y0), gphi - phi0, gv)
    o, parts = 0, []
    for rows, cols in ((W, 8), (W, 1), (W, W), (W, 1), (2, W), (2, 1)):
        parts.append(theta[:, o:o + rows * cols].reshape(n, rows, cols))
        o += rows * cols
    W1, b1, W2, b2, W3, b3 = parts
    z = torch.zeros(n, 4, dtype=torch.float64, device=DEV)
    z[:, 3] = v0
    ap = torch.tensor([[a0, a1]], dtype=torch.float64, device=DEV).repeat(n, 1)
    E = torch.zeros(n, dtype=torch.float64, device=DEV)
    L = p["lf"] + p["lr"]
    rate = p["delta_rate_max"] * p["Ts"] / p["delta_max"]
    zs, us = [z], []
    for h in range(T):
        x, y, ph, v = z.unbind(1)
        dx, dy = g[0] - x, g[1] - y
        if p.get("feature_frame"):
            dx, dy = torch.cos(ph) * dx + torch.sin(ph) * dy, -torch.sin(ph) * dx + torch.cos(ph) * dy
        f = torch.stack([dx / p["dxi_n"], dy / p["deta_n"], _wrap(g[2] - ph) / p["dphi_n"], (g[3] - v) / p["dv_n"],
                         ap[:, 0], ap[:, 1], v / p["dv_n"], torch.full_like(x, (T - h) / T)], 1)[:, :, None]
        a = torch.tanh(b3 + W3 @ torch.tanh(b2 + W2 @ torch.tanh(b1 + W1 @ f)))[:, :, 0]
        st = torch.minimum(torch.maximum(a[:, 0], ap[:, 0] - rate), ap[:, 0] + rate).clamp(-1, 1)
        ap = torch.stack([st, a[:, 1]], 1)
        E = E + (ap * ap).sum(1)
        td = torch.tan(p["delta_max"] * st)
        tb = p["lr"] / L * td
        u = 0.5 * (p["u_min"] + p["u_max"]) + 0.5 * (p["u_max"] - p["u_min"]) * a[:, 1]
        z = torch.stack([x + p["Ts"] * v * (torch.cos(ph) - torch.sin(ph) * tb),
                         y + p["Ts"] * v * (torch.sin(ph) + torch.cos(ph) * tb),
                         ph + p["Ts"] * v * td / L, v + p["Ts"] * u], 1)
        zs.append(z)
        us.append(ap)
    x, y, ph, v = z.unbind(1)
    J = p["w_pos"] * torch.hypot(x - g[0], y - g[1]) + p["w_phi"] * _wrap(ph - g[2]).abs() \
        + p["w_v"] * (v - g[3]).abs() + p["w_effort"] * E / T
    return torch.stack(zs, 1), torch.stack(us, 1), J


def _collides(sc, z, tau):
    """Whether some obstacle point lies inside the vehicle at states z
    [n, 4], tau seconds ahead."""
    p = sc["preset"]
    x0, y0, phi0 = _f32(sc["state"])[:3]
    o = torch.from_numpy(_f32(sc["obs"])).to(DEV)
    c0, s0 = math.cos(phi0), math.sin(phi0)
    wx, wy = o[:, 0] + tau * o[:, 2] - x0, o[:, 1] + tau * o[:, 3] - y0
    px, py = c0 * wx + s0 * wy, -s0 * wx + c0 * wy
    hit = []
    for part in z.split(max(1, (1 << 25) // max(1, len(o)))):
        x, y, ph = part[:, 0, None], part[:, 1, None], part[:, 2, None]
        dx, dy, c, s = px - x, py - y, torch.cos(ph), torch.sin(ph)
        qx, qy = c * dx + s * dy, -s * dx + c * dy
        if p.get("footprint"):
            inside = torch.zeros_like(qx, dtype=torch.bool)
            for piece in p["footprint"]:
                v = _f32(piece)
                ok = torch.ones_like(inside)
                for a, b in zip(v, np.roll(v, -1, 0)):
                    ok &= (b[0] - a[0]) * (qy - a[1]) - (b[1] - a[1]) * (qx - a[0]) > 0
                inside |= ok
        else:
            inside = ((qx - p["c_off"]).abs() < p["half_len"]) & (qy.abs() < p["half_wid"])
        hit.append(inside.any(1))
    return torch.cat(hit)


def _judge64(sc, theta):
    """Costs (inf where a state collides or leaves the speed limits), states
    and controls of parameter rows theta."""
    z, u, J = _rollout64(sc, theta)
    free = torch.ones(len(theta), dtype=torch.bool, device=DEV)
    p = sc["preset"]
    for h in range(sc["T"] + 1):
        k = free.nonzero()[:, 0]
        if len(sc["obs"]) and len(k):
            free[k[_collides(sc, z[k, h], h * p["Ts"])]] = False
        if p.get("v_limits") and h:
            free &= (z[:, h, 3] >= p["v_min"]) & (z[:, h, 3] <= p["v_max"])
    return torch.where(free, J, torch.inf), z, u


def _train64(case, seed):
    """The training steps in 64 bits: Gaussian negative log-likelihood, Adam."""
    v = torch.from_numpy(_net_params(seed)).to(DEV).double()
    H, I, O = 256, proposal.N_IN, 2 * proposal.N_THETA
    x, th = (t.double() for t in _pairs(case, seed))
    m, s = torch.zeros_like(v), torch.zeros_like(v)
    b, losses = case["batch"], []
    for k in range(case["steps"]):
        i = k % (x.shape[0] // b) * b
        v.requires_grad_(True)
        mean, ls = _net64(v, x[i:i + b])
        loss = (ls + 0.5 * (th[i:i + b] - mean) ** 2 * torch.exp(-2 * ls)).mean()
        g, = torch.autograd.grad(loss, v)
        losses.append(loss.detach())
        v = v.detach()
        m, s = 0.9 * m + 0.1 * g, 0.999 * s + 0.001 * g * g
        v = v - 1e-3 * (m / (1 - 0.9 ** (k + 1))) / (torch.sqrt(s / (1 - 0.999 ** (k + 1))) + 1e-8)
    return dict(loss=torch.stack(losses), params=v, grads=g)


def _net64(v, x):
    H, I, O = 256, proposal.N_IN, 2 * proposal.N_THETA
    W1, b1, W2, b2, W3, b3 = torch.split(v, [H * I, H, H * H, H, O * H, O])
    h = torch.relu(x @ W1.reshape(H, I).T + b1)
    h = torch.relu(h @ W2.reshape(H, H).T + b2)
    y = h @ W3.reshape(O, H).T + b3
    return y[:, :O // 2], y[:, O // 2:].clamp(-3.0, 1.0)


def _encode64(case, seed):
    b = _encode_scenes(case, seed)
    obs = torch.from_numpy(_f32(b["obs"])).to(DEV)
    p, rows = b["preset"], []
    for sc in b["scenes"]:
        x0, y0, phi0, v0, a0, a1 = _f32(sc["state"])
        gx, gy, gphi, gv = _f32(sc["goal"])
        c, s = math.cos(phi0), math.sin(phi0)
        o = obs[sc["obs_offset"]:sc["obs_offset"] + sc["M"]]
        dx, dy = o[:, 0] - x0, o[:, 1] - y0
        px, py = c * dx + s * dy, -s * dx + c * dy
        w = (1 - torch.hypot(px, py) / 20.0).clamp(min=0)
        k = ((torch.atan2(py, px) + math.pi) * (64 / (2 * math.pi))).floor().long().clamp(0, 63)
        h = torch.zeros(64, dtype=torch.float64, device=DEV).index_add_(0, k, w)
        d = gphi - phi0
        d -= 2 * math.pi * math.floor((d + math.pi) / (2 * math.pi))
        rest = [(c * (gx - x0) + s * (gy - y0)) / p["dxi_n"], (-s * (gx - x0) + c * (gy - y0)) / p["deta_n"],
                d / p["dphi_n"], (gv - v0) / p["dv_n"], a0, a1, v0 / p["dv_n"], 1.0]
        rows.append(torch.cat([h / (1 + h), torch.tensor(rest, dtype=torch.float64, device=DEV)]))
    return torch.stack(rows)


def exact(case, seed):
    kind = case["kind"]
    if kind == "plan":
        # the costs of all samples; the winner's outputs hang on which of
        # them is the least
        sc = _scene(case, seed)
        N, W = sc["N"], case["width"]
        n_theta = 12 * W + W * W + 2
        costs = []
        for part in torch.arange(N, device=DEV).split(max(1, (1 << 25) // n_theta)):
            theta = _normals(part, n_theta, sc["t_index"], 0, sc["seed"])
            if case.get("n_prop"):
                mean, std = (t.double() for t in _proposal_of(case, seed, n_theta))
                own = mean + std * _normals(part, n_theta, sc["t_index"], 1, sc["seed"])
                theta = torch.where((part < case["n_prop"])[:, None], own, theta)
            costs.append(_judge64(sc, theta)[0])
        return dict(best=None, params=None, controls=None, trajectory=None, costs=torch.cat(costs), first_hit=None)
    if kind == "rollout":
        sc = _scene(case, seed)
        costs, z, u = _judge64(sc, _theta(case, seed).double())
        return dict(costs=costs, first_hit=None, traj=z.transpose(0, 1).contiguous(),
                    ctrl=u.transpose(0, 1).contiguous())
    if kind == "train":
        return _train64(case, seed)
    if kind == "evaluate":
        x = _encode64(case, seed)
        mean, ls = _net64(torch.from_numpy(_net_params(seed)).to(DEV).double(), x)
        return dict(x=x, mean=mean, std=torch.exp(ls))
    if kind == "gemm":
        A, B = _gemm_operands(case, seed)
        return A.double() @ B.double().T
    # the hill climb, the mission and the batch chain winners or hold
    # dozens of scenes: no value of their own in 64 bits
    return None
