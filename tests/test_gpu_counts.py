"""Work counters of timed plan steps and loops: the same from run to run,
the states up to each sample's first collision where the check takes a step's
samples together, the candidates that the warp-per-sample check tests where
nothing collides, and zero after a step with another check."""
import numpy as np
import pytest
import torch

from paper_1904_06680_gb300 import inputs, npp

pytestmark = pytest.mark.gpu


def _planner(sc, **options):
    pl = npp.Planner(sc["preset"], max_N=sc["N"], max_T=sc["T"], max_M=len(sc["obs"]))
    npp.npp_set_timing(pl.h, True)
    for name, value in options.items():
        npp.npp_set_option(pl.h, name, value)
    return pl


def _plan(pl, sc, M=None):
    obs = torch.tensor(sc["obs"][:M], dtype=torch.float32, device="cuda")
    pl.plan(sc["state"], sc["goal"], obs, sc["N"], sc["T"], sc["seed"], sc["t_index"])
    return npp.npp_last_counts(pl.h), pl.result(sc["N"], sc["T"])["first_hit"]


@pytest.mark.parametrize("N,T,M", [(1024, 12, 300), (3001, 40, 801), (16384, 40, 2000)])
def test_same_from_run_to_run(N, T, M):
    sc = inputs.tiny_scene(N + T, N=N, T=T, M=M, box=14.0)
    pl = _planner(sc)
    (tests, states, steps), fh = _plan(pl, sc)
    assert states == np.where(fh < 0, T + 1, fh + 1).sum()
    assert steps == N * T and tests > 0 and len(np.unique(fh)) > 1
    for _ in range(4):
        assert _plan(pl, sc)[0] == (tests, states, steps)
    pl.close()


def test_candidates_of_the_warp_per_sample_check():
    """Without collisions every state is checked by both (in two chunks the
    state between them once): points beyond the rectangle's corners, a vehicle
    that moves 3 cm."""
    sc = inputs.tiny_scene(7, N=2000, T=2, M=4000, box=4.0, clear=2.5, vmax=0.0)
    sc["state"][3] = 0.0
    pl, ch = _planner(sc, chunks=1), _planner(sc, chunks=2)
    (a, fa), (b, fb) = _plan(pl, sc), _plan(ch, sc)
    assert np.all(fa == -1) and np.all(fb == -1)
    assert a == b and a[0] > 0 and a[1] == 2000 * 3
    pl.close()
    ch.close()


@pytest.mark.parametrize("options", [{"collide_variant": 2}, {}])
def test_zero_after_another_check(options):
    sc = inputs.tiny_scene(8, N=2000, T=20, M=400, box=14.0)
    pl = _planner(sc)
    assert _plan(pl, sc)[0][1] > 0
    for name, value in options.items():
        npp.npp_set_option(pl.h, name, value)
    assert _plan(pl, sc, 140)[0] == (0, 0, 0)
    pl.close()


@pytest.mark.parametrize("rounds", [1, 3])
def test_loop(rounds):
    """A loop's counters are its first round's: at the first sampling time,
    those of the plan step."""
    sc = inputs.tiny_scene(9, N=2000, T=20, M=400, box=14.0)
    sc["t_index"] = 0
    pl = _planner(sc)
    want = _plan(pl, sc)[0]
    if rounds > 1:
        npp.npp_set_loop_restarts(pl.h, rounds, 0.1)
    obs = torch.tensor(sc["obs"], dtype=torch.float32, device="cuda")
    L = npp.npp_loop_create(pl.h, sc["state"], sc["goal"][None], inputs.EPS, obs, len(sc["obs"]), sc["N"], sc["T"],
                            sc["seed"], max_log=1)
    npp.npp_loop_run(L, 1)
    assert npp.npp_last_counts(pl.h) == want
    npp.npp_loop_destroy(L)
    pl.close()
