"""The plan-step tuner counts the library's own choice of a collision check
among its candidates, so a tuned planner is never left with a slower check than
an untuned one has; it applies the fastest and remembers it."""
import pytest
import torch

from paper_1904_06680_gb300 import autotune, inputs, npp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,N,T,M", [(16, 20480, 60, 20), (32, 4096, 40, 1000), (64, 3000, 30, 600)])
def test_own_choice_is_a_candidate(width, N, T, M):
    sc = inputs.tiny_scene(N + M, N=N, T=T, M=M, width=width, box=20.0)
    pl = npp.Planner(sc["preset"], max_N=N, max_T=T, max_M=M)
    obs = torch.tensor(sc["obs"], dtype=torch.float32, device="cuda")
    for _ in range(2):                    # measured, then from the cache
        best, ms = autotune.tune_plan_step(pl, sc["state"], sc["goal"], obs, N, T, sc["seed"])
        assert sorted(ms) == sorted(str(v) for v in (-1, 0, 1, 2, 3, 4))
        assert ms[str(best)] == min(ms.values()) <= ms["-1"]
    pl.close()
