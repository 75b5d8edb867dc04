"""Goals kept across the steps of a rollout: every scenario type through
switches, Bezier segments and auto-resets equals per-call steps (which evaluate
each goal from its record), in the warp-specialised rollout, whose noise side
evaluates the goals, and in the persistent one."""
import pytest
import torch

from gpu_helpers import DEV
from paper_2306_09537_gb300 import qs
from paper_2306_09537_gb300.env import QuadSwarmEnv

pytestmark = pytest.mark.gpu
FEATS = ("floor", "walls", "motor_noise", "obs_noise", "dr", "collisions", "downwash", "auto_reset")


@pytest.mark.parametrize("n,E", [(1, 70), (2, 33), (7, 21), (32, 5), (50, 4)])
@pytest.mark.parametrize("shape", [(1, 0), (1, 7), (128, 0), (64, 9)])
def test_rollout_goals_equal_steps(n, E, shape):
    T, K = 40, min(6, n - 1)
    kw = dict(seed=8, device=DEV, scenarios=qs.SCENARIOS, episode_steps=13, bez_seg=3.0, se_period=5.0)
    a, b = (QuadSwarmEnv(E, n, K, FEATS, **kw) for _ in range(2))
    qs.qs_set_rollout_shape(a.h, shape[0], shape[1], False)
    acts = torch.rand(T, a.D, 4, generator=torch.Generator(device=DEV).manual_seed(2), device=DEV)
    obs, rew = torch.empty(T, a.D, a.obs_dim, device=DEV), torch.empty(T, a.D, device=DEV)
    a.rollout(acts, obs, rew, None)
    for t in range(T):
        o, r, _ = b.step(acts[t])
        assert torch.equal(obs[t], o) and torch.equal(rew[t], r), t
    assert torch.equal(a.get_goals(), b.get_goals())
