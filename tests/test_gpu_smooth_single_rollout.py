"""Persistent rollouts of single drones with smooth contacts (an instance without
staging and rows in shared memory) equal per-call steps, with and without
scenario goals (whose values it keeps there), across episodes."""
import pytest
import torch

from gpu_helpers import DEV
from paper_2306_09537_gb300 import qs
from paper_2306_09537_gb300.env import QuadSwarmEnv

pytestmark = pytest.mark.gpu
FEATS = ("smooth", "motor_noise", "obs_noise", "dr", "auto_reset")
MOVING = ("static", "dynamic", "shrink_expand", "pursuit_lissajous", "pursuit_bezier")


@pytest.mark.parametrize("E,block", [(1, 32), (33, 32), (1537, 64), (300, 128), (1025, 256)])
@pytest.mark.parametrize("K,scenarios", [(0, ()), (8, ()), (0, MOVING), (2, MOVING)])
def test_rollout_equals_steps(E, block, K, scenarios):
    T = 9
    a, b = (QuadSwarmEnv(E, 1, K, FEATS, seed=4, device=DEV, scenarios=scenarios, episode_steps=5) for _ in range(2))
    qs.qs_set_rollout_shape(a.h, block, 4, True)
    acts = torch.rand(T, E, 4, generator=torch.Generator(device=DEV).manual_seed(1), device=DEV)
    obs, rew = torch.empty(T, E, a.obs_dim, device=DEV), torch.empty(T, E, device=DEV)
    done = torch.empty(T, E, dtype=torch.uint8, device=DEV)
    a.rollout(acts, obs, rew, done)
    for t in range(T):
        o, r, d = b.step(acts[t])
        assert torch.equal(obs[t], o) and torch.equal(rew[t], r) and torch.equal(done[t], d), t
    assert torch.equal(a.get_state()["state"], b.get_state()["state"])
