"""A rollout after a reset with another seed draws that seed's noise, also where
the rollout replays a captured graph (a stream of its own, the same buffers)."""
import pytest
import torch

from gpu_helpers import DEV
from paper_2306_09537_gb300.env import QuadSwarmEnv

pytestmark = pytest.mark.gpu
FEATS = ("floor", "walls", "motor_noise", "obs_noise", "dr", "collisions", "auto_reset")


@pytest.mark.parametrize("n,K", [(1, 0), (5, 3)])
def test_rollout_equals_steps_after_each_reset(n, K):
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        a, b = (QuadSwarmEnv(70, n, K, FEATS, seed=1, device=DEV, stream=s) for _ in range(2))
        acts = torch.rand(6, a.D, 4, generator=torch.Generator(device=DEV).manual_seed(1), device=DEV)
        obs = torch.empty(6, a.D, a.obs_dim, device=DEV)
        for seed in (1, 2, 2, 3):
            a.reset(seed)
            b.reset(seed)
            a.rollout(acts, obs)
            want = torch.stack([b.step(acts[t])[0].clone() for t in range(6)])
            s.synchronize()
            assert torch.equal(obs, want), seed
