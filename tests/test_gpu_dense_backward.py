"""The backward instance for batches of several waves (six CTAs an SM) against
the one for small batches: the first envs of a large handle and a small handle
hold the same drones, so their losses and gradients agree up to the rounding of
the two compilations (a few hundred operations of 6e-8 relative each)."""
import pytest
import torch

from gpu_helpers import DEV
from paper_2306_09537_gb300 import workloads as W
from paper_2306_09537_gb300.env import QuadSwarmEnv, RolloutFn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("feats", [("smooth", "motor_noise"), ("floor", "walls", "collisions", "motor_noise"),
                                   ("floor", "walls", "collisions", "motor_noise", "event_time")])
def test_dense_backward_agrees_with_small_batches(feats):
    n, T, C, small = 8, 6, 4, 12
    big = torch.cuda.get_device_properties(0).multi_processor_count * 4 * 32 // n + 40  # past one wave of four CTAs an SM
    x = torch.from_numpy(W.contact_swarm_states(3, big, n)).to(DEV)
    acts = torch.from_numpy(W.actions(3, T, big * n)).to(DEV)
    out = []
    for E in (big, small):
        env = QuadSwarmEnv(E, n, 6, feats, seed=6, device=DEV)
        env.set_state(goals=torch.zeros(E, 3, device=DEV))
        a, s = acts[:, :E * n].contiguous().requires_grad_(), x[:E * n].contiguous().requires_grad_()
        loss = RolloutFn.apply(a, s, env, C)
        g = torch.autograd.grad(loss.sum(), (a, s))
        env.sync()
        out.append((loss[:small * n], g[0][:, :small * n], g[1][:small * n]))
    assert torch.equal(out[0][0], out[1][0])
    for p, q in zip(out[0][1:], out[1][1:]):
        assert float((p - q).abs().max()) <= 1e-5 * float(q.abs().max())
