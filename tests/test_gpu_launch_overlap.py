"""Kernels brought onto the device while the stream's previous one ends see
everything earlier work wrote: a closed loop (each step's commands computed
from the last observations by torch on the same stream, two handles in turn)
gives the same bits with and without a wait after every call, and when the
loop is captured into a CUDA graph."""
import numpy as np
import pytest
import torch

from gpu_helpers import DEV
from paper_2306_09537_gb300 import workloads as W
from paper_2306_09537_gb300.env import QuadSwarmEnv, RolloutFn

pytestmark = pytest.mark.gpu
FEATS = ("floor", "walls", "motor_noise", "obs_noise", "dr", "collisions", "auto_reset")


def loop(envs, steps, wait, T=0):
    out = []
    for env in envs:
        env.reset(3)
    for _ in range(steps):
        for env in envs:
            a = torch.sigmoid(env.obs[:, 3:7] * 0.3)  # a stand-in policy
            if T:
                o = torch.empty(T, env.D, env.obs_dim, device=DEV)
                env.rollout(torch.stack([a + 0.01 * t for t in range(T)]), o, None, None)
                env.obs.copy_(o[-1])
            else:
                env.step(a)
            if wait:
                torch.cuda.synchronize()
            out.append(env.obs.clone())
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("swarm,E", [(1, 1), (1, 8192), (1, 65536), (8, 300), (8, 8192), (64, 40), ("mixed", 200)])
@pytest.mark.parametrize("T", [0, 3])
def test_closed_loop_needs_no_waits(swarm, E, T):
    sizes = W.uneven_swarm_sizes(1, E) if swarm == "mixed" else swarm
    K = 0 if swarm == 1 else 6
    envs = [QuadSwarmEnv(E, sizes, K, FEATS, seed=s, device=DEV) for s in (3, 4)]
    for a, b in zip(loop(envs, 6, True, T), loop(envs, 6, False, T)):
        assert torch.equal(a, b)


def test_captured_steps_and_gradients():
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        a, b = (QuadSwarmEnv(500, 8, 6, FEATS, seed=5, device=DEV, stream=s) for _ in range(2))
        act = torch.rand(a.D, 4, device=DEV)
        for _ in range(2):
            a.step(act)
            b.step(act)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            for _ in range(4):
                a.step(act)
        for _ in range(3):
            g.replay()
        for _ in range(12):
            b.step(act)
        s.synchronize()
        assert torch.equal(a.obs, b.obs) and torch.equal(a.get_state()["state"], b.get_state()["state"])
    d = QuadSwarmEnv(64, 8, 6, ("smooth", "motor_noise"), seed=5, device=DEV)
    x, u = torch.from_numpy(W.random_states(2, d.D)).to(DEV), torch.from_numpy(W.actions(2, 9, d.D)).to(DEV)
    got = []
    for wait in (True, False):
        for _ in range(3):
            v = (u * 1.0).requires_grad_()
            loss = RolloutFn.apply(v, x, d, 4)
            if wait:
                torch.cuda.synchronize()
            got.append(torch.autograd.grad((loss * 0.5).sum(), v)[0])
    torch.cuda.synchronize()
    assert all(torch.equal(got[0], h) for h in got[1:])
    assert np.isfinite(got[0].cpu().numpy()).all()
