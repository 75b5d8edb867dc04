"""A CUDA graph that mixes overlapped launches with torch kernels, copies and a
second handle on a side stream (edges of both kinds, and joins) replays to the
same bits as the same calls made one by one."""
import pytest
import torch

from gpu_helpers import DEV
from paper_2306_09537_gb300 import qs
from paper_2306_09537_gb300.env import QuadSwarmEnv

pytestmark = pytest.mark.gpu
FEATS = ("floor", "walls", "motor_noise", "obs_noise", "dr", "collisions", "auto_reset")


@pytest.mark.parametrize("sizes,K", [([1] * 3000, 0), ([1] * 45000, 1), ([8] * 300, 6), ([1, 4, 9, 33] * 8, 2), ([64] * 20, 6)])
def test_captured_closed_loop_with_a_side_stream(sizes, K):
    main, side = torch.cuda.Stream(), torch.cuda.Stream()

    def handles():
        return (QuadSwarmEnv(len(sizes), sizes, K, FEATS, seed=5, device=DEV, stream=main),
                QuadSwarmEnv(700, 3, 2, FEATS, seed=6, device=DEV, stream=side))

    def loop(a, b, log):  # commands from observations; b's from a's and back, over a join each way
        for t in range(3):
            a.step(torch.sigmoid(a.obs[:, 3:7] * 0.3))
            a.step(a.obs[:, 3:7].abs().clamp(max=1.0))
            side.wait_stream(main)
            with torch.cuda.stream(side):
                act = torch.full((b.D, 4), 0.5, device=DEV) + 0.1 * torch.tanh(a.reward[:1])
                b.step(act)
                b.step(act * 0.9)
                log[t, 1].copy_(b.reward.sum())
            main.wait_stream(side)
            a.step(torch.sigmoid(b.obs[:1, 3:7]).expand(a.D, 4).contiguous())
            log[t, 0].copy_(a.obs.double().sum())

    with torch.cuda.stream(main):
        (a, b), (c, d) = handles(), handles()
        logs = [torch.zeros(3, 2, device=DEV, dtype=torch.float64) for _ in range(2)]
        for env in (a, b, c, d):
            env.obs.zero_(), env.reward.zero_()
        torch.cuda.synchronize()
        for _ in range(3):
            loop(a, b, logs[0])
        torch.cuda.synchronize()
        loop(c, d, logs[1])
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=main):
            loop(c, d, logs[1])
        g.replay()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(logs[0], logs[1])
        for p, q in ((a, c), (b, d)):
            assert torch.equal(p.obs, q.obs) and torch.equal(p.reward, q.reward)


@pytest.mark.parametrize("sizes,K", [([1] * 40000, 3), ([8] * 300, 6), ([1, 4, 9, 33] * 8, 2)])
def test_captured_rollout_without_its_own_graph(sizes, K):
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        a, b = (QuadSwarmEnv(len(sizes), sizes, K, FEATS, seed=5, device=DEV, stream=s) for _ in range(2))
        acts = torch.rand(4, a.D, 4, generator=torch.Generator(device=DEV).manual_seed(1), device=DEV)
        rows = [torch.empty(4, a.D, a.obs_dim, device=DEV) for _ in range(2)]
        for env in (a, b):
            qs.qs_set_rollout_shape(env.h, qs.qs_get_rollout_shape(env.h)[0], 3, False)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            a.rollout(acts * 0.5, rows[0])
            a.rollout(acts, rows[0])
        g.replay()
        b.rollout(acts * 0.5, rows[1])
        b.rollout(acts, rows[1])
        s.synchronize()
        assert torch.equal(rows[0], rows[1])
