"""Rows of the per-call steps and of the warp-specialised rollout wherever the
buffer starts (8 bytes off a 16-byte boundary) and in page-locked memory, for odd
drone counts: equal bits in every kernel and shape, nothing written around
them."""
import pytest
import torch

from gpu_helpers import DEV
from paper_2306_09537_gb300 import qs
from paper_2306_09537_gb300.env import QuadSwarmEnv

pytestmark = pytest.mark.gpu
FEATS = ("floor", "walls", "motor_noise", "obs_noise", "dr", "collisions")
WS = qs.QS_BLOCK_WARP_SPECIALISED
PAD = 64


def guarded(n, where):
    """A buffer of n floats between guard words: (the whole, the buffer, its offset)."""
    base = torch.full((n + 2 * PAD,), -7.0, device=None if where == "pinned" else DEV)
    base = base.pin_memory() if where == "pinned" else base
    lo = PAD + (2 if where == "offset" else 0)
    return base, base[lo:lo + n], lo


def untouched(base, lo, n):
    return bool((base[:lo] == -7.0).all()) and bool((base[lo + n:] == -7.0).all())


def reference(E, n, K, acts):
    """Rows of every step from the handle's own (aligned) buffer, default shape."""
    env = QuadSwarmEnv(E, n, K, FEATS, seed=4, device=DEV)
    return [env.step(a)[0].clone() for a in acts]


@pytest.mark.parametrize("where", ["aligned", "offset", "pinned"])
@pytest.mark.parametrize("E,n,block", [(E, n, block) for E, n in ((1, 1), (31, 1), (33, 1), (1537, 1), (41, 7))
                                       for block in (32, 256, WS)] + [(9, 33, 64), (9, 33, 256), (3, 65, 128)])
@pytest.mark.parametrize("K", [0, 8])
def test_step_rows(E, n, block, K, where):
    env = QuadSwarmEnv(E, n, K, FEATS, seed=4, device=DEV)
    qs.qs_set_block(env.h, 1 << (n - 1).bit_length(), block)
    acts = torch.rand(3, env.D, 4, generator=torch.Generator(device=DEV).manual_seed(1), device=DEV)
    size = env.D * env.obs_dim
    base, obs, lo = guarded(size, where)
    for a, want in zip(acts, reference(E, n, K, acts)):
        qs.qs_step(env.h, a, obs, env.reward, env.done)
        torch.cuda.synchronize()
        assert torch.equal(obs.view(env.D, env.obs_dim).to(DEV), want)
    assert untouched(base, lo, size)


@pytest.mark.parametrize("E,n,K,block", [(33, 1, 0, 32), (1537, 1, 8, 256), (33, 1, 8, WS), (41, 7, 6, WS), (7, 40, 8, 64)])
def test_step_host_rows(E, n, K, block):
    env = QuadSwarmEnv(E, n, K, FEATS, seed=4, device=DEV)
    qs.qs_set_block(env.h, 1 << (n - 1).bit_length(), block)
    acts = torch.rand(2, env.D, 4, generator=torch.Generator(device=DEV).manual_seed(1), device=DEV)
    size = env.D * env.obs_dim
    base, obs, lo = guarded(size + 2, "pinned")
    obs = obs[2:]  # 8 bytes off
    for a, want in zip(acts, reference(E, n, K, acts)):
        qs.qs_step_host(env.h, a.cpu().pin_memory(), obs, torch.empty(env.D).pin_memory(), None)
        assert torch.equal(obs.view(env.D, env.obs_dim).to(DEV), want)
    assert untouched(base, lo + 2, size)


@pytest.mark.parametrize("where", ["aligned", "offset", "pinned"])
@pytest.mark.parametrize("sizes", [[1], [1] * 31, [1] * 1537, [7] * 41, [32] * 3, [1, 2, 1, 5, 32, 3] * 3, [64] * 3, [33, 1, 7] * 5])
@pytest.mark.parametrize("K", [0, 5, 8])
def test_warp_specialised_rollout_rows(sizes, K, where):
    T, E = 3, len(sizes)
    a, b = (QuadSwarmEnv(E, sizes, K, FEATS, seed=4, device=DEV) for _ in range(2))
    qs.qs_set_rollout_shape(a.h, WS, 0, False)
    acts = torch.rand(T, a.D, 4, generator=torch.Generator(device=DEV).manual_seed(1), device=DEV)
    size = T * a.D * a.obs_dim
    base, obs, lo = guarded(size, where)
    a.rollout(acts, obs, None, None)
    torch.cuda.synchronize()
    got = obs.view(T, a.D, a.obs_dim).to(DEV)
    for t in range(T):
        assert torch.equal(got[t], b.step(acts[t])[0]), t
    assert untouched(base, lo, size)
