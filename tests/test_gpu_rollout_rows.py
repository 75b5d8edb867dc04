"""Observation rows of the persistent rollout leave as blocks (bulk copies of
16-byte units): rows must equal per-call steps wherever the buffer starts
(8 bytes off a 16-byte boundary), for odd drone counts, for swarms whose rows
do not follow one another, and in host memory, with nothing written around
them."""
import numpy as np
import pytest
import torch

from gpu_helpers import DEV
from paper_2306_09537_gb300 import qs
from paper_2306_09537_gb300.env import QuadSwarmEnv

pytestmark = pytest.mark.gpu
FEATS = ("floor", "walls", "motor_noise", "obs_noise", "dr", "collisions")


@pytest.mark.parametrize("where", ["aligned", "offset", "pinned"])
@pytest.mark.parametrize("sizes,K", [([1, 2, 1, 4, 8, 3, 16, 7, 1, 33] * 3, 6), ([7] * 41, 5), ([2] * 33, 1), ([3] * 7, 0),
                                     ([1, 1, 2, 1], 8), ([64] * 3, 7), ([127, 128, 100], 8), ([5], 2)])
@pytest.mark.parametrize("block", [128, 256])
def test_rows_equal_steps(sizes, K, where, block):
    T, E, D = 3, len(sizes), int(sum(sizes))
    a, b = (QuadSwarmEnv(E, np.asarray(sizes), K, FEATS, seed=4, device=DEV) for _ in range(2))
    qs.qs_set_rollout_shape(a.h, block, 0, False)
    acts = torch.rand(T, D, 4, generator=torch.Generator(device=DEV).manual_seed(1), device=DEV)
    n, pad = T * D * a.obs_dim, 64
    base = torch.full((n + 2 * pad,), -7.0, device=None if where == "pinned" else DEV)
    base = base.pin_memory() if where == "pinned" else base
    lo = pad + (2 if where == "offset" else 0)
    obs = base[lo:lo + n].view(T, D, a.obs_dim)
    a.rollout(acts, obs, None, None)
    a.sync()
    want = torch.stack([b.step(acts[t])[0].clone() for t in range(T)])
    torch.cuda.synchronize()
    assert torch.equal(obs.to(DEV), want)
    assert bool((base[:lo] == -7.0).all()) and bool((base[lo + n:] == -7.0).all())
