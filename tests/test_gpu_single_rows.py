"""Rows of single-drone handles in the persistent rollout: stored by their lanes
while their neighbour fields are few (up to 640 an SM in all), sent through shared
memory beyond, both equal to per-call steps wherever the buffer starts, with
nothing written around them."""
import pytest
import torch

from gpu_helpers import DEV
from paper_2306_09537_gb300 import qs
from paper_2306_09537_gb300.env import QuadSwarmEnv

pytestmark = pytest.mark.gpu
FEATS = {"common": ("floor", "walls", "motor_noise", "obs_noise", "dr"), "smooth": ("smooth", "motor_noise", "obs_noise", "dr"),
         "downwash": ("floor", "walls", "motor_noise", "obs_noise", "downwash")}


@pytest.mark.parametrize("feats", sorted(FEATS))
@pytest.mark.parametrize("K", [0, 2, 3, 6, 8])
@pytest.mark.parametrize("E,block,where", [(1, 32, "aligned"), (31, 32, "offset"), (33, 64, "pinned"), (1537, 32, "pinned"),
                                           (1537, 128, "offset"), (700, 256, "aligned")])
def test_rows_equal_steps(feats, K, E, block, where):
    check(feats, K, E, block, where)


@pytest.mark.parametrize("feats", ["common", "smooth"])
@pytest.mark.parametrize("K,block,where", [(1, 32, "offset"), (2, 32, "aligned"), (3, 64, "offset"), (8, 32, "pinned"),
                                           (8, 128, "offset"), (6, 256, "aligned")])
@pytest.mark.parametrize("past", [0, 1])
def test_both_sides_of_the_line(feats, K, block, where, past):
    check(feats, K, 640 * torch.cuda.get_device_properties(DEV).multi_processor_count // K + past, block, where)


def check(feats, K, E, block, where):
    T = 3
    a, b = (QuadSwarmEnv(E, 1, K, FEATS[feats], seed=4, device=DEV) for _ in range(2))
    qs.qs_set_rollout_shape(a.h, block, 0, False)
    acts = torch.rand(T, E, 4, generator=torch.Generator(device=DEV).manual_seed(1), device=DEV)
    n, pad = T * E * a.obs_dim, 64
    base = torch.full((n + 2 * pad,), -7.0, device=None if where == "pinned" else DEV)
    base = base.pin_memory() if where == "pinned" else base
    lo = pad + (2 if where == "offset" else 0)
    obs = base[lo:lo + n].view(T, E, a.obs_dim)
    a.rollout(acts, obs, None, None)
    a.sync()
    want = torch.stack([b.step(acts[t])[0].clone() for t in range(T)])
    torch.cuda.synchronize()
    assert torch.equal(obs.to(DEV), want)
    assert bool((base[:lo] == -7.0).all()) and bool((base[lo + n:] == -7.0).all())
