"""Per-call steps of single drones past two waves of CTAs (launched without overlap,
their rows sent through shared memory or stored by the lanes by the number of
substeps) equal rollouts and, in the middle of a stream of overlapped launches
and torch's own, need no waits."""
import pytest
import torch

from gpu_helpers import DEV
from paper_2306_09537_gb300 import qs
from paper_2306_09537_gb300.env import QuadSwarmEnv

pytestmark = pytest.mark.gpu
COMMON = ("floor", "walls", "motor_noise", "obs_noise", "dr")


@pytest.mark.parametrize("where", ["aligned", "offset", "pinned"])
@pytest.mark.parametrize("feats,K,substeps,kw", [
    (COMMON, 0, 2, {}), (COMMON, 0, 3, {}), (COMMON, 1, 4, {}), (COMMON, 1, 5, {}), (COMMON, 8, 2, {}),
    (COMMON, 0, 2, {"scenarios": ("static", "pursuit_lissajous")}), (("smooth", "motor_noise", "obs_noise"), 0, 2, {})])
def test_large_single_drone_step(feats, K, substeps, kw, where):
    E, T = torch.cuda.get_device_properties(DEV).multi_processor_count * 1536 + 1537, 3
    a, b = (QuadSwarmEnv(E, 1, K, feats, seed=4, device=DEV, substeps=substeps, **kw) for _ in range(2))
    other = QuadSwarmEnv(600, 8, 2, COMMON + ("collisions",), seed=5, device=DEV)
    acts = torch.rand(T, E, 4, generator=torch.Generator(device=DEV).manual_seed(1), device=DEV)
    n, pad = E * a.obs_dim, 64
    base = torch.full((n + 2 * pad,), -7.0, device=None if where == "pinned" else DEV)
    base = base.pin_memory() if where == "pinned" else base
    lo = pad + (2 if where == "offset" else 0)
    obs, got, policy = base[lo:lo + n].view(E, a.obs_dim), [], torch.rand(other.D, 4, device=DEV)
    for t in range(T):
        other.step(policy)
        qs.qs_step(a.h, acts[t] * 1.0, obs, a.reward, a.done)
        policy = torch.sigmoid(other.obs[:, :4])
        other.step(policy)
        if where == "pinned":
            torch.cuda.synchronize()
        got.append((obs.to(DEV, copy=True), a.reward.clone()))
    rows, rew = torch.empty(T, E, a.obs_dim, device=DEV), torch.empty(T, E, device=DEV)
    b.rollout(acts, rows, rew, None)
    torch.cuda.synchronize()
    for t in range(T):
        assert torch.equal(got[t][0], rows[t]) and torch.equal(got[t][1], rew[t]), t
    assert torch.equal(a.get_state()["state"], b.get_state()["state"])
    assert bool((base[:lo] == -7.0).all()) and bool((base[lo + n:] == -7.0).all())
