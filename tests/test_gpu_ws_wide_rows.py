"""The warp-specialised kernels with the longest observation rows: swarms of
33..64 (64 lanes a CTA) and K = 8 need more than 48 KiB of shared memory. The
rollout and the resident server must equal per-call steps."""
import pytest
import torch

from gpu_helpers import DEV
from paper_2306_09537_gb300 import qs
from paper_2306_09537_gb300.env import QuadSwarmEnv

pytestmark = pytest.mark.gpu
FEATS = ("floor", "walls", "motor_noise", "obs_noise", "dr", "collisions")


@pytest.mark.parametrize("n,K", [(64, 8), (64, 7), (40, 8), (32, 8), (1, 8)])
@pytest.mark.parametrize("extended", [False, True])
def test_ws_rollout_and_server_with_long_rows(n, K, extended):
    feats, kw = FEATS + (("downwash",) if extended else ()), dict(seed=4, device=DEV)
    if extended:
        kw["scenarios"] = ("static", "pursuit_lissajous")
    T, E = 4, 5
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        a, b, c = (QuadSwarmEnv(E, n, K, feats, stream=s, **kw) for _ in range(3))
        qs.qs_set_rollout_shape(a.h, qs.QS_BLOCK_WARP_SPECIALISED, 0, True)
        acts = torch.rand(T, a.D, 4, generator=torch.Generator(device=DEV).manual_seed(1), device=DEV)
        obs, rew = torch.empty(T, a.D, a.obs_dim, device=DEV), torch.empty(T, a.D, device=DEV)
        a.rollout(acts, obs, rew, None)
        s.synchronize()
        host = acts.cpu()
        with c.serve(slots=1) as srv:
            served = []
            for t in range(T):
                srv.slots[0].copy_(host[t])
                o, r, _ = srv.step(0)
                served.append((o.clone(), r.clone()))
        for t in range(T):
            o, r, _ = b.step(acts[t])
            assert torch.equal(obs[t], o) and torch.equal(rew[t], r), t
            assert torch.equal(served[t][0], o.cpu()) and torch.equal(served[t][1], r.cpu()), t
