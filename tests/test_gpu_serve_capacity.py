"""The largest handles the resident server takes: as many CTAs as the device
keeps at once (32 drone lanes a CTA: six an SM; 64 lanes, swarms of 33..64:
three an SM, two with scenarios, downwash or smooth contacts), whose served
steps equal per-call ones, and no more."""
import pytest
import torch

from gpu_helpers import DEV
from paper_2306_09537_gb300 import qs
from paper_2306_09537_gb300.env import QuadSwarmEnv

pytestmark = pytest.mark.gpu
FEATS = {"common": ("floor", "walls", "motor_noise", "obs_noise", "dr", "collisions"),
         "downwash": ("floor", "walls", "motor_noise", "collisions", "downwash"), "smooth": ("smooth", "motor_noise", "dr")}


@pytest.mark.parametrize("n,K,feats,ctas", [(64, 6, "common", 3), (33, 8, "common", 3), (64, 0, "common", 3),
                                            (64, 8, "downwash", 2), (40, 6, "smooth", 2), (1, 0, "common", 6),
                                            (8, 8, "common", 6), (32, 8, "downwash", 6), (5, 6, "smooth", 6)])
def test_server_capacity(n, K, feats, ctas):
    width = 1 << (n - 1).bit_length()
    per_cta = max(32, width) // width
    most = ctas * torch.cuda.get_device_properties(DEV).multi_processor_count * per_cta
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        a, b = (QuadSwarmEnv(most, n, K, FEATS[feats], seed=4, device=DEV, stream=s) for _ in range(2))
        act = torch.rand(a.D, 4, generator=torch.Generator(device=DEV).manual_seed(1), device=DEV)
        host = act.cpu()
        with a.serve() as srv:
            srv.actions.copy_(host)
            for _ in range(2):
                obs, reward, _ = srv.step()
        for _ in range(2):
            want, want_r, _ = b.step(act)
        assert torch.equal(obs, want.cpu()) and torch.equal(reward, want_r.cpu())
        over = QuadSwarmEnv(most + 1, n, K, FEATS[feats], seed=4, device=DEV, stream=s)
        with pytest.raises(qs.QSError):
            over.serve()
