"""Neighbour lists when many distances agree in their upper bits: the words
the pair pass sorts drop the low bits of a key, so these lists are decided by
the exact keys. Drones hover (their binary32 positions stay) on a lattice with
jitter of a few units in the last place; lists and collision flags must equal
the canonical ones bit for bit."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from gpu_helpers import DEV, nominal, pair, set_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[2] * 40, [3, 4] * 20, [5, 7, 8] * 20, [9, 15, 16] * 12, [17, 32] * 8, [33, 63, 64] * 4,
                                   [65, 127, 128] * 3, [1, 2, 4, 8, 9, 16, 30, 64, 128] * 2])
@pytest.mark.parametrize("K", [1, 6, 8])
def test_near_ties_decided_by_exact_keys(sizes, K):
    env, o = pair(sizes, K, ("collisions", "record_knn"), seed=5, alpha_c=1.0)
    D, E = env.D, env.E
    rng = np.random.RandomState(17 + K + len(sizes))
    st = np.zeros((D, 30), np.float32)
    st[:, 0:3] = 0.5 * rng.randint(-2, 3, (D, 3)) + rng.uniform(-3e-6, 3e-6, (D, 3)) + (0.0, 0.0, 4.0)
    st[:, 6:15] = np.eye(3, dtype=np.float32).ravel()
    st[:, 18:22] = np.float32(np.sqrt(0.5))
    st[:, 26:30] = 0.5
    prm = np.tile(np.asarray(nominal(env), np.float32), (E, 1))
    set_both(env, o, st, prm, np.zeros((E, 3), np.float32))
    env.step(torch.full((D, 4), 0.5, device=DEV))
    ev, knn = env.get_events(knn=True)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    bk, bh = O.pairs_f32(st[:, 0:3], prm[:, 6], off, K)
    assert np.array_equal(knn.cpu().numpy().astype(np.int32), bk)
    assert np.array_equal((ev.cpu().numpy() & O.EV_HIT_QUAD) != 0, bh.astype(bool))
