"""The x-transforms and the channel mixing of the spectral branch at the edges of their
tiles: odd mode counts, one mode, 2m = N, rows that are no multiple of 64, several x
chunks per channel (few channels on a long axis), odd batches, more modes than the tiled
kernels take; forward and gradients against the oracle."""
import numpy as np
import pytest
import torch

from oracle import fno as ofno
from tests.test_gpu_fno import setup, unflatten

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,m,B,N", [(8, 1, 1, 4), (8, 5, 3, 10), (16, 7, 1, 130), (8, 16, 1, 192), (32, 32, 1, 64),
                                     (8, 33, 1, 66), (7, 3, 5, 64), (64, 2, 3, 12)])
def test_spectral_branch_edges(cuda, W, m, B, N):
    net, P = setup(cuda, W, m, 2, 16, seed=m)
    rng = np.random.default_rng(N)
    x = rng.standard_normal((B, 7, N, N)).astype(np.float32)
    t = rng.standard_normal((B, N, N)).astype(np.float32)
    xd = torch.tensor(x, device=cuda)
    out = net.forward(B, N, xd, torch.empty((B, N, N), dtype=torch.float32, device=cuda)).cpu().numpy()
    ref, cache = ofno.forward(P, x.astype(np.float64), m)
    assert np.linalg.norm(out - ref) / np.linalg.norm(ref) < 2e-5
    g = torch.empty(net.count, dtype=torch.float32, device=cuda)
    net.gradients(B, N, xd, torch.tensor(t, device=cuda), g)
    G = ofno.backward(P, cache, ref, t.astype(np.float64), m)
    got = unflatten(g.cpu().numpy(), P)
    for k in G:
        err = np.linalg.norm(got[k] - G[k]) / max(np.linalg.norm(G[k]), 1e-30)
        assert err < 1e-4, (k, err)
    net.close()
