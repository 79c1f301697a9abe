"""Weight gradients of the pointwise layers (pixel contraction in 32 x 32 output blocks,
groups of 32 pixels) at the widths and pixel counts where its tiles are ragged: every
width class, a pixel count that is no multiple of 32, features that start on a 4-byte
boundary only, and a batch reused at a smaller size; against the oracle."""
import numpy as np
import pytest
import torch

from oracle import fno as ofno
from paper_1807_01885_gb300 import bem
from tests.test_gpu_fno import setup, unflatten

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,m,L,H,B,N", [(32, 4, 2, 64, 2, 18), (64, 3, 1, 64, 1, 22), (1, 2, 1, 7, 3, 6),
                                         (16, 5, 3, 32, 3, 40), (7, 3, 2, 8, 1, 96), (32, 16, 2, 16, 2, 48)])
def test_gradients_at_ragged_sizes(cuda, W, m, L, H, B, N):
    net, P = setup(cuda, W, m, L, H, seed=W + N)
    rng = np.random.default_rng(N)
    for b in (B, 1):                   # the second call runs in buffers sized for the first
        x = rng.standard_normal((b, 7, N, N)).astype(np.float32)
        t = rng.standard_normal((b, N, N)).astype(np.float32)
        raw = torch.empty(x.size + 1, dtype=torch.float32, device=cuda)
        xd = raw[1:].view(b, 7, N, N)   # 4-byte aligned only
        xd.copy_(torch.tensor(x))
        g = torch.empty(net.count, dtype=torch.float32, device=cuda)
        loss = net.gradients(b, N, xd, torch.tensor(t, device=cuda), g)
        out, cache = ofno.forward(P, x.astype(np.float64), m)
        assert loss == pytest.approx(ofno.loss(out, t.astype(np.float64)), rel=1e-5)
        G = ofno.backward(P, cache, out, t.astype(np.float64), m)
        got = unflatten(g.cpu().numpy(), P)
        for k in G:
            err = np.linalg.norm(got[k] - G[k]) / max(np.linalg.norm(G[k]), 1e-30)
            assert err < 1e-4, (b, k, err)
    net.close()
