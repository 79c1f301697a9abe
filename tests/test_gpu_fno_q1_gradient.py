"""The gradient of the projection's first matrix, in isolation and under cancellation: the
layers are the identity (W = I, no modes) on features of 16 significant bits, so that the
products da v are all that is summed, with signs that cancel (random targets); against
the oracle.

Tolerance (relative, over all entries): per pixel, da carries the rounding of out (2e-7 of
out - target), of gelu' (1e-7) and of a few float products (1e-7), the float sums 1e-7;
together 3e-7 rms, doubled."""
import numpy as np
import pytest
import torch

from oracle import fno as ofno
from paper_1807_01885_gb300 import bem
from tests.test_gpu_fno import flatten, unflatten

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,N", [(8, 16, 64), (16, 32, 64), (32, 64, 64), (32, 7, 34), (7, 16, 64)])
def test_q1_gradient_under_cancellation(cuda, W, H, N):
    m, r = 2, np.random.default_rng(W + H)
    bf = lambda a: torch.tensor(a, dtype=torch.float32).bfloat16().double().numpy()
    P = ofno.init_params(r, 7, W, m, 1, H)
    P = {k: np.zeros_like(v, dtype=np.float64) for k, v in P.items()}
    P["P_w"][np.arange(W), np.arange(W) % 7] = 1.0
    P["W_w"][0] = np.eye(W)
    P["Q1_w"], P["Q1_b"] = bf(r.standard_normal((H, W)) / np.sqrt(W)), bf(0.1 * r.standard_normal(H))
    P["Q2_w"] = bf(r.standard_normal(P["Q2_w"].shape) / np.sqrt(H))
    net = bem.Fno(width=W, modes=m, layers=1, hidden=H)
    vec, _ = flatten(P)
    net.set_params(torch.tensor(vec, dtype=torch.float32, device=cuda))
    x = r.standard_normal((1, 7, N, N)).astype(np.float32)
    x = (x.view(np.uint32) & np.uint32(0xffffff00)).view(np.float32)   # 16 significant bits
    t = r.standard_normal((1, N, N)).astype(np.float32)
    g = torch.empty(net.count, dtype=torch.float32, device=cuda)
    net.gradients(1, N, torch.tensor(x, device=cuda), torch.tensor(t, device=cuda), g)
    out, cache = ofno.forward(P, x.astype(np.float64), m)
    G = ofno.backward(P, cache, out, t.astype(np.float64), m)["Q1_w"]
    got = unflatten(g.cpu().numpy(), P)["Q1_w"]
    assert np.linalg.norm(got - G) / np.linalg.norm(G) < 6e-7
    net.close()
