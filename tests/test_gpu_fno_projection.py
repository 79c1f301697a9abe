"""The projection's gelu on its negative tail, where an approximation of erfc shows
undamped: a network whose only layer is the identity (W = I, no modes) and whose only
hidden unit is v[0], so that out = gelu(x[0]) exactly, on all three paths (one-pass
inference, inference on a grid that it does not take, the training forward, whose loss
against the exact gelu is the mean square of the error).  x lies on the bfloat16 grid.

Tolerance (rms over x in [-4, -2]): an error of 1e-8 in erfc is 1e-8 |x| / 2, and ten
float roundings of a value are 1e-6 of it."""
import numpy as np
import pytest
import torch

from oracle.fno import gelu
from paper_1807_01885_gb300 import bem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H", [(8, 8), (16, 64), (32, 16)])
@pytest.mark.parametrize("N", [16, 18])
def test_negative_tail(cuda, W, H, N):
    m = 2
    net = bem.Fno(width=W, modes=m, layers=1, hidden=H)
    P = dict(P_w=np.zeros((W, 7)), P_b=np.zeros(W), R=np.zeros((2, W, W, 2 * m, m)), W_w=np.eye(W), W_b=np.zeros(W),
             Q1_w=np.zeros((H, W)), Q1_b=np.zeros(H), Q2_w=np.zeros(H), Q2_b=np.zeros(1))
    P["P_w"][0, 0] = P["Q1_w"][0, 0] = P["Q2_w"][0] = 1.0
    net.set_params(torch.tensor(np.concatenate([v.reshape(-1) for v in P.values()]), dtype=torch.float32, device=cuda))
    x = torch.zeros((1, 7, N, N), device=cuda)
    x[0, 0] = torch.linspace(-4.0, -2.0, N * N, device=cuda).bfloat16().float().view(N, N)
    z = x[0, 0].double().cpu().numpy()
    exact = gelu(z)
    rms = lambda v: float(np.sqrt(np.mean(np.square(v))))
    tol = rms(1e-8 * z / 2) + 1e-6 * rms(exact)
    out = net.forward(1, N, x, torch.empty((1, N, N), device=cuda))
    assert rms(out[0].double().cpu().numpy() - exact) < tol
    loss = net.gradients(1, N, x, torch.tensor(exact, dtype=torch.float32, device=cuda).view(1, N, N))
    assert np.sqrt(loss) < tol
    net.close()
