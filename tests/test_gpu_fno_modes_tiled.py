"""The register-tiled x-transforms (from 12 modes and 304 channels, or blocks of 64 rows, on)
against the plain kernels, which the same network takes for one sample at a time: odd mode
counts, several groups of slices, 2m = N, a partial last block of rows.

Forward: the sums have the same order, so every sample is equal bit for bit.  Gradients:
with a power-of-two batch every value of a sample is scaled exactly, and only the order
of the sums over samples and pixels differs: float roundings of a few hundred additions,
1e-6, tripled."""
import numpy as np
import pytest
import torch

from paper_1807_01885_gb300 import bem
from tests.test_gpu_fno import setup, unflatten

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,m,B,N", [(32, 12, 16, 34), (32, 13, 16, 66), (32, 24, 16, 66), (32, 31, 16, 130),
                                     (32, 32, 16, 64), (16, 16, 32, 80), (8, 15, 64, 98), (64, 17, 8, 40)])
def test_batch_equals_single_samples(cuda, W, m, B, N):
    net, P = setup(cuda, W, m, 2, 16, seed=m)
    g = torch.Generator(device=cuda).manual_seed(N)
    x = torch.randn((B, 7, N, N), generator=g, device=cuda)
    t = torch.randn((B, N, N), generator=g, device=cuda)
    assert B * W >= 304 > W * -(-N // 64)
    out = net.forward(B, N, x, torch.empty_like(t))
    for b in range(B):
        assert torch.equal(net.forward(1, N, x[b:b + 1].contiguous(), torch.empty_like(t[:1]))[0], out[b])
    grad = torch.empty(net.count, device=cuda)
    loss = net.gradients(B, N, x, t, grad)
    want, want_loss = torch.zeros(net.count, device=cuda, dtype=torch.float64), 0.0
    for b in range(B):
        one = torch.empty_like(grad)
        want_loss += net.gradients(1, N, x[b:b + 1].contiguous(), t[b:b + 1].contiguous(), one) / B
        want += one.double() / B
    assert loss == pytest.approx(want_loss, rel=1e-6)
    got, ref = unflatten(grad.cpu().numpy(), P), unflatten(want.cpu().numpy(), P)
    for k in ref:
        assert np.linalg.norm(got[k] - ref[k]) < 3e-6 * np.linalg.norm(ref[k]), k
    net.close()


@pytest.mark.parametrize("m,N", [(16, 640), (13, 618)])
def test_few_channels_on_a_long_axis(cuda, m, N):
    """Here only the inverse is tiled.  A network of 8 channels (plain kernels) and the same
    one among 24 more whose weights are zero."""
    small, P = setup(cuda, 8, m, 2, 16, seed=m)
    wide = {k: v for k, v in P.items()}
    for k, axes in dict(P_w=[0], P_b=[0], R_re=[1, 2], R_im=[1, 2], W_w=[1, 2], W_b=[1], Q1_w=[1]).items():
        wide[k] = np.pad(P[k], [(0, 24 if a in axes else 0) for a in range(P[k].ndim)])
    order = ["P_w", "P_b", "R_re", "R_im", "W_w", "W_b", "Q1_w", "Q1_b", "Q2_w", "Q2_b"]
    net = bem.Fno(width=32, modes=m, layers=2, hidden=16)
    net.set_params(torch.tensor(np.concatenate([wide[k].reshape(-1) for k in order]), dtype=torch.float32, device=cuda))
    assert 32 < 304 <= 32 * -(-N // 64)
    g = torch.Generator(device=cuda).manual_seed(N)
    x = torch.randn((1, 7, N, N), generator=g, device=cuda)
    t = torch.randn((1, N, N), generator=g, device=cuda)
    a, b = (n.forward(1, N, x, torch.empty_like(t)) for n in (small, net))
    assert float((a - b).norm() / a.norm()) < 1e-6
    ga, gb = torch.empty(small.count, device=cuda), torch.empty(net.count, device=cuda)
    assert small.gradients(1, N, x, t, ga) == pytest.approx(net.gradients(1, N, x, t, gb), rel=1e-6)
    got, ref = unflatten(gb.cpu().numpy(), wide), unflatten(ga.cpu().numpy(), P)
    for k in ref:
        part = got[k][tuple(slice(0, n) for n in ref[k].shape)]
        assert np.linalg.norm(part - ref[k]) < 3e-6 * np.linalg.norm(ref[k]), k
    small.close()
    net.close()
