"""Values that are not finite in a gradient pass: a NaN or an infinity anywhere in the
features or the target spreads over the whole network (every mode of the spectral branch
sees every pixel), so no gradient entry may come out finite."""
import numpy as np
import pytest
import torch

from paper_1807_01885_gb300 import bem

pytestmark = pytest.mark.gpu

# widths of every pointwise kernel; N = 18: a ragged last group of pixels
CASES = [(1, 7, 16), (7, 8, 16), (8, 16, 18), (16, 16, 16), (32, 64, 18), (64, 64, 16)]


def network(cuda, W, H):
    net = bem.Fno(width=W, modes=3, layers=2, hidden=H)
    g = torch.Generator(device=cuda).manual_seed(W)
    w = 0.3 * torch.randn(net.count, generator=g, device=cuda)
    return net, w, g


@pytest.mark.parametrize("W,H,N", CASES)
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_gradients_of_a_bad_pixel_are_not_finite(cuda, W, H, N, bad):
    net, w, g = network(cuda, W, H)
    net.set_params(w)
    for where in ("features", "target"):
        x = torch.randn((2, 7, N, N), generator=g, device=cuda)
        t = torch.randn((2, N, N), generator=g, device=cuda)
        grad = torch.zeros(net.count, device=cuda)
        loss = net.gradients(2, N, x, t, grad)
        assert np.isfinite(loss) and bool(torch.isfinite(grad).all())
        if where == "features":
            x[1, 2, N - 1, N - 1] = bad
        else:
            t[0, N // 2, 3] = bad
        loss = net.gradients(2, N, x, t, grad)
        assert not np.isfinite(loss)
        assert int(torch.isfinite(grad).sum()) == 0, where
    net.close()
