"""One-pass inference at the edges of its tiles: one, two and four chunks per row (N = 16
to 2048, chunk lengths that do not divide the row), every width, mode counts on both sides
of a 16-column block, one layer (lift, then the last layer), ragged hidden widths, a handle
that has trained before, and grids that take the other path; against the oracle (small) or
the training pass's own forward (large)."""
import numpy as np
import pytest
import torch

from oracle import fno as ofno
from paper_1807_01885_gb300 import bem
from tests.test_gpu_fno import setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,m,L,H,B,N", [(8, 1, 1, 1, 3, 16), (16, 8, 2, 7, 2, 32), (32, 9, 3, 64, 1, 48),
                                         (32, 16, 1, 16, 5, 32), (8, 12, 4, 8, 2, 112), (16, 16, 2, 32, 1, 528),
                                         (8, 5, 2, 16, 1, 34)])
def test_inference_matches_oracle(cuda, W, m, L, H, B, N):
    net, P = setup(cuda, W, m, L, H, seed=N)
    x = np.random.default_rng(N).standard_normal((B, 7, N, N)).astype(np.float32)
    xd = torch.tensor(x, device=cuda)
    out = torch.empty((B, N, N), dtype=torch.float32, device=cuda)
    net.forward(B, N, xd, out)
    first = out.clone()
    ref, _ = ofno.forward(P, x.astype(np.float64), m)
    assert np.linalg.norm(first.cpu().numpy() - ref) / np.linalg.norm(ref) < 2e-5
    net.gradients(B, N, xd, torch.zeros_like(out))       # the handle now holds training buffers
    net.forward(B, N, xd, out)
    assert torch.equal(out, first)
    net.close()


@pytest.mark.parametrize("W,m,N", [(8, 16, 1040), (16, 4, 2048), (8, 16, 1536)])
def test_long_rows_match_the_training_forward(cuda, W, m, N):
    """The loss of the training pass against a zero target is the mean square of its output."""
    net, _ = setup(cuda, W, m, 2, 16, seed=W)
    g = torch.Generator(device=cuda).manual_seed(N)
    x = torch.randn((1, 7, N, N), generator=g, device=cuda)
    out = torch.empty((1, N, N), dtype=torch.float32, device=cuda)
    net.forward(1, N, x, out)
    target = out.clone()
    loss = net.gradients(1, N, x, target)
    scale = float((out.double() ** 2).mean())
    assert loss < (2e-5) ** 2 * scale
    net.close()
