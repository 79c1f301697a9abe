"""Block shapes of the product's passes: every grid size in both precisions (one warp per
block at the small end, several blocks per SM at the large one) and every radix, against
numpy's FFT of the zero-padded product with the library's own table."""
import numpy as np
import pytest
import torch

from paper_1807_01885_gb300 import bem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [16, 32, 64, 128, 512, 1024, 2048])
@pytest.mark.parametrize("precision,tol", [("fp32", 2e-6), ("fp64", 1e-12)])
def test_every_grid_size(cuda, N, precision, tol):
    p = np.random.default_rng(N).standard_normal((N, N))
    with bem.Kernel(N, 1.0 / N, 8.0 / N, 2.0, 0.3, 1.0, 0.25, precision=precision) as k:
        K = k.table().cpu().numpy()
        i = np.minimum(np.arange(2 * N), 2 * N - np.arange(2 * N))
        pd = torch.tensor(p, device=cuda, dtype=k.torch_dtype)
        ref = np.fft.irfft2(np.fft.rfft2(pd.double().cpu().numpy(), s=(2 * N, 2 * N)) * K[i], s=(2 * N, 2 * N))[:N, :N]
        for radix in [None] + ([(3, 3), (4, 4)] if precision == "fp32" else []):
            if radix is not None:
                k.set_radix(*radix)
            u = k.matvec(pd).double().cpu().numpy()
            assert np.linalg.norm(u - ref) / np.linalg.norm(ref) < tol
        assert k.check_guards() == 0
