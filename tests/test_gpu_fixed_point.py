"""The double product's fixed-point transforms where block scaling can go wrong: every grid
size, a single loaded cell, rows of very different size, values near both ends of the
double range, an alternating field (all of it in the highest wave number), zero, and values
that are not finite.  Reference: numpy's FFT of the zero-padded product with the library's
own table.  Tolerance: the double FFT error of both sides, a few 2^-53 times the square root
of the number of stages, doubled for the four transforms, and the reference's own (the
alternating field's output is N times smaller against the low wave numbers' rounding)."""
import numpy as np
import pytest
import torch

from paper_1807_01885_gb300 import bem

pytestmark = pytest.mark.gpu


def fields(N):
    r = np.random.default_rng(N)
    w = r.standard_normal((N, N))
    spike = np.zeros((N, N))
    spike[N // 3, N // 2] = 3.7
    edge = np.zeros((N, N))
    edge[-1, -1] = -1.0
    return dict(white=w, contact=np.maximum(w - 1.0, 0.0), spike=spike, edge=edge, rows=w * 10.0 ** r.uniform(-12, 12, (N, 1)),
                alternating=np.where(np.add.outer(np.arange(N), np.arange(N)) % 2 == 0, 1.0, -1.0))


@pytest.mark.parametrize("N", [16, 32, 64, 128, 256, 1024, 2048])
@pytest.mark.parametrize("body", ["stiff", "rigid"])
def test_fixed_point_product(cuda, N, body):
    mat = (8.0 / N, 2.0, 0.3, 1.0, 0.25) if body == "stiff" else (3.0 / N, 1.0, 0.4, np.inf, 0.3)
    with bem.Kernel(N, 1.0 / N, *mat) as k:
        K = k.table().cpu().numpy()
        K = K[np.minimum(np.arange(2 * N), 2 * N - np.arange(2 * N))]

        def product(p):
            return k.matvec(torch.tensor(p, device=cuda)).cpu().numpy()

        for name, p in fields(N).items():
            ref = np.fft.irfft2(np.fft.rfft2(p, s=(2 * N, 2 * N)) * K, s=(2 * N, 2 * N))[:N, :N]
            u = product(p)
            err = np.linalg.norm(u - ref) / np.linalg.norm(ref)
            assert err < (1e-14 if name != "alternating" else 1e-13), (name, err)
            # block scaling by powers of two: exact scaling of the result, also where the
            # transforms of a double product would leave the range on the way
            assert np.array_equal(product(p * 2.0 ** 200), u * 2.0 ** 200), name
            assert np.array_equal(product(p * 2.0 ** -200), u * 2.0 ** -200), name
        assert np.array_equal(product(np.zeros((N, N))), np.zeros((N, N)))
        for bad in (np.nan, np.inf, -np.inf):
            p = fields(N)["white"].copy()
            p[N // 2, 1] = bad
            assert not np.isfinite(product(p)).any()
        assert k.check_guards() == 0


def test_product_leaves_the_solve_alone(cuda):
    """A solve after products on the same handle equals one on a handle that made none."""
    N = 64
    f = torch.tensor(np.add.outer((np.arange(N) - 31.5) ** 2, (np.arange(N) - 31.5) ** 2) / (2.0 * N * N), device=cuda)
    out = []
    for products in (0, 3):
        with bem.Kernel(N, 1.0 / N, 0.2, 1.0, 0.3, np.inf, 0.3) as k:
            for _ in range(products):
                k.matvec(torch.ones_like(f))
            p, res = k.solve(f, "depth", 0.02, tol=1e-10)
            assert res["status"] == 0
            out.append(p)
    assert torch.equal(out[0], out[1])
