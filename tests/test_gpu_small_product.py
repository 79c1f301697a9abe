"""The one-launch float product of small grids against the three passes (which a handle
takes while its passes are timed) on every size it serves, and in place inside a chain of
products with no synchronisation.  Tolerance: the two contract products and sums
differently, a few float roundings per stage."""
import numpy as np
import pytest
import torch

from paper_1807_01885_gb300 import bem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [16, 32, 64])
def test_equals_the_passes(cuda, N):
    with bem.Kernel(N, 1.0 / N, 8.0 / N, 2.0, 0.3, 1.0, 0.25, precision="fp32") as k:
        p = torch.tensor(np.random.default_rng(N).standard_normal((N, N)), device=cuda, dtype=torch.float32)
        before = bem.bem_launch_count()
        u = k.matvec(p)
        assert bem.bem_launch_count() - before == 1
        bem.bem_set_pass_timing(k.handle, True)
        v = k.matvec(p)
        bem.bem_set_pass_timing(k.handle, False)
        assert bem.bem_launch_count() - before == 4
        assert float((u - v).norm() / v.norm()) < 5e-7
        # a chain in which each product overwrites its own input
        a, b = p.clone(), p.clone()
        for _ in range(6):
            k.matvec(a, a)
        for _ in range(6):
            b = k.matvec(b)
            torch.cuda.synchronize()
        assert torch.equal(a, b)
        assert k.check_guards() == 0

