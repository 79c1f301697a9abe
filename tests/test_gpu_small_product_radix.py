"""The one-launch float product does not depend on the radices that a handle's passes were
given (by bem_set_radix, a tuning file or bem_autotune): one launch and the same result bit
for bit, also after a rebuild in place; the passes themselves (which a handle takes while
they are timed) follow the choice and agree to rounding."""
import numpy as np
import pytest
import torch

from paper_1807_01885_gb300 import bem
from paper_1807_01885_gb300.tuning import RadixCache

pytestmark = pytest.mark.gpu

MATERIAL = (2.0, 0.3, 1.0, 0.25)


def one_launch(k, p):
    before = bem.bem_launch_count()
    u = k.matvec(p)
    assert bem.bem_launch_count() - before == 1
    return u


@pytest.mark.parametrize("N", [16, 32, 64])
def test_any_radix_keeps_the_one_launch_product(cuda, N):
    p = torch.tensor(np.random.default_rng(N).standard_normal((N, N)), device=cuda, dtype=torch.float32)
    with bem.Kernel(N, 1.0 / N, 8.0 / N, *MATERIAL, precision="fp32") as k:
        first = one_launch(k, p)
        for choice in [(4, 4), (3, 4), (4, 3), (3, 3)]:
            k.set_radix(*choice)
            assert torch.equal(one_launch(k, p), first)
            bem.bem_set_pass_timing(k.handle, True)
            v = k.matvec(p)
            bem.bem_set_pass_timing(k.handle, False)
            assert float((v - first).norm() / first.norm()) < 5e-7
        RadixCache(fixed=(4, 4)).apply(k)
        assert torch.equal(one_launch(k, p), first)
        k.rebuild(1.0 / N, 5.0 / N, *MATERIAL)
        with bem.Kernel(N, 1.0 / N, 5.0 / N, *MATERIAL, precision="fp32") as other:
            assert torch.equal(one_launch(k, p), one_launch(other, p))
        k.autotune(reps=2)
        one_launch(k, p)
        assert k.check_guards() == 0
