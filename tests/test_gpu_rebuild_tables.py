"""A rebuild in place makes the tables that depend on the operator, not those of the grid
size alone: the double product's twiddles are made with the handle.  Rebuilt and fresh
handles give the same product bit for bit."""
import numpy as np
import pytest
import torch

from paper_1807_01885_gb300 import bem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [16, 32, 256, 2048])
def test_rebuild_leaves_the_fixed_point_twiddles(cuda, N):
    new = (5.0 / N, 1.0, 0.4, np.inf, 0.3)
    p = torch.tensor(np.random.default_rng(N).standard_normal((N, N)), device=cuda)
    with bem.Kernel(N, 1.0 / N, 8.0 / N, 2.0, 0.3, 1.0, 0.25) as k, bem.Kernel(N, 1.0 / N, *new) as fresh, \
            bem.Kernel(8, 1.0 / 8, 1.0, 2.0, 0.3, 1.0, 0.25) as small:   # N = 8: no fixed point
        k.matvec(p)
        counts = []
        for h, n in ((small, 8), (k, N)):
            before = bem.bem_launch_count()
            h.rebuild(1.0 / n, *new)
            counts.append(bem.bem_launch_count() - before)
        assert counts[0] == counts[1]
        assert torch.equal(k.matvec(p), fresh.matvec(p))
        assert k.check_guards() == 0 and fresh.check_guards() == 0
