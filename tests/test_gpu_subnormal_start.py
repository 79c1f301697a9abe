"""Warm starts with pressures so small that the first rescaling to the given force takes
them to zero: those cells are not in contact, and the solve is the one from the same start
without them.  Single cells of otherwise loaded groups and whole groups alike; products of
such pressures lie far below the rounding of the others, so the results are equal."""
import numpy as np
import pytest
import torch

from paper_1807_01885_gb300 import bem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [16, 64, 256])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_subnormal_cells_leave_the_contact_set(cuda, N, precision):
    x = (np.arange(N) + 0.5) / N - 0.5
    with bem.Kernel(N, 1.0 / N, 0.2, 1.0, 0.3, np.inf, 0.3, precision=precision) as k:
        dt = k.torch_dtype
        f = torch.tensor(np.add.outer(x ** 2, x ** 2) / 2.0, device=cuda, dtype=dt)
        tol, tiny = (1e-8, 1.4e-45) if precision == "fp32" else (1e-10, 5e-324)
        p0, res0 = k.solve(f, "force", 1e-3, tol=tol)
        assert res0["status"] == 0
        starts = [torch.where(p0 > 0, 4.0 * p0, torch.full_like(p0, fill)) for fill in (0.0, tiny)]
        starts.append(torch.where(torch.rand_like(p0) < 0.3, starts[0], starts[1]))
        assert float(starts[1].min()) > 0.0
        got = [k.solve(f, "force", 1e-3, tol=tol, p_init=s) for s in starts]
        for p, res in got[1:]:
            assert res["status"] == 0 and res["iters"] == got[0][1]["iters"]
            assert torch.equal(p, got[0][0])
        outs = [torch.empty_like(p0)]
        prob = bem.make_problem(f, bem.BEM_CTRL_FORCE, 1e-3, tol=tol, p_init=starts[1])
        st, _ = bem.bem_solve_batch([k.handle], [prob], outs)
        assert st == 0 and torch.equal(outs[0], got[0][0])
        assert k.check_guards() == 0
