"""The Calderon preconditioner reports a failure of either of its two mass solves:
an infinite entry breaks the first one down, and the second, whose right-hand side
is not a number, ends at once."""
import numpy as np
import pytest

from paper_2104_04609_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nv", [150, 21000])  # the mixed kernel, the FP64 one
def test_first_mass_solve_breaks_down(nv):
    import torch

    from paper_2104_04609_gb300 import binding as B

    v, t = inputs.fibonacci_hull(nv)
    S = B.Solver(v, t, 2.0, 3.0, 1.5, precond=B.OSRC_PRECOND_CALDERON)
    try:
        x = torch.from_numpy(np.random.default_rng(1).standard_normal((1, 2 * nv)) + 0j).cuda()
        z = S.precond(x)
        assert torch.isfinite(torch.view_as_real(z)).all()
        bad = x.clone()
        bad[0, 7] = complex(float("inf"), 0.0)
        with pytest.raises(B.OsrcError) as e:
            S.precond(bad)
        assert e.value.status == B.OSRC_BREAKDOWN
        assert torch.equal(S.precond(x), z)
    finally:
        S.close()
