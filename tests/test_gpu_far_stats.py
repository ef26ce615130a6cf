"""Counters of the far field's timed launches: launches, right-hand sides and
which launches took each pair of triangles once."""
import numpy as np
import pytest

from paper_2104_04609_gb300 import inputs

pytestmark = pytest.mark.gpu


# (vertices, vectors): launches, right-hand sides, symmetric launches
@pytest.mark.parametrize("nv,nrhs,expected", [(150, 1, (1, 1, 0)), (150, 3, (1, 3, 0)), (1155, 1, (1, 1, 1)),
                                              (1155, 5, (1, 5, 1)), (1155, 8, (1, 8, 0)), (1155, 9, (2, 9, 1)),
                                              (1155, 12, (2, 12, 1))])
def test_counts(nv, nrhs, expected):
    import torch

    from paper_2104_04609_gb300 import binding as B

    v, t = inputs.fibonacci_hull(nv)
    S = B.Solver(v, t, 3.0, 4.0, 1.5)
    try:
        rng = np.random.default_rng(nrhs)
        x = torch.from_numpy(rng.standard_normal((nrhs, 2 * nv)) + 0j).cuda()
        S.apply(x)
        for _ in range(2):
            B.osrc_profile_enable(S.pb, True)
            S.apply(x)
            n, ms = B.osrc_far_kernel_stats(S.pb)
            assert ms > 0.0
            assert (n, B.osrc_far_kernel_rhs(S.pb), B.osrc_far_kernel_symmetric(S.pb)) == expected
        B.osrc_profile_enable(S.pb, False)
    finally:
        S.close()
