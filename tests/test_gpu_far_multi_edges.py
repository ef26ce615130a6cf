"""Far field of several right-hand sides at the edges of its launch rules: 2 to
8 vectors a launch, a single one left over, blocks of 32, 64 and 128 test
triangles with source tiles that do not divide, a mesh without far pairs, plain
and centred phases, vectors of unlike sizes; against rows of the FP64 oracle's
matrix.

Tolerance: as for one right-hand side (FP32 evaluation of sums over up to 4e4
source points): 1e-5 per vector."""
import numpy as np
import pytest

from paper_2104_04609_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nv,k", [(4, 1.0), (9, 1.5), (33, 2.0), (1025, 4.0), (1026, 60.0), (2049, 60.0), (2050, 4.0)])
@pytest.mark.parametrize("nrhs", [2, 3, 7, 9, 18])
def test_multi_apply_at_size_edges(nv, k, nrhs):
    import torch

    import oracle as O
    from paper_2104_04609_gb300 import binding as B

    if nv == 4:
        v = np.array([[1, 1, 1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1]], dtype=np.float64)
        t = inputs.orient_outward(v, np.array([[0, 1, 2], [0, 1, 3], [0, 2, 3], [1, 2, 3]], dtype=np.int32))
    else:
        v, t = inputs.fibonacci_hull(nv)
    k1, rho = 1.3 * k, 1.5
    rng = np.random.default_rng(nv + nrhs)
    x = rng.standard_normal((nrhs, 2 * nv)) + 1j * rng.standard_normal((nrhs, 2 * nv))
    x[0] *= 1e8
    x[-1] *= 1e-8
    rows = np.unique(np.concatenate([[0, nv - 1], rng.integers(0, nv, 2)]))
    S = B.Solver(v, t, k, k1, rho)
    try:
        y = S.apply(torch.from_numpy(x).cuda()).cpu().numpy()
    finally:
        S.close()
    R1, R2 = O.pmchwt_rows(v, t, k, k1, rho, rows, nss=4)
    for r in range(nrhs):
        for got, ref in ((y[r, rows], R1 @ x[r]), (y[r, nv + rows], R2 @ x[r])):
            err = np.abs(got - ref).max() / np.abs(ref).max()
            assert err < 1e-5, f"{nv} vertices, vector {r} of {nrhs}: {err}"
