"""Far-field apply at the edges of its size rules: test triangles per block
(2048 and 4096 triangles), lanes of the gather (400 and 1500 vertices), blocks
and source splits that do not divide, meshes with no far pair at all; against
rows of the FP64 oracle's matrix.

Tolerance: FP32 evaluation of sums over up to 4e4 source points (unit roundoff
6e-8, phases k r below 32 pi in the plain variant), the 1e-5 of the other
operator tests."""
import numpy as np
import pytest

from paper_2104_04609_gb300 import inputs

pytestmark = pytest.mark.gpu


def _tetra():
    v = np.array([[1, 1, 1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1]], dtype=np.float64)
    return v, inputs.orient_outward(v, np.array([[0, 1, 2], [0, 1, 3], [0, 2, 3], [1, 2, 3]], dtype=np.int32))


@pytest.mark.parametrize("nv,k", [(4, 1.0), (9, 1.5), (33, 2.0), (400, 3.0), (401, 3.0), (1025, 4.0), (1026, 60.0),
                                  (1500, 4.0), (1501, 60.0), (2049, 4.0), (2050, 4.0)])
def test_apply_at_size_edges(nv, k):
    import torch

    import oracle as O
    from paper_2104_04609_gb300 import binding as B

    v, t = _tetra() if nv == 4 else inputs.fibonacci_hull(nv)
    k1, rho = 1.3 * k, 1.5
    rng = np.random.default_rng(nv)
    x = rng.standard_normal(2 * nv) + 1j * rng.standard_normal(2 * nv)
    rows = np.unique(np.concatenate([[0, nv - 1], rng.integers(0, nv, 4)]))
    S = B.Solver(v, t, k, k1, rho)
    try:
        y = S.apply(torch.from_numpy(x).cuda().reshape(1, -1)).cpu().numpy().ravel()
    finally:
        S.close()
    R1, R2 = O.pmchwt_rows(v, t, k, k1, rho, rows, nss=4)
    ref = np.concatenate([R1 @ x, R2 @ x])
    got = np.concatenate([y[rows], y[nv + rows]])
    for part in (slice(0, len(rows)), slice(len(rows), None)):
        err = np.abs(got[part] - ref[part]).max() / np.abs(ref[part]).max()
        assert err < 1e-5, f"{nv} vertices: {err}"
