"""Field evaluation at the edges of its source splits: fewer triangles than a
tile, target counts around a block, one target, two objects; against the
oracle's FP64 field.  Tolerance as in the other field tests: FP64 sums, 1e-10."""
import numpy as np
import pytest

from paper_2104_04609_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nv,npts", [(4, 1), (4, 129), (10, 127), (33, 128), (150, 1), (150, 1000), (401, 257)])
@pytest.mark.parametrize("objects", [1, 2])
def test_field_split_edges(nv, npts, objects):
    import torch

    import oracle as O
    from paper_2104_04609_gb300 import binding as B

    if nv == 4:
        v = np.array([[1, 1, 1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1]], dtype=np.float64)
        t = inputs.orient_outward(v, np.array([[0, 1, 2], [0, 1, 3], [0, 2, 3], [1, 2, 3]], dtype=np.int32))
    else:
        v, t = inputs.fibonacci_hull(nv)
    obj = None
    k0, k1, rho = 2.0, 3.0, 1.5
    if objects == 2:
        t = np.concatenate([t, t + len(v)]).astype(np.int32)
        v = np.concatenate([v - [2.0, 0, 0], v + [2.0, 0, 0]])
        obj = ([3.0, 1.2], [1.5, 0.8])
    rng = np.random.default_rng(nv + npts)
    # targets away from the surface: deep inside an object or outside
    pts = rng.standard_normal((npts, 3))
    pts *= (np.where(rng.random(npts) < 0.5, 0.15, 6.0) / np.linalg.norm(pts, axis=1))[:, None]
    if objects == 2:
        pts[:, 0] += np.where(np.linalg.norm(pts, axis=1) < 1.0, 2.0, 0.0)
    x = rng.standard_normal(2 * len(v)) + 1j * rng.standard_normal(2 * len(v))
    S = B.Solver(v, t, k0, k1, rho, objects=obj)
    try:
        u, reg = S.field(torch.from_numpy(x).cuda(), torch.from_numpy(pts).cuda(), B.OSRC_INC_PLANEWAVE, [0, 0, 1.0])
        u, reg = u.cpu().numpy(), reg.cpu().numpy()
    finally:
        S.close()
    if obj is None:
        ref = O.field(v, t, k0, k1, rho, x, pts)
    else:
        ref = O.field_objects(v, t, k0, obj[0], obj[1], x, pts)
    ref = ref[0] if isinstance(ref, tuple) else ref
    assert np.abs(u - ref).max() < 1e-10 * np.abs(ref).max()
    inside = np.zeros(npts, dtype=np.int32)
    for m in range(objects):
        c = np.array([2.0 * (2 * m - 1), 0, 0]) if objects == 2 else np.zeros(3)
        inside[np.linalg.norm(pts - c, axis=1) < 0.2] = m + 1
    assert (reg == inside).all()
