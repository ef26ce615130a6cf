"""Rounding errors of the symmetric far field where they are not hidden behind
those of FP32 coordinates and phases (several objects or a large body, phases
from float-float centroid distances), for random vectors: the relative error
against the FP64 assembled operator in unit roundoffs u = 2^-24.

A sum of n terms of random sign, added one after the other, is off by about
0.29 u sqrt(n / 2) of its size (roundings of 0.29 u rms of a partial sum that
grows as a random walk).  A pair's 12 products and the 32 pairs of a tile give
0.7 u and 1.2 u, the kernel values about 1 u: 1.7 u together, and the bound is
2 u (products added to the tile's sums one by one measured 2.1 to 2.3 u)."""
import numpy as np
import pytest

from paper_2104_04609_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [1])
@pytest.mark.parametrize("objects", [True, False])
def test_error_in_roundoffs(objects, nrhs):
    import torch

    from paper_2104_04609_gb300 import binding as B

    k = 30.0
    v0, t0 = inputs.fibonacci_hull(600)
    at = [(-3.0, -1.5, 0.0), (-3.0, 1.5, 0.0), (3.0, -1.5, 0.0), (3.0, 1.5, 0.0)]
    if objects:
        v = np.concatenate([v0 + np.array(a) for a in at])
        t = np.concatenate([t0 + i * len(v0) for i in range(4)]).astype(np.int32)
        mat = ([k * 1500.0 / 1450.0] * 2 + [k * 1500.0 / 3600.0] * 2, [0.95] * 2 + [1.9] * 2)
    else:
        v, t = inputs.bumpy_ellipsoid(2400)
        mat = None
    nv = len(v)
    rng = np.random.default_rng(nrhs)
    x = rng.standard_normal((nrhs, 2 * nv)) + 1j * rng.standard_normal((nrhs, 2 * nv))
    out = []
    for precision in (B.OSRC_FP32_MATFREE, B.OSRC_FP64_DENSE):
        S = B.Solver(v, t, k, 2.4 * k, 1.9, objects=mat, precision=precision)
        try:
            out.append(S.apply(torch.from_numpy(x).cuda()).cpu().numpy())
        finally:
            S.close()
    for y, ref in zip(*out):
        assert np.linalg.norm(y - ref) < 2.0 * 2.0 ** -24 * np.linalg.norm(ref)
