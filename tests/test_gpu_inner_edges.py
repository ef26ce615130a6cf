"""Inner solves (M^-1, OSRC) at the edges of the mixed kernel's launch shapes:
systems of one thread block and of clusters, one and two rows per thread, rows
with more entries than a thread keeps in registers, two objects; against the
oracle's sparse direct solves.  And the rotations of a GMRES run longer than
one staged tile (512): the residual estimate against the residual of the
returned solution.

Tolerances: the solves stop at a relative residual of 1e-10 with condition
numbers of 10 to 100 (1e-8 and 1e-7, as in the other inner-solver tests); the
estimate agrees with the recomputed residual to the FP32 operator's 1e-6 of
the right-hand side."""
import numpy as np
import pytest

from paper_2104_04609_gb300 import inputs

pytestmark = pytest.mark.gpu


def _bipyramid(m):
    """Double pyramid over an m-gon: two vertices of degree m."""
    a = 2.0 * np.pi * np.arange(m) / m
    v = np.concatenate([np.stack([np.cos(a), np.sin(a), 0 * a], 1), [[0, 0, 1.0], [0, 0, -1.0]]])
    i = np.arange(m)
    t = np.concatenate([np.stack([i, (i + 1) % m, 0 * i + m], 1), np.stack([(i + 1) % m, i, 0 * i + m + 1], 1)])
    return v, t.astype(np.int32)


@pytest.mark.parametrize("kind,nv", [("bipyramid", 5), ("hull", 33), ("bipyramid", 60), ("hull", 768), ("hull", 769),
                                     ("hull", 1280), ("hull", 1281), ("hull", 2600), ("pair", 900)])
def test_mass_and_osrc(kind, nv):
    import scipy.sparse.linalg as sla
    import torch

    import oracle as O
    from paper_2104_04609_gb300 import binding as B

    k0, k1, rho = 3.0, 4.0, 1.5
    objects = None
    if kind == "bipyramid":
        v, t = _bipyramid(nv - 2)
    elif kind == "hull":
        v, t = inputs.fibonacci_hull(nv)
    else:
        v0, t0 = inputs.fibonacci_hull(nv // 2)
        v = np.concatenate([v0, v0 + np.array([4.0, 0, 0])])
        t = np.concatenate([t0, t0 + len(v0)]).astype(np.int32)
        objects = ([k1, k1], [rho, rho])
    rng = np.random.default_rng(nv)
    x = rng.standard_normal(2 * nv) + 1j * rng.standard_normal(2 * nv)
    S = B.Solver(v, t, k0, k1, rho, objects=objects)
    try:
        xt = torch.from_numpy(x).cuda().reshape(1, -1)
        m = S.mass_solve(xt).cpu().numpy().ravel()
        z = S.precond(xt).cpu().numpy().ravel()
    finally:
        S.close()
    M, Sm = O.mass_stiffness(v, t)
    lu = sla.splu(M.tocsc().astype(np.complex128))
    ref = np.concatenate([lu.solve(x[:nv]), lu.solve(x[nv:])])
    assert np.linalg.norm(m - ref) < 1e-8 * np.linalg.norm(ref)
    ke = O.damped_wavenumber(k1, O.mean_edge_length(v, t))
    ref = np.concatenate(O.osrc_apply(M, Sm, x[:nv], x[nv:], k1, ke, 4, np.pi / 3))
    assert np.linalg.norm(z - ref) < 1e-7 * np.linalg.norm(ref)


def test_long_arnoldi():
    import torch

    from paper_2104_04609_gb300 import binding as B

    v, t = inputs.fibonacci_hull(1500)
    S = B.Solver(v, t, 40.0, 55.0, 1.5, precond=B.OSRC_PRECOND_MASS)
    try:
        b = S.rhs_planewave([[0.0, 0.0, 1.0]])
        x, info = S.solve(b, tol=1e-12, maxit=600, raise_on_nonconvergence=False)
        assert info.iterations == 600
        r = S.mass_solve(b - S.apply(x))
        res = float(torch.linalg.norm(r) / torch.linalg.norm(S.mass_solve(b)))
    finally:
        S.close()
    assert abs(res - info.precond_residual) < 0.02 * res + 1e-5, (res, info.precond_residual)
