"""Inner solves (M^-1, OSRC) on meshes with vertices of high degree, whose rows
have more entries than a thread of the mixed kernel keeps in registers: poles of
UV spheres and bipyramids up to degree 3000, in one block and in clusters;
against the oracle's sparse direct solves.

Tolerances: a relative residual of 1e-10 bounds the relative error by that times
the condition number of the system; the OSRC sums add ten solutions of the
hardest system's condition or less, a factor of 10."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _bipyramid(m):
    a = 2.0 * np.pi * np.arange(m) / m
    v = np.concatenate([np.stack([np.cos(a), np.sin(a), 0 * a], 1), [[0, 0, 1.0], [0, 0, -1.0]]])
    i = np.arange(m)
    t = np.concatenate([np.stack([i, (i + 1) % m, 0 * i + m], 1), np.stack([(i + 1) % m, i, 0 * i + m + 1], 1)])
    return v, t.astype(np.int32)


def _uv_sphere(rings, seg):
    th = np.pi * np.arange(1, rings) / rings
    ph = 2 * np.pi * np.arange(seg) / seg
    ring = np.stack([np.outer(np.sin(th), np.cos(ph)), np.outer(np.sin(th), np.sin(ph)),
                     np.outer(np.cos(th), np.ones(seg))], -1).reshape(-1, 3)
    v = np.concatenate([[[0, 0, 1.0]], ring, [[0, 0, -1.0]]])
    s = np.arange(seg)
    n = (s + 1) % seg
    t = [np.stack([0 * s, 1 + s, 1 + n], 1)]
    for r in range(rings - 2):
        a, b = 1 + r * seg, 1 + (r + 1) * seg
        t += [np.stack([a + s, b + s, b + n], 1), np.stack([a + s, b + n, a + n], 1)]
    last = 1 + (rings - 2) * seg
    t.append(np.stack([0 * s + len(v) - 1, last + n, last + s], 1))
    return v, np.concatenate(t).astype(np.int32)


def _solve(v, t, k1, precond=True):
    import torch

    from paper_2104_04609_gb300 import binding as B

    nv = len(v)
    rng = np.random.default_rng(nv)
    x = rng.standard_normal(2 * nv) + 1j * rng.standard_normal(2 * nv)
    S = B.Solver(v, t, 3.0, k1, 1.5)
    try:
        xt = torch.from_numpy(x).cuda().reshape(1, -1)
        m = S.mass_solve(xt).cpu().numpy().ravel()
        z = S.precond(xt).cpu().numpy().ravel() if precond else None
    finally:
        S.close()
    return x, m, z


@pytest.mark.parametrize("kind,size", [("bipyramid", (7,)), ("bipyramid", (8,)), ("bipyramid", (200,)),
                                       ("uv", (16, 8)), ("uv", (24, 60)), ("uv", (6, 200))])
def test_mass_and_osrc(kind, size):
    import scipy.sparse.linalg as sla

    import oracle as O

    v, t = _bipyramid(*size) if kind == "bipyramid" else _uv_sphere(*size)
    nv, k1 = len(v), 4.0
    x, m, z = _solve(v, t, k1)
    M, Sm = O.mass_stiffness(v, t)
    lu = sla.splu(M.tocsc().astype(np.complex128))
    ref = np.concatenate([lu.solve(x[:nv]), lu.solve(x[nv:])])
    assert np.linalg.norm(m - ref) < 1e-10 * np.linalg.cond(M.toarray()) * np.linalg.norm(ref)
    ke = O.damped_wavenumber(k1, O.mean_edge_length(v, t))
    ref = np.concatenate(O.osrc_apply(M, Sm, x[:nv], x[nv:], k1, ke, 4, np.pi / 3))
    cond = np.linalg.cond((M - Sm / ke ** 2).toarray())
    assert np.linalg.norm(z - ref) < 1e-9 * cond * np.linalg.norm(ref)


def test_mass_degree_3000():
    """Two rows of 3001 entries, shared memory mostly theirs."""
    import scipy.sparse.linalg as sla

    import oracle as O

    v, t = _bipyramid(3000)
    x, m, _ = _solve(v, t, 4.0, precond=False)
    M, _ = O.mass_stiffness(v, t)
    lu = sla.splu(M.tocsc().astype(np.complex128))
    ref = np.concatenate([lu.solve(x[:len(v)]), lu.solve(x[len(v):])])
    assert np.linalg.norm(m - ref) < 1e-10 * np.linalg.cond(M.toarray()) * np.linalg.norm(ref)
