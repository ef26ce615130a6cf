"""Calls whose device memory runs out, on a context with a budget: they return
OSRC_OUT_OF_MEMORY, again when repeated, and leave the handle as it was, so
that an apply still gives the same bits and the call itself succeeds once
there is room."""
import contextlib

import numpy as np
import pytest

from paper_2104_04609_gb300 import inputs

pytestmark = pytest.mark.gpu

BUDGET = 1 << 27


@contextlib.contextmanager
def _filled(B, S, leave):
    """Takes up the context's budget but for about `leave` bytes (by meshes)."""
    meshes = []
    try:
        for nv in (20000, 2000, 200, 20):
            v, t = inputs.fibonacci_hull(nv)
            while True:
                before = B.osrc_mem_used(S.ctx)
                if before + 160 * nv > BUDGET - leave:  # a mesh takes about 96 bytes a vertex
                    break
                meshes.append(B.osrc_mesh_create(S.ctx, v, t))
                assert B.osrc_mem_used(S.ctx) - before <= 160 * nv
        yield
    finally:
        for m in meshes:
            B.osrc_mesh_destroy(m)


def _runs_out(B, S, call, leave):
    """call() fails twice with the budget nearly used up, the one-vector apply
    is undisturbed in between, and afterwards call() succeeds."""
    import torch

    rng = np.random.default_rng(3)
    n = 2 * S.nv
    x = torch.from_numpy(rng.standard_normal((1, n)) + 1j * rng.standard_normal((1, n))).cuda()
    ref = S.apply(x).cpu().numpy()
    with _filled(B, S, leave):
        for _ in range(2):
            with pytest.raises(B.OsrcError) as e:
                call()
            assert e.value.status == B.OSRC_OUT_OF_MEMORY
            assert np.array_equal(S.apply(x).cpu().numpy(), ref)
    return call()


@pytest.mark.parametrize("leave", [1 << 12, 1 << 18])
def test_field(leave):
    """Neither the source points' data (168 KB) nor the regions of 2e5 targets fit."""
    import torch

    import oracle as O
    from paper_2104_04609_gb300 import binding as B

    v, t = inputs.fibonacci_hull(150)
    pts = np.random.default_rng(1).standard_normal((200000, 3))
    pts *= 3.0 / np.linalg.norm(pts, axis=1)[:, None]
    S = B.Solver(v, t, 2.0, 3.0, 1.5, mem_budget_bytes=BUDGET)
    try:
        x = torch.from_numpy(np.random.default_rng(2).standard_normal(2 * S.nv) + 0j).cuda()
        p = torch.from_numpy(pts).cuda()
        u = torch.zeros(len(pts), dtype=torch.complex128, device="cuda")
        _runs_out(B, S, lambda: B.osrc_field_eval(S.pb, x, p, u, B.OSRC_INC_PLANEWAVE, [0, 0, 1.0]),
                  leave)
        got = u[:50].cpu().numpy()
    finally:
        S.close()
    ref = O.field(v, t, 2.0, 3.0, 1.5, x.cpu().numpy(), pts[:50])[0]
    assert np.abs(got - ref).max() < 1e-10 * np.abs(ref).max()


# leave: nothing of the several-vector buffers, their densities only (1.5 MB),
# all but the partial sums (44 MB)
@pytest.mark.parametrize("leave", [1 << 14, 1 << 20, 3 << 20])
@pytest.mark.parametrize("nv,nrhs", [(1155, 3), (1155, 8), (1155, 9)])
def test_several_vectors(nv, nrhs, leave):
    import torch

    from paper_2104_04609_gb300 import binding as B

    v, t = inputs.fibonacci_hull(nv)
    rng = np.random.default_rng(nv + nrhs)
    S = B.Solver(v, t, 3.0, 4.0, 1.5, mem_budget_bytes=BUDGET)
    try:
        x = torch.from_numpy(rng.standard_normal((nrhs, 2 * nv)) + 1j * rng.standard_normal((nrhs, 2 * nv))).cuda()
        y = _runs_out(B, S, lambda: S.apply(x), leave).cpu().numpy()
        one = np.concatenate([S.apply(x[r:r + 1]).cpu().numpy() for r in range(nrhs)])
    finally:
        S.close()
    assert np.linalg.norm(y - one) < 1e-5 * np.linalg.norm(one)


def test_one_vector_beside_several():
    """A captured one-vector apply is replayed after the first several-vector
    apply, and the two run on streams of their own: the same bits as alone."""
    import torch

    from paper_2104_04609_gb300 import binding as B

    v, t = inputs.fibonacci_hull(1155)
    rng = np.random.default_rng(5)
    S = B.Solver(v, t, 3.0, 4.0, 1.5)
    try:
        x = torch.from_numpy(rng.standard_normal((4, 2 * S.nv)) + 1j * rng.standard_normal((4, 2 * S.nv))).cuda()
        x1, y1 = x[:1].clone(), torch.empty_like(x[:1])
        ref1 = S.apply(x1).cpu().numpy()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            B.osrc_pmchwt_apply(S.pb, x1, y1)
        refm = S.apply(x).cpu().numpy()
        g.replay()
        assert np.array_equal(y1.cpu().numpy(), ref1)
        s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
        ym = torch.empty_like(x)
        for _ in range(10):
            y1.zero_()
            ym.zero_()
            torch.cuda.synchronize()
            B.osrc_pmchwt_apply(S.pb, x, ym, 4, stream=s1)
            B.osrc_pmchwt_apply(S.pb, x1, y1, 1, stream=s2)
            torch.cuda.synchronize()
            assert np.array_equal(ym.cpu().numpy(), refm) and np.array_equal(y1.cpu().numpy(), ref1)
    finally:
        S.close()


# the basis (101 KB) does not fit, or one of the vectors of 4800 bytes after it
@pytest.mark.parametrize("leave", [1 << 12, 111000, 115000, 120000, 125000])
def test_solve(leave):
    import torch

    from paper_2104_04609_gb300 import binding as B

    v, t = inputs.fibonacci_hull(150)
    S, T = (B.Solver(v, t, 2.0, 3.0, 1.5, mem_budget_bytes=b) for b in (BUDGET, 0))
    try:
        b = S.rhs_planewave([[0.0, 0.0, 1.0]])
        x, info = _runs_out(B, S, lambda: S.solve(b, tol=1e-6, maxit=20, raise_on_nonconvergence=False), leave)
        ref, _ = T.solve(b, tol=1e-6, maxit=20, raise_on_nonconvergence=False)
        assert torch.equal(x, ref)
        # growing the basis fails: the old one is gone, and the shorter solve makes it again
        with _filled(B, S, 1 << 12):
            with pytest.raises(B.OsrcError) as e:
                S.solve(b, tol=1e-6, maxit=4000)
            assert e.value.status == B.OSRC_OUT_OF_MEMORY
            x, _ = S.solve(b, tol=1e-6, maxit=20, raise_on_nonconvergence=False)
        assert torch.equal(x, ref)
    finally:
        S.close()
        T.close()


# successive buffers of the packed system and of the block workspaces
@pytest.mark.parametrize("leave", [1 << 14, 600000, 1960000, 2300000, 3000000, 3420000])
def test_dense_batched(leave):
    import torch

    from paper_2104_04609_gb300 import binding as B

    v, t = inputs.fibonacci_hull(150)
    S, T = (B.Solver(v, t, 2.0, 3.0, 1.5, mem_budget_bytes=b, precision=B.OSRC_FP64_DENSE) for b in (BUDGET, 0))
    try:
        b = S.rhs_planewave(inputs.plane_wave_dirs(5, seed=2))
        x, ref = torch.empty_like(b), torch.empty_like(b)
        _runs_out(B, S, lambda: B.osrc_dense_batched_solve(S.pb, b, x, tol=1e-8, inner_maxit=40), leave)
        B.osrc_dense_batched_solve(T.pb, b, ref, tol=1e-8, inner_maxit=40)
        assert torch.equal(x, ref)
        # a larger block fails: the next smaller one makes its workspace again
        b2 = S.rhs_planewave(inputs.plane_wave_dirs(64, seed=3))
        with _filled(B, S, 1 << 14):
            with pytest.raises(B.OsrcError) as e:
                B.osrc_dense_batched_solve(S.pb, b2, torch.empty_like(b2), tol=1e-8, inner_maxit=40)
            assert e.value.status == B.OSRC_OUT_OF_MEMORY
            B.osrc_dense_batched_solve(S.pb, b, x.zero_(), tol=1e-8, inner_maxit=40)
        assert torch.equal(x, ref)
    finally:
        S.close()
        T.close()


@pytest.mark.parametrize("objects", [1, 2])
@pytest.mark.parametrize("npts", [1, 1000, 20000])
def test_field_without_room_for_splits(npts, objects):
    """Room for the source points only: the field is evaluated without splits
    over the sources, the regions the same and the values to FP64 rounding of
    sums of up to 3528 terms (3528 x 1.1e-16 of their size, 4e-13)."""
    import torch

    from paper_2104_04609_gb300 import binding as B

    v, t = inputs.fibonacci_hull(150)
    obj = None
    if objects == 2:
        v, t = np.concatenate([v - [2.0, 0, 0], v + [2.0, 0, 0]]), np.concatenate([t, t + len(v)]).astype(np.int32)
        obj = ([3.0, 1.2], [1.5, 0.8])
    rng = np.random.default_rng(npts)
    pts = rng.standard_normal((npts, 3))
    pts *= (np.where(rng.random(npts) < 0.5, 0.15, 6.0) / np.linalg.norm(pts, axis=1))[:, None]
    if objects == 2:
        pts[:, 0] += np.where(np.linalg.norm(pts, axis=1) < 1.0, rng.choice([-2.0, 2.0], npts), 0.0)
    S, T = (B.Solver(v, t, 2.0, 3.0, 1.5, mem_budget_bytes=b, objects=obj) for b in (BUDGET, 0))
    try:
        x = torch.from_numpy(rng.standard_normal(2 * S.nv) + 1j * rng.standard_normal(2 * S.nv)).cuda()
        p = torch.from_numpy(pts).cuda()
        with _filled(B, S, 6 * len(t) * 96 + 64):
            u, reg = S.field(x, p, B.OSRC_INC_PLANEWAVE, [0, 0, 1.0])
        ref, regref = T.field(x, p, B.OSRC_INC_PLANEWAVE, [0, 0, 1.0])
        assert torch.equal(reg, regref)
        assert float((u - ref).abs().max() / ref.abs().max()) < 4e-13
    finally:
        S.close()
        T.close()
