"""Far field with each pair of triangles evaluated once (2048 triangles on):
numbers of 128-triangle groups odd and even, full and ragged; several launches
over the group offsets; objects, the Mueller formulation, attenuation and large
phases, against the FP64 assembled operator of the same discretisation; the
same bits from call to call, on memory that other arrays have used.

Tolerance: FP32 evaluation of sums over up to 1.2e5 source points (unit roundoff
6e-8, phases k r below 32 pi in the plain variant): 1e-5, as for the operator's
other tests."""
import numpy as np
import pytest

from paper_2104_04609_gb300 import inputs

pytestmark = pytest.mark.gpu


def _err(y, ref):
    n = ref.shape[-1] // 2
    return max(np.linalg.norm(y[:n] - ref[:n]) / np.linalg.norm(ref[:n]),
               np.linalg.norm(y[n:] - ref[n:]) / np.linalg.norm(ref[n:]))


def _both(v, t, k0, k1, rho, **kw):
    import torch

    from paper_2104_04609_gb300 import binding as B

    rng = np.random.default_rng(len(v))
    x = rng.standard_normal((1, 2 * len(v))) + 1j * rng.standard_normal((1, 2 * len(v)))
    out = []
    for precision in (B.OSRC_FP32_MATFREE, B.OSRC_FP64_DENSE):
        S = B.Solver(v, t, k0, k1, rho, precision=precision, **kw)
        try:
            out.append(S.apply(torch.from_numpy(x).cuda()).cpu().numpy().ravel())
        finally:
            S.close()
    return out


# 16 full groups; 16 and 17 with a ragged last one of 4 (below the rule: 2046); 17 full
@pytest.mark.parametrize("nv", [1025, 1026, 1028, 1090, 1155])
@pytest.mark.parametrize("k", [3.0, 60.0])
def test_groups(nv, k):
    v, t = inputs.fibonacci_hull(nv)
    y, ref = _both(v, t, k, 1.3 * k, 1.5)
    assert _err(y, ref) < 1e-5


@pytest.mark.parametrize("k", [3.0, 40.0])
@pytest.mark.parametrize("kind", ["objects", "objects_att", "muller", "att"])
def test_materials(k, kind):
    from paper_2104_04609_gb300 import binding as B

    if kind.startswith("objects"):
        v, t = inputs.fibonacci_hull(530)
        v, t = np.vstack([v - [2.0, 0, 0], v + [2.0, 0, 0]]), np.vstack([t, t + len(v)])
        k1 = [1.3 * k, 0.8 * k]
        y, ref = _both(v, t, k, None, None, objects=(k1, [1.5, 0.8]), k_int_im=0.2 if kind == "objects_att" else 0.0)
    else:
        v, t = inputs.fibonacci_hull(1100)
        if kind == "muller":
            y, ref = _both(v, t, k, 1.3 * k, 1.5, formulation=B.OSRC_MULLER)
        else:
            y, ref = _both(v, t, k, 1.3 * k, 1.5, k_int_im=0.2)
    assert _err(y, ref) < 1e-5


def test_launches_and_bits():
    """160 groups take several launches; repeated applies give the same bits,
    also after other arrays have filled the device's free memory, and rows of
    the FP64 oracle."""
    import torch

    import oracle as O
    from paper_2104_04609_gb300 import binding as B

    v, t = inputs.icosphere(5)
    nv, k0, k1, rho = len(v), 2.0, 3.0, 1.5
    rng = np.random.default_rng(1)
    x = rng.standard_normal((5, 2 * nv)) + 1j * rng.standard_normal((5, 2 * nv))
    xs = torch.from_numpy(x).cuda()
    rows = rng.integers(0, nv, 3)
    R1, R2 = O.pmchwt_rows(v, t, k0, k1, rho, rows, nss=4)
    filled = [torch.full((1 << 26,), 1e3, device="cuda") for _ in range(4)]
    del filled
    torch.cuda.empty_cache()
    S = B.Solver(v, t, k0, k1, rho)
    try:
        for r in (1, 3, 5):
            y = [S.apply(xs[:r].clone()).cpu().numpy() for _ in range(12)]
            assert all(np.array_equal(y[0], z) for z in y[1:])
            for i in range(r):
                for got, ref in ((y[0][i, rows], R1 @ x[i]), (y[0][i, nv + rows], R2 @ x[i])):
                    assert np.abs(got - ref).max() / np.abs(ref).max() < 1e-5
    finally:
        S.close()


@pytest.mark.parametrize("nv", [1155, 2100])
def test_memory_budget(nv):
    """A context with a memory budget gives the partial sums less room (more
    launches): the same operator."""
    import torch

    from paper_2104_04609_gb300 import binding as B

    v, t = inputs.fibonacci_hull(nv)
    rng = np.random.default_rng(nv)
    x = torch.from_numpy(rng.standard_normal((3, 2 * nv)) + 1j * rng.standard_normal((3, 2 * nv))).cuda()
    out = []
    for budget in (0, 1 << 33):
        S = B.Solver(v, t, 3.0, 4.0, 1.5, mem_budget_bytes=budget)
        try:
            out.append((S.apply(x[:1]).cpu().numpy(), S.apply(x).cpu().numpy()))
        finally:
            S.close()
    for a, b in zip(*out):
        for r in range(len(a)):
            assert _err(b[r], a[r]) < 1e-5
