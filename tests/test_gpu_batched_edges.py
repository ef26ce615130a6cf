"""Edges of the batched solve's block kernels: numbers of right-hand sides whose
padded block width does and does not divide the threads of a block, the
narrowest and the widest block, and inner iteration limits that end a cycle
before and at convergence.

Tolerances: the refinement stops on a true residual of 1e-10; the solution then
agrees with the direct one to cond(A) times that (below 1e2 for this mesh and
these wavenumbers): 1e-8, as for the solve's other tests."""
import numpy as np
import pytest

import oracle as O
from paper_2104_04609_gb300.inputs import fibonacci_hull, plane_wave_dirs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def system():
    import __graft_entry__

    __graft_entry__.build()
    from paper_2104_04609_gb300 import binding as B

    v, t = fibonacci_hull(150)
    S = B.Solver(v, t, 2.0, 3.0, 1.5, precision=B.OSRC_FP64_DENSE)
    yield B, S, O.pmchwt_matrix(v, t, 2.0, 3.0, 1.5, nss=S.params.n_ss)
    S.close()


# one refinement's inner limit: 9 and 12 iterations (the limit ends cycles), 65
# and 200 (convergence does; 65 is past one tile of the rotations' staging)
@pytest.mark.parametrize("nrhs,inner_maxit", [(1, 200), (7, 65), (20, 200), (20, 9), (65, 65), (128, 200), (128, 12)])
@pytest.mark.parametrize("inner_tol", [1e-3, 1e-5])
def test_batched_block_widths(system, nrhs, inner_maxit, inner_tol):
    B, S, A = system
    b = S.rhs_planewave(plane_wave_dirs(nrhs, seed=100 + nrhs))
    b[nrhs // 2] *= 1e6  # columns of unlike sizes
    x = torch.zeros_like(b)
    info = B.osrc_dense_batched_solve(S.pb, b, x, tol=1e-10, max_refine=100, inner_tol=inner_tol,
                                      inner_maxit=inner_maxit)
    assert info["residual"] <= 1e-10
    xs = x.cpu().numpy()
    ref = np.linalg.solve(A, b.cpu().numpy().T).T
    err = np.linalg.norm(xs - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert err.max() < 1e-8, err.max()
