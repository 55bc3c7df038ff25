"""A hierarchy of one grid: every preconditioner is the exact solve on it, the
additive columns, their sum and the V-cycle alike, so that one update solves the
system (FP64 and double-word; the mixed solve refines).

Bars: the correction agrees with a dense FP64 solve to 1e-11 (the explicit
inverse of a matrix of condition below 1e3), the solution's residual with the
tolerance 1e-8 of the solve."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mg as omg
from paper_2402_12833_gb300 import problems as pb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_12833_gb300 import build, mpcg
    build.build()
    mpcg.load()
    return mpcg


@pytest.mark.parametrize("kind", ["stencil", "ssor", "sparse"])
@pytest.mark.parametrize("opts", [dict(), dict(sum_columns=1, m=1), dict(vcycle=1, m=1)])
@pytest.mark.parametrize("precision", ["fp64", "fp64_dw", "mixed"])
def test_one_grid_is_the_exact_solve(M, kind, opts, precision):
    prec = {"fp64": M.MPCG_FP64, "fp64_dw": M.MPCG_FP64_DW, "mixed": M.MPCG_MIXED}[precision]
    prob = pb.poisson_random(2, 17, 2)
    A = omg.Hierarchy(2, None, prob.stencil, 1, nodes=17, faces=prob.faces).A[-1]
    if kind == "sparse":
        H = M.AlgebraicHierarchy(pb.stencil_csr(prob), max_levels=1, precision=prec, **opts)
    else:
        smoother = M.MPCG_SMOOTHER_SSOR if kind == "ssor" else M.MPCG_SMOOTHER_JACOBI
        H = M.Hierarchy(torch.from_numpy(np.ascontiguousarray(prob.stencil)).cuda(), 2, 17, 1, precision=prec,
                        smoother=smoother, **opts)
    b = torch.from_numpy(prob.b).cuda()
    want = np.linalg.solve(A.toarray(), prob.b)
    z = torch.zeros((1, b.numel()), dtype=torch.float64, device="cuda")
    M.mg_corrections(H.h, b, z)
    assert np.abs(z[0].cpu().numpy() - want).max() <= 1e-11 * np.abs(want).max()
    x = torch.zeros_like(b)
    status, its, _, _ = H.solve(b, x, rtol=1e-8, maxit=20, histories=False)
    assert status == M.MPCG_OK and its <= (1 if precision != "mixed" else 4)
    assert np.linalg.norm(prob.b - A @ x.cpu().numpy()) <= 1.01e-8 * np.linalg.norm(prob.b)
