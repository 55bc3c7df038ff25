"""The FP32 Gram sums P^T A P and P^T r, taken with the product A P or in a
launch of their own, through the updates they determine: x_1 = P alpha with
alpha = (P^T A P)^+ P^T r, and x_2, whose second block is A-orthogonalised
against the first.  (The residual follows x for any alpha, so a point counted
twice or a warp left out would only slow a solve down.)

Bars (set before the first run).  x_1 is the A-orthogonal projection onto the
columns, so a relative perturbation eta of the columns and their products moves
it by a few times kappa eta, with kappa the condition of the scaled Gram matrix;
rounding a smooth column to FP32 perturbs it by up to nodes u in the A-norm, u =
2^-24.  Hence 4 kappa nodes u for x_1, and four times that for x_2.  In the oracle,
with the structured grids below, an overlap of two groups a warp that is counted
twice or a lane left out moves x_1 by 15 to 1000 times the bar, a single segment
left out by 5 to 9000 times (a twentieth at 129^3, one of 18,163).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import amg as oamg
from oracle import mg as omg
from oracle import mpcg as ompcg
from paper_2402_12833_gb300 import problems as pb

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


@pytest.fixture(scope="module")
def M():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_12833_gb300 import build, mpcg
    build.build()
    mpcg.load()
    return mpcg


def _check(M, H, O, A, b, nodes):
    Z = O.mg_columns(b)
    G = Z.T @ (A @ Z)
    d = 1 / np.sqrt(np.diag(G))
    bar = 4 * np.linalg.cond(d[:, None] * G * d) * nodes * U
    bd = torch.from_numpy(b).cuda()
    for k in (1, 2):
        x = torch.zeros_like(bd)
        status, its, _, _ = H.solve(bd, x, rtol=1e-14, maxit=k, histories=False)
        ref = ompcg.mpcg(A, b, O.mg_columns, rtol=0.0, maxit=k).x
        err = np.linalg.norm(x.cpu().numpy() - ref) / np.linalg.norm(ref)
        assert status == M.MPCG_NOT_CONVERGED and its == k
        assert err <= (bar if k == 1 else 4 * bar), (k, err, bar)


GRIDS = [
    (3, 21, 3, 0x3F),     # ragged rows: warps overlap by two groups
    (3, 37, 3, 0x15),
    (3, 45, 3, 0x3F),
    (3, 33, 4, 0x3F),     # whole rows fill the warps
    (3, 65, 6, 0x15),     # six columns: the most that keep P's rows in registers
    (3, 81, 4, 0x3F),     # past the size up to which the stored stencil's product takes the sums
    (2, 97, 5, 0x3F),
    (2, 65, 5, 0x3F),
    (2, 129, 7, 0x5),     # seven columns: P's rows are read again for the sums
    (2, 257, 8, 0x5),
    (2, 513, 9, 0x5),
    (2, 1025, 10, 0x5)]   # ten columns


@pytest.mark.parametrize("dim,nodes,levels,faces,operator",
                         [g + (o,) for g in GRIDS for o in ("half", "kappa", "full")] + [(3, 129, 7, 0x15, "kappa")])
def test_structured_products(M, dim, nodes, levels, faces, operator):
    kap = 10.0 ** np.random.default_rng(1).uniform(-1, 1, (nodes - 1,) * dim)
    st = pb.assemble_diffusion(dim, nodes, kappa=kap, faces=faces)
    b = pb.normal(2, int(np.prod(pb.grid_shape(dim, nodes, faces))))
    H = M.Hierarchy(torch.from_numpy(np.ascontiguousarray(st)).cuda(), dim, nodes, levels, faces=faces,
                    precision=M.MPCG_MIXED, half_stencil=0 if operator == "full" else 1)
    if operator == "kappa":
        M.mg_attach_q1_kappa(H.h, torch.from_numpy(np.ascontiguousarray(kap)).reshape(-1).cuda())
    O = omg.Hierarchy(dim, None, st, levels, nodes=nodes, faces=faces)
    _check(M, H, O, O.A[-1], b, nodes)


@pytest.mark.parametrize("nodes,amg", [
    (65, dict(coarse_size=20)), (193, dict(coarse_size=20)), (129, dict(coarse_size=4, max_levels=8))])
def test_sparse_product(M, nodes, amg):
    A = pb.stencil_csr(pb.fracture_network(1e2, nodes=nodes))
    A.sort_indices()
    O = oamg.AlgebraicHierarchy(A, **amg)
    H = M.AlgebraicHierarchy(A, precision=M.MPCG_MIXED, **amg)
    _check(M, H, O, A, pb.normal(3, A.shape[0]), nodes)
