"""The kernels at the sizes where their index arithmetic changes form: rows
that end inside a warp or a 128-point segment, rows longer than a block, grids
just below and above the size at which a smoothing becomes two launches or a
restriction chain stops, coarsest grids beyond the tail's dense part, the widest
blocks, small algebraic grids, and the learned column's partial batches.

Bars (set before the first run).  FP32 products: |y - A x| <= 64 u |A||x|
entrywise, u = 2^-24 (at most 27 products and roundings).  FP64 columns: 1e-12 of
a column's largest entry, FP32 columns: 2e-5 (two sweeps, transfers and a dense
coarse solve of well-conditioned grids).  Solves: the true residual, taken with
the oracle's operator, within the tolerance, and the oracle's count within one.
Learned column: equal bits where only the workspace differs, 1e-4 of the
gradient's norm for a batch against its images (the split of dL/dy into two
bfloat16 keeps 16 bits), 1e-6 for losses.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import amg as oamg
from oracle import learned as OL
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


def _problem(dim, nodes, levels, faces=0x3F, seed=1):
    kap = 10.0 ** np.random.default_rng(seed).uniform(-1, 1, (nodes - 1,) * dim)
    st = pb.assemble_diffusion(dim, nodes, kappa=kap, faces=faces)
    n = int(np.prod(pb.grid_shape(dim, nodes, faces)))
    return pb.Problem(dim, nodes, levels, st, pb.normal(seed + 1, n), kappa=kap, name="edge", faces=faces)


def _pair(M, prob, precision, **opts):
    st = torch.from_numpy(np.ascontiguousarray(prob.stencil)).cuda()
    H = M.Hierarchy(st, prob.dim, prob.nodes, prob.levels, faces=prob.faces, precision=precision, **opts)
    return H, omg.Hierarchy(prob.dim, None, prob.stencil, prob.levels, nodes=prob.nodes, faces=prob.faces)


def _columns(call, H, O, n, levels, bar):
    r = pb.normal(9, n)
    Z = torch.zeros((levels, n), dtype=torch.float64, device="cuda")
    call(H.h, torch.from_numpy(r).cuda(), Z)
    got, ref = Z.cpu().numpy(), O.mg_columns(r)
    for l in range(levels):
        assert np.abs(got[l] - ref[:, l]).max() <= bar * np.abs(ref[:, l]).max(), l


@pytest.mark.parametrize("dim,nodes,levels,faces", [
    (2, 9, 2, 0x3F),      # a row of 7 points: several rows to a warp
    (2, 35, 2, 0x1),      # 33 and 34 points: one past a warp
    (2, 129, 6, 0x3C),    # 129 points: one past a segment
    (2, 273, 5, 0x5),     # free faces, two segments and a rest
    (3, 5, 2, 0x3F),
    (3, 13, 3, 0x2A),     # free faces
    (3, 37, 3, 0x3F),
    (3, 49, 4, 0x15)])
def test_f32_products_and_columns(M, dim, nodes, levels, faces):
    prob = _problem(dim, nodes, levels, faces)
    H, O = _pair(M, prob, M.MPCG_MIXED)
    A = O.A[-1]
    for c in (1, 4, 7, 12):
        X = pb.normal(50 + c, c * prob.b.size).reshape(c, -1)
        Y = torch.zeros((c, prob.b.size), dtype=torch.float64, device="cuda")
        M.mg_apply_operator_f32(H.h, levels - 1, torch.from_numpy(X).cuda(), Y, c)
        err, bound = np.abs(Y.cpu().numpy() - (A @ X.T).T), (abs(A) @ np.abs(X).T).T
        assert np.all(err <= 64 * U * bound), (c, float((err / bound).max()))
    _columns(M.mg_corrections_f32, H, O, prob.b.size, levels, 2e-5)


@pytest.mark.parametrize("dim,nodes,levels,faces", [
    (2, 17, 4, 0x3F),     # the whole cycle below the tail
    (2, 49, 2, 0x3F),     # coarsest grid of 529 unknowns: a launch of its own
    (2, 97, 5, 0x1),      # a restriction chain that ends inside a group
    (2, 289, 6, 0x3F),    # rows longer than a block, two-launch smoothing
    (2, 545, 6, 0x5),
    (3, 21, 2, 0x3F),
    (3, 41, 4, 0x3F),     # below 2^16 points
    (3, 49, 5, 0x2A)])    # above
def test_fp64_columns(M, dim, nodes, levels, faces):
    prob = _problem(dim, nodes, levels, faces)
    H, O = _pair(M, prob, M.MPCG_FP64)
    _columns(M.mg_corrections, H, O, prob.b.size, levels, 1e-12)


@pytest.mark.parametrize("precision", ["fp64", "fp64_dw", "mixed"])
@pytest.mark.parametrize("dim,nodes,levels,m", [
    (2, 129, 7, 10),      # a window of 70 directions
    (2, 257, 8, 3),
    (2, 513, 9, 1),       # no window
    (3, 41, 4, 12),       # the widest window
    (3, 49, 5, 2)])
def test_solves_with_wide_blocks_and_windows(M, precision, dim, nodes, levels, m):
    st = pb.assemble_diffusion(dim, nodes)
    n = (nodes - 2) ** dim
    prob = pb.Problem(dim, nodes, levels, st, pb.normal(3, n), name="edge")
    H, O = _pair(M, prob, {"fp64": M.MPCG_FP64, "fp64_dw": M.MPCG_FP64_DW, "mixed": M.MPCG_MIXED}[precision], m=m)
    b = torch.from_numpy(prob.b).cuda()
    x = torch.zeros_like(b)
    status, k, _, _ = H.solve(b, x, rtol=1e-8, maxit=200)
    assert status == M.MPCG_OK
    assert np.linalg.norm(prob.b - O.A[-1] @ x.cpu().numpy()) <= 1.01e-8 * np.linalg.norm(prob.b)
    if precision != "mixed":   # whose restarts add iterations
        ref = ompcg.mpcg(O.A[-1], prob.b, O.mg_columns, m=m, rtol=1e-8, maxit=200)
        assert abs(k - ref.iters) <= 1, (k, ref.iters)


def test_solve_with_the_widest_block(M):
    """Twelve grids (4097 nodes per side): a block of twelve columns."""
    prob = pb.Problem(2, 4097, 12, pb.assemble_diffusion(2, 4097), pb.normal(3, 4095 ** 2), name="edge")
    H = M.Hierarchy(torch.from_numpy(np.ascontiguousarray(prob.stencil)).cuda(), 2, 4097, 12, m=1,
                    precision=M.MPCG_MIXED)
    b = torch.from_numpy(prob.b).cuda()
    x, y = torch.zeros_like(b), torch.zeros_like(b)
    status, _, _, _ = H.solve(b, x, rtol=1e-8, maxit=200, histories=False)
    M.mg_apply_operator(H.h, 11, x, y, 1)
    assert status == M.MPCG_OK and (b - y).norm() <= 1.01e-8 * b.norm()


@pytest.mark.parametrize("dim,nodes,count", [(2, 65, 24), (2, 129, 8), (3, 33, 5)])
def test_mixed_batch_equals_single_solves_bitwise(M, dim, nodes, count):
    """Grids whose smoothing takes another width in a batch than alone."""
    probs = [pb.diffusion_macro(dim, nodes, 300 + i, rhs="normal", rhs_seed=400 + i) for i in range(count)]
    dev = [torch.from_numpy(np.ascontiguousarray(p.stencil)).cuda() for p in probs]
    B = M.BatchedHierarchy(dev, dim, nodes, probs[0].levels, precision=M.MPCG_MIXED)
    b = torch.from_numpy(np.stack([p.b for p in probs])).cuda()
    x = torch.zeros_like(b)
    status, its = B.solve(b, x, rtol=1e-8, maxit=2000)
    assert status == M.MPCG_OK
    for i in range(count):
        H = M.Hierarchy(dev[i], dim, nodes, probs[0].levels, precision=M.MPCG_MIXED)
        xs = torch.zeros_like(b[i])
        status, k, _, _ = H.solve(b[i].contiguous(), xs, rtol=1e-8, maxit=2000)
        assert status == M.MPCG_OK and its[i] == k and torch.equal(x[i], xs), i


@pytest.mark.parametrize("nodes,faces", [(21, 0x3F), (21, 0x2A), (37, 0x15), (45, 0x3F)])
def test_matrix_free_rows(M, nodes, faces):
    """Ragged rows through the operator rebuilt from kappa, with its Gram sums."""
    prob = _problem(3, nodes, 3, faces)
    H, O = _pair(M, prob, M.MPCG_MIXED)
    M.mg_attach_q1_kappa(H.h, torch.from_numpy(np.ascontiguousarray(prob.kappa)).reshape(-1).cuda())
    b = torch.from_numpy(prob.b).cuda()
    x = torch.zeros_like(b)
    status, _, _, _ = H.solve(b, x, rtol=1e-8, maxit=500)
    assert status == M.MPCG_OK
    assert np.linalg.norm(prob.b - O.A[-1] @ x.cpu().numpy()) <= 1.01e-8 * np.linalg.norm(prob.b)


@pytest.mark.parametrize("nodes,amg", [
    (33, dict(max_levels=2)),                     # the finest grid takes the dense correction
    (65, dict(max_levels=2)),                     # which is past the limit here
    (65, dict(max_levels=3, coarse_size=20)),
    (193, dict(max_levels=3, coarse_size=20)),    # grid 1 is past it
    (129, dict(coarse_size=20))])
def test_algebraic_coarse_correction(M, nodes, amg):
    prob = pb.fracture_network(1e2, nodes=nodes)
    A = pb.stencil_csr(prob)
    A.sort_indices()
    O = oamg.AlgebraicHierarchy(A, **amg)
    for precision in (M.MPCG_FP64, M.MPCG_MIXED):
        H = M.AlgebraicHierarchy(A, precision=precision, **amg)
        if precision == M.MPCG_FP64:
            _columns(M.mg_corrections, H, O, A.shape[0], O.levels, 1e-12)
        b = torch.from_numpy(prob.b).cuda()
        x = torch.zeros_like(b)
        status, _, _, _ = H.solve(b, x, rtol=1e-8, maxit=1000)
        assert status == M.MPCG_OK
        assert np.linalg.norm(prob.b - A @ x.cpu().numpy()) <= 1.01e-8 * np.linalg.norm(prob.b)


def _fields(prob, B):
    R = np.stack([pb.normal(40 + k, prob.n) for k in range(B)])
    R /= np.linalg.norm(R, axis=1, keepdims=True)
    E = np.stack([pb.normal(70 + k, prob.n) for k in range(B)])
    return torch.from_numpy(R.astype(np.float32)).cuda(), torch.from_numpy(E.astype(np.float32)).cuda()


def _net(M, nodes):
    prob = pb.diffusion_macro(2, nodes, 22, rhs="normal", rhs_seed=1)
    return prob, M.Hierarchy(torch.from_numpy(np.ascontiguousarray(prob.stencil)).cuda(), 2, nodes, prob.levels,
                             precision=M.MPCG_MIXED)


def test_forward_workspace_of_a_hierarchy(M):
    """Calls of growing and shrinking image counts and a call after detaching
    give the bits of a hierarchy's first call."""
    prob, H = _net(M, 65)
    R, _ = _fields(prob, 5)
    theta = OL.init_params(5)
    M.mg_learned_attach(H.h, theta)
    for step, c in enumerate((2, 5, 1, 3)):
        if step == 3:
            M.mg_learned_detach(H.h)
            M.mg_learned_attach(H.h, theta)
        _, H1 = _net(M, 65)
        M.mg_learned_attach(H1.h, theta)
        y, want = torch.zeros_like(R[:c]), torch.zeros_like(R[:c])
        M.mg_learned_forward(H.h, R[:c].contiguous(), y, c)
        M.mg_learned_forward(H1.h, R[:c].contiguous(), want, c)
        assert torch.equal(y, want), c


@pytest.mark.parametrize("nodes,B", [(33, 12), (65, 1), (129, 9)])
def test_gradient_of_a_batch_is_the_mean_of_its_images(M, nodes, B):
    prob, H = _net(M, nodes)
    R, E = _fields(prob, B)
    theta = OL.init_params(5)
    g, loss = M.mg_learned_grad(H.h, theta, R, E, B)
    one = [M.mg_learned_grad(H.h, theta, R[k:k + 1].contiguous(), E[k:k + 1].contiguous(), 1) for k in range(B)]
    want = np.mean([o[0] for o in one], axis=0)
    assert np.linalg.norm(g - want) <= 1e-4 * np.linalg.norm(want)
    assert abs(loss - np.mean([o[1] for o in one])) <= 1e-6 * abs(loss)


def test_training_set_products_and_batches(M):
    """Fourteen pairs of two problems in a mixed order, with a learning rate of
    zero: the epoch's loss is the mean of the pairs' own losses, so every pair
    has met its own residual, error and product."""
    prob, H = _net(M, 33)
    prob2 = pb.diffusion_macro(2, 33, 5, rhs="normal", rhs_seed=1)
    H2 = M.Hierarchy(torch.from_numpy(np.ascontiguousarray(prob2.stencil)).cuda(), 2, 33, prob2.levels,
                     precision=M.MPCG_MIXED)
    R, E = _fields(prob, 14)
    which = [0] * 13 + [1]
    theta = OL.init_params(5)
    want = [M.mg_learned_grad((H, H2)[which[k]].h, theta, R[k:k + 1].contiguous(), E[k:k + 1].contiguous(), 1)[1]
            for k in range(14)]
    params = theta.copy()
    loss = M.mg_learned_train([H.h, H2.h], which, R, E, params, epochs=1, batch=1, lr=0.0)
    assert np.array_equal(params, theta)
    assert abs(loss[0] - np.mean(want)) <= 1e-6 * abs(np.mean(want))


def test_batches_of_several_pairs(M):
    """Pairs of two problems in a mixed order, a multiple of the batch each, with a
    learning rate of zero: the epoch's loss is the mean of the pairs' own losses.
    And a batch that the pairs do not fill, of the second of two problems: one Adam
    step along the gradient of its pairs (the first step moves a weight by lr g /
    (|g| + eps): for entries above a thousandth of the largest, whose sign the
    order of the sums cannot turn, within 1e-3 lr)."""
    prob, H = _net(M, 33)
    prob2 = pb.diffusion_macro(2, 33, 5, rhs="normal", rhs_seed=1)
    H2 = M.Hierarchy(torch.from_numpy(np.ascontiguousarray(prob2.stencil)).cuda(), 2, 33, prob2.levels,
                     precision=M.MPCG_MIXED)
    R, E = _fields(prob, 12)
    which = [0, 1, 0, 0, 1, 0, 0, 1, 0, 0, 1, 0]
    theta = OL.init_params(5)
    want = [M.mg_learned_grad((H, H2)[which[k]].h, theta, R[k:k + 1].contiguous(), E[k:k + 1].contiguous(), 1)[1]
            for k in range(12)]
    params = theta.copy()
    loss = M.mg_learned_train([H.h, H2.h], which, R, E, params, epochs=1, batch=4, lr=0.0)
    assert np.array_equal(params, theta)
    assert abs(loss[0] - np.mean(want)) <= 1e-6 * abs(np.mean(want))

    lr = 1e-3
    R3, E3 = R[:3].contiguous(), E[:3].contiguous()
    g, l3 = M.mg_learned_grad(H2.h, theta, R3, E3, 3)
    params = theta.copy()
    loss = M.mg_learned_train([H.h, H2.h], [1, 1, 1], R3, E3, params, epochs=1, batch=8, lr=lr, eps=1e-12)
    big = np.abs(g) > 1e-3 * np.abs(g).max()
    assert big.sum() > 1000 and abs(loss[0] - l3) <= 1e-6 * abs(l3)
    assert np.abs((params - theta)[big] + lr * np.sign(g[big])).max() <= 1e-3 * lr + 1e-7 * np.abs(theta).max()


def test_double_word_elasticity_with_the_fused_sweep(M):
    """65^3 nodes, 3 unknowns each: the fine grid's second sweep is one launch.  The
    double-word solve takes the FP64 solve's updates within one and gives its
    solution (both stop on the same recursion; 1e-9 of the norm), and its residual
    with the FP64 operator meets the tolerance."""
    prob = pb.elasticity_cantilever(65)
    st = torch.from_numpy(np.ascontiguousarray(prob.stencil)).cuda()
    b = torch.from_numpy(prob.b).cuda()
    got = []
    for precision in (M.MPCG_FP64, M.MPCG_FP64_DW):
        H = M.Hierarchy(st, 3, 65, prob.levels, dofs_per_node=3, faces=prob.faces, precision=precision)
        x, y = torch.zeros_like(b), torch.zeros_like(b)
        status, k, _, _ = H.solve(b, x, rtol=1e-8, maxit=100, histories=False)
        M.mg_apply_operator(H.h, prob.levels - 1, x, y, 1)
        assert status == M.MPCG_OK and (b - y).norm() <= 1.01e-8 * b.norm()
        got.append((k, x))
        H.close()
    assert abs(got[0][0] - got[1][0]) <= 1
    assert (got[0][1] - got[1][1]).norm() <= 1e-9 * got[0][1].norm()
