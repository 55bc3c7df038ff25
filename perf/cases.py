"""The solves and network passes this library is used for, as measurable cases.

Every case goes through the public Python binding (paper_2402_12833_gb300.mpcg)
with device tensors, as the benchmark and the tests do:

  solve      one mpcg_solve of a structured problem from a zero start
  batch      one mpcg_solve_batched of many uneven 2D problems
  algebraic  one mpcg_solve on a smoothed-aggregation hierarchy
  forward    one mg_learned_forward of the learned column's network
  train      one epoch of mg_learned_train

A program that uses the solver builds the hierarchy once per operator and then
solves for its right-hand sides, so the operator, the hierarchy and the
right-hand side are prepared and the solve is what runs.

Tolerances.  The default is 1e-8.  Mixed precision on high-contrast
coefficients refines further (1e-10, and 1e-12 for the fracture network, whose
smooth load leaves an error well above the residual), so that what comes back
is determined to more digits than FP32 rounding can move: there the number of x
updates moves by a few per cent with the rounding of the FP32 sums (the tests
allow that as well), and for that reason it is not among the outputs.
"""
import math

import numpy as np
import torch

from paper_2402_12833_gb300 import mpcg as M
from paper_2402_12833_gb300 import problems as pb

DEV = "cuda"
FP64, MIXED, DW = "fp64", "mixed", "fp64_dw"
PRECISION = {FP64: M.MPCG_FP64, MIXED: M.MPCG_MIXED, DW: M.MPCG_FP64_DW}
WINDOW = 5                     # stored search blocks: the default, and what all but a few programs use
MAXIT = 20000


def _solve_case(name, operator, dim, nodes, levels, precision, rtol, faces=0x3F, matrix_free=False, m=WINDOW):
    c = {"call": "solve", "operator": operator, "dim": dim, "nodes": nodes, "levels": levels,
         "precision": precision, "rtol": rtol, "faces": faces, "matrix_free": matrix_free, "m": m}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one 65^2 Poisson problem (3,969 unknowns), default arithmetic; launches count
        _solve_case("poisson2d_65_fp64", "poisson", 2, 65, 5, FP64, 1e-8),
        # a small 3D problem inside a time or Newton loop, mixed precision
        _solve_case("poisson3d_33_mixed", "poisson", 3, 33, 4, MIXED, 1e-8),
        # the headline: 129^3 nodes, N(0,1) load, mixed precision
        _solve_case("poisson3d_129_mixed", "poisson", 3, 129, 6, MIXED, 1e-8),
        # the same in double-word arithmetic (FP64-accurate iterates)
        _solve_case("poisson3d_129_fp64_dw", "poisson", 3, 129, 6, DW, 1e-8),
        # default arithmetic on a ragged grid (96 elements: rows of 95 unknowns, coarsest 7^3 nodes)
        _solve_case("poisson3d_97_fp64", "poisson", 3, 97, 5, FP64, 1e-8),
        # element coefficients given: matrix-free fine operator, natural conditions on three faces, 112 elements
        _solve_case("diffusion3d_113_matrix_free", "kappa", 3, 113, 5, MIXED, 1e-10, faces=0x15, matrix_free=True),
        # high-contrast coefficients on a large 2D grid
        _solve_case("diffusion2d_1025_mixed", "kappa", 2, 1025, 9, MIXED, 1e-10),
        # 3 unknowns per node: the clamped cube under a body force
        _solve_case("elasticity3d_65_mixed", "elasticity", 3, 65, 5, MIXED, 1e-8, faces=0x1),
        # many uneven problems in one call
        {"name": "batch2d_48_mixed", "call": "batch", "count": 48, "largest": 257, "sides": 4, "rtol": 1e-10},
        # a fracture network on the algebraic hierarchy
        {"name": "fracture2d_545_algebraic", "call": "algebraic", "nodes": 545, "kf": 1e4, "rtol": 1e-12},
        # the learned column's network, four residuals at once
        {"name": "learned_forward_1025", "call": "forward", "nodes": 1025, "images": 4},
        # its training: forward, backward and Adam over 64 pairs in batches of 8
        {"name": "learned_train_129", "call": "train", "nodes": 129, "pairs": 64, "batch": 8},
    ]


def _elements(rng, lo, hi, coarse, least):
    """q * 2^(levels - 1) elements per side, log-uniform between lo and hi, q drawn from coarse."""
    while True:
        e = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        q = rng.choice(coarse)
        k = round(math.log2(e / q))
        if k >= least - 1 and lo <= q << k <= hi:
            return q << k, k + 1


def draw(rng):
    m = rng.choice([3, 4, WINDOW, WINDOW, 6, 8])
    kind = rng.choice(["poisson2d", "poisson3d", "poisson3d", "poisson3d", "matrix_free", "kappa2d", "elasticity",
                       "batch", "algebraic", "forward", "train"])
    if kind == "poisson2d":
        e, levels = _elements(rng, 32, 1024, (3, 4, 5, 6, 7, 9), 3)
        return _solve_case(None, "poisson", 2, e + 1, levels, rng.choice([FP64, MIXED, DW]), 1e-8, m=m)
    if kind == "poisson3d":
        precision = rng.choice([FP64, MIXED, MIXED, DW])
        e, levels = _elements(rng, 16, 96 if precision == FP64 else 128, (3, 4, 5, 6, 7, 9), 2)
        return _solve_case(None, "poisson", 3, e + 1, levels, precision, 1e-8, m=m)
    if kind == "matrix_free":
        e, levels = _elements(rng, 16, 128, (4, 5, 6, 7), 2)
        return _solve_case(None, "kappa", 3, e + 1, levels, MIXED, 1e-10, rng.choice([0x3F, 0x15, 0x1F]), True, min(m, WINDOW))
    if kind == "kappa2d":
        e, levels = _elements(rng, 64, 1024, (4, 5, 6, 7), 3)
        return _solve_case(None, "kappa", 2, e + 1, levels, MIXED, 1e-10, m=min(m, WINDOW))
    if kind == "elasticity":
        e, levels = _elements(rng, 8, 64, (2, 3, 4, 5, 6), 2)
        return _solve_case(None, "elasticity", 3, e + 1, levels, rng.choice([MIXED, MIXED, DW]), 1e-8, 0x1, m=m)
    if kind == "batch":
        return {"call": "batch", "count": rng.randint(6, 48), "largest": rng.choice([65, 129, 257]),
                "sides": rng.randrange(1 << 20), "rtol": 1e-10}
    if kind == "algebraic":
        return {"call": "algebraic", "nodes": rng.randint(64, 545), "kf": 10.0 ** rng.uniform(0, 4), "rtol": 1e-12}
    if kind == "forward":
        # the 2D network takes 2^k + 1 nodes per side
        k = rng.randint(6, 10)
        return {"call": "forward", "nodes": 1 + 2 ** k, "images": rng.randint(1, 3 if k == 10 else 12)}
    return {"call": "train", "nodes": rng.choice([33, 65, 129]), "pairs": rng.randint(9, 64), "batch": rng.choice([4, 8])}


# ---------------------------------------------------------------------------
# problems, assembled on the GPU in the library's stencil format
# ---------------------------------------------------------------------------

def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + salt)
    return g


def _offsets(dim):
    return [tuple((s // 3 ** k) % 3 - 1 for k in range(dim)) for s in range(3 ** dim)]


def _macro_kappa(dim, nodes, gen):
    """log10(kappa) uniform in [-2, 4] on a 16^dim macro grid, per element."""
    v = 10.0 ** (-2.0 + 6.0 * torch.rand((16,) * dim, generator=gen, device=DEV, dtype=torch.float64))
    m = (16 * torch.arange(nodes - 1, device=DEV)) // (nodes - 1)
    for ax in range(dim):
        v = v.index_select(ax, m)
    return v


def _eliminate(dim, planes, faces):
    """Rows of the unknown nodes, couplings to the nodes of Dirichlet faces zero."""
    flags = [((faces >> 2 * a) & 1, (faces >> 2 * a + 1) & 1) for a in range(dim)]
    sl = tuple(slice(lo, planes.shape[-1 - a] - hi) for a, (lo, hi) in reversed(list(enumerate(flags))))
    out = planes[(Ellipsis,) + sl].clone()
    for q in range(out.shape[0]):
        for a, o in enumerate(_offsets(dim)[q % 3 ** dim]):
            if o and flags[a][o > 0]:
                out[q].select(out.dim() - 2 - a, 0 if o < 0 else -1).zero_()
    return out


def _assemble(dim, nodes, elem, coef, faces):
    """Planes [3^dim, z, y, x] of the scalar operator with element matrix elem and element coefficients coef."""
    ne = nodes - 1
    planes = torch.zeros((3 ** dim,) + (nodes,) * dim, dtype=torch.float64, device=DEV)
    for a in range(2 ** dim):
        abits = [(a >> k) & 1 for k in range(dim)]
        sl = tuple(slice(abits[k], abits[k] + ne) for k in reversed(range(dim)))
        for b in range(2 ** dim):
            s = sum((((b >> k) & 1) - abits[k] + 1) * 3 ** k for k in range(dim))
            planes[(s,) + sl] += float(elem[a, b]) * coef
    return _eliminate(dim, planes, faces)


def _assemble_elasticity(nodes, faces):
    """Planes [81, z, y, x, component] of Q1 elasticity (E = 1, nu = 0.3)."""
    ne = nodes - 1
    K = pb.q1_elasticity(1.0 / ne)
    full = torch.zeros((3, 27, 3) + (nodes,) * 3, dtype=torch.float64, device=DEV)
    for la in range(8):
        abits = [(la >> k) & 1 for k in range(3)]
        sl = tuple(slice(abits[k], abits[k] + ne) for k in (2, 1, 0))
        for lb in range(8):
            s = sum((((lb >> k) & 1) - abits[k] + 1) * 3 ** k for k in range(3))
            for a in range(3):
                for b in range(3):
                    full[(b, s, a) + sl] += float(K[3 * la + a, 3 * lb + b])
    full = full.reshape((81, 3) + (nodes,) * 3)
    return torch.stack([_eliminate(3, full[:, a], faces) for a in range(3)], dim=-1)


def _body_force(nodes, faces, force):
    """Consistent load of a constant body force on the unknown nodes."""
    w = torch.full((nodes,), 1.0 / (nodes - 1), dtype=torch.float64, device=DEV)
    w[0] = w[-1] = 0.5 / (nodes - 1)
    vol = w[:, None, None] * w[None, :, None] * w[None, None, :]
    sl = tuple(slice((faces >> 2 * a) & 1, nodes - ((faces >> 2 * a + 1) & 1)) for a in (2, 1, 0))
    return vol[sl][..., None] * force


def _problem(case, seed):
    """(planes, b, kappa): planes [S, ...grid] and b [...grid] with x last (then the component, for elasticity)."""
    dim, nodes, faces = case["dim"], case["nodes"], case["faces"]
    gen = _gen(seed)
    if case["operator"] == "elasticity":
        planes = _assemble_elasticity(nodes, faces)
        return planes, _body_force(nodes, faces, torch.randn(3, generator=gen, device=DEV, dtype=torch.float64)), None
    kappa = _macro_kappa(dim, nodes, gen) if case["operator"] == "kappa" else \
        torch.ones((nodes - 1,) * dim, dtype=torch.float64, device=DEV)
    planes = _assemble(dim, nodes, pb.q1_stiffness(dim, 1.0 / (nodes - 1)), kappa, faces)
    b = torch.randn(planes.shape[1:], generator=gen, device=DEV, dtype=torch.float64)
    return planes, b, kappa


def _batch_sides(case):
    """Sides of the batch, uniform over 33, 65, 129, 257 up to the largest, at least one of the largest."""
    sides = [s for s in (33, 65, 129, 257) if s <= case["largest"]]
    rng = np.random.default_rng(case["sides"])
    got = [int(s) for s in rng.choice(sides, case["count"] - 1)] + [case["largest"]]
    return {s: got.count(s) for s in sorted(set(got))}


def _batch_problems(case, seed):
    """Per side the planes [count, 9, y, x] and right-hand sides [count, y, x] of that many diffusion problems."""
    gen, out = _gen(seed, 1), {}
    for side, count in _batch_sides(case).items():
        ke = pb.q1_stiffness(2, 1.0 / (side - 1))
        planes = torch.stack([_assemble(2, side, ke, _macro_kappa(2, side, gen), 0x3F) for _ in range(count)])
        out[side] = planes, torch.randn((count, side - 2, side - 2), generator=gen, device=DEV, dtype=torch.float64)
    return out


def _fracture(case, seed):
    return pb.fracture_network(case["kf"], nodes=case["nodes"], seed=1 + int(seed) % (1 << 30))


def _error_fields(case, planes, gen, count):
    """Errors of the kind a solve leaves behind (a few modes per direction plus noise) and their residuals, scaled
    by the residual's norm: (rhat, e), float32."""
    n1 = case["nodes"] - 2
    t = torch.arange(1, n1 + 1, device=DEV, dtype=torch.float64) / (n1 + 1)
    sines = torch.sin(math.pi * t[:, None] * torch.arange(1, 25, device=DEV)[None, :])
    amp = torch.randn((count, 24, 24), generator=gen, device=DEV, dtype=torch.float64)
    e = sines @ amp @ sines.T / 24 + 0.05 * torch.randn((count, n1, n1), generator=gen, device=DEV, dtype=torch.float64)
    r = torch.stack([_apply(planes[None], x[None], 2)[0] for x in e])
    norm = torch.linalg.vector_norm(r, dim=(1, 2), keepdim=True)
    return (r / norm).float().reshape(count, -1).contiguous(), (e / norm).float().reshape(count, -1).contiguous()


def _network(seed):
    return pb.net_init_params(1 + int(seed) % (1 << 20))


# ---------------------------------------------------------------------------
# prepare, run
# ---------------------------------------------------------------------------

def prepare(case, seed):
    call = case["call"]
    s = {"call": call, "rtol": case.get("rtol")}
    if call == "solve":
        planes, b, kappa = _problem(case, seed)
        s["h"] = M.Hierarchy(planes.reshape(planes.shape[0], -1), case["dim"], case["nodes"], case["levels"],
                             dofs_per_node=3 if case["operator"] == "elasticity" else 1, faces=case["faces"],
                             m=case["m"], precision=PRECISION[case["precision"]])
        if case["matrix_free"]:
            M.mg_attach_q1_kappa(s["h"].h, kappa.reshape(-1))
        s["b"] = b.reshape(-1).contiguous()
        s["x"] = torch.zeros_like(s["b"])
    elif call == "batch":
        s["hs"], s["bs"], s["xs"] = [], [], []
        for side, (planes, b) in _batch_problems(case, seed).items():
            levels = pb.levels_for_nodes(side)
            s["hs"].append(M.BatchedHierarchy([p.reshape(9, -1) for p in planes], 2, side, levels, m=WINDOW,
                                              precision=M.MPCG_MIXED))
            s["bs"].append(b.reshape(b.shape[0], -1).contiguous())
            s["xs"].append(torch.zeros_like(s["bs"][-1]))
    elif call == "algebraic":
        prob = _fracture(case, seed)
        s["h"] = M.AlgebraicHierarchy(pb.stencil_csr(prob), m=WINDOW, precision=M.MPCG_MIXED)
        s["b"] = torch.from_numpy(prob.b).to(DEV)
        s["x"] = torch.zeros_like(s["b"])
    else:
        gen = _gen(seed, 2)
        nodes = case["nodes"]
        planes = _assemble(2, nodes, pb.q1_stiffness(2, 1.0 / (nodes - 1)), _macro_kappa(2, nodes, gen), 0x3F)
        s["h"] = M.Hierarchy(planes.reshape(9, -1), 2, nodes, _levels2d(nodes), m=WINDOW, precision=M.MPCG_MIXED)
        if call == "forward":
            s["r"], _ = _error_fields(case, planes, gen, case["images"])
            s["y"] = torch.empty_like(s["r"])
            M.mg_learned_attach(s["h"].h, _network(seed))
        else:
            s["r"], s["e"] = _error_fields(case, planes, gen, case["pairs"])
            s["params"], s["batch"] = _network(seed), case["batch"]
    return s


def _levels2d(nodes):
    """The deepest hierarchy whose coarsest grid keeps at least 4 elements per side."""
    e, levels = nodes - 1, 1
    while e % 2 == 0 and e // 2 >= 4:
        e, levels = e // 2, levels + 1
    return levels


def run(s):
    if s["call"] in ("solve", "algebraic"):
        s["x"].zero_()
        s["h"].solve(s["b"], s["x"], rtol=s["rtol"], maxit=MAXIT, histories=False)
        return s["x"]
    if s["call"] == "batch":
        for x in s["xs"]:
            x.zero_()
        M.mpcg_solve_batched(s["hs"], s["bs"], s["xs"], rtol=s["rtol"], maxit=MAXIT)
        return s["xs"]
    if s["call"] == "forward":
        M.mg_learned_forward(s["h"].h, s["r"], s["y"], s["r"].shape[0])
        return s["y"]
    params = s["params"].copy()     # the weights a training program starts from
    M.mg_learned_train([s["h"].h], [0] * s["r"].shape[0], s["r"], s["e"], params, epochs=1, batch=s["batch"])
    return params


# ---------------------------------------------------------------------------
# work: the method's own traffic and arithmetic
# ---------------------------------------------------------------------------

# x updates such a solve takes (typical counts over seeds, rounded)
UPDATES = {"poisson2": 16, "poisson3": 14, "kappa2": 240, "kappa3": 130, "elasticity3": 36, "algebraic": 330}


def _solve_work(n, cols, stencil, half, word, updates, m=WINDOW):
    """Bytes and operations of `updates` iterations with `cols` columns: the operator (`half` words a row where it is
    read by symmetry, `stencil` products a column), the search blocks of the window, Z, x and r, each once a pass."""
    blocks = [min(k, m) for k in range(int(updates))]
    nbytes = sum((2 * c * cols + 2 * cols + 4) * word + half * word for c in blocks) * n + 16 * n
    flops = sum(2 * (2 * c * cols ** 2 + stencil * cols + cols * (cols + 2)) for c in blocks) * n
    return nbytes, flops


def _unknowns(case):
    per = [case["nodes"] - ((case["faces"] >> 2 * a) & 1) - ((case["faces"] >> 2 * a + 1) & 1)
           for a in range(case["dim"])]
    return math.prod(per) * (3 if case["operator"] == "elasticity" else 1)


def work(case):
    call = case["call"]
    if call == "solve":
        dim = case["dim"]
        vec = case["operator"] == "elasticity"
        stencil = 81 if vec else 3 ** dim
        half = 1 if case["matrix_free"] else (41 if vec else (3 ** dim + 1) // 2)
        nbytes, flops = _solve_work(_unknowns(case), case["levels"], stencil, half,
                                    4 if case["precision"] == MIXED else 8, UPDATES["%s%d" % (case["operator"], dim)],
                                    case["m"])
    elif call == "batch":
        nbytes = flops = 0.0
        for side, count in _batch_sides(case).items():
            b, f = _solve_work((side - 2) ** 2, pb.levels_for_nodes(side), 9, 5, 4, UPDATES["kappa2"])
            nbytes, flops = nbytes + b * count, flops + f * count
    elif call == "algebraic":
        nbytes, flops = _solve_work(case["nodes"] * (case["nodes"] - 1), 5, 9, 5, 4, UPDATES["algebraic"])
    else:
        n = (case["nodes"] - 2) ** 2
        macs = 9 * (2 * 16 + 16 * 16 + 16 * 16 + 16)
        if call == "forward":
            nbytes, flops = case["images"] * n * 8 + n * 8, case["images"] * n * 2 * macs
        else:
            nbytes, flops = case["pairs"] * n * 8 + n * 8 * 9, case["pairs"] * n * 6 * macs
    return {"bytes": float(nbytes), "flops": float(flops)}


# ---------------------------------------------------------------------------
# exact: the solutions in 64 bits by conjugate gradients in plain torch
# ---------------------------------------------------------------------------

def _apply(planes, x, dim):
    """A x for a batch: planes [nb, 3^dim, ...grid], x [nb, ...grid]."""
    xp = torch.nn.functional.pad(x, (1, 1) * dim)
    y = torch.zeros_like(x)
    for s, off in enumerate(_offsets(dim)):
        sl = tuple(slice(1 + off[a], 1 + off[a] + x.shape[-1 - a]) for a in reversed(range(dim)))
        y.addcmul_(planes[:, s], xp[(slice(None),) + sl])
    return y


def _apply_vector(planes, x):
    """The same for 3 unknowns per node: planes [81, z, y, x, a], x [z, y, x, a]."""
    xp = torch.nn.functional.pad(x, (0, 0) + (1, 1) * 3)
    y = torch.zeros_like(x)
    for s, off in enumerate(_offsets(3)):
        sl = tuple(slice(1 + off[a], 1 + off[a] + x.shape[2 - a]) for a in (2, 1, 0))
        for b in range(3):
            y.addcmul_(planes[27 * b + s], xp[sl + (slice(b, b + 1),)])
    return y


def _conjugate_gradients(apply, diag, b, dims):
    """x with A x = b to the limit of 64 bits: Jacobi-preconditioned CG, restarted on the true residual."""
    def dot(u, v):
        return (u * v).sum(dim=dims, keepdim=True)

    x = torch.zeros_like(b)
    nb = dot(b, b)
    for _ in range(4):
        r = b - apply(x)
        d, z = torch.zeros_like(b), r / diag
        p, rz = z, dot(r, z)
        start = dot(r, r).clamp_min(1e-300)
        if bool((start <= 1e-32 * nb).all()):
            break
        for k in range(60000):
            q = apply(p)
            a = rz / dot(p, q).clamp_min(1e-300)
            d = d + a * p
            r = r - a * q
            if k % 25 == 24 and bool((dot(r, r) <= 1e-20 * start).all()):
                break
            z = r / diag
            new = dot(r, z)
            p = z + (new / rz.clamp_min(1e-300)) * p
            rz = new
        x = x + d
    return x


def _exact_forward(case, planes, r, params):
    """The network in 64 bits, with the bfloat16 rounding of weights, inputs and activations that it is defined with."""
    def bf(v):
        return v.to(torch.bfloat16).to(torch.float64)

    n1 = case["nodes"] - 2
    c = torch.log10(planes[4]) / 3.0
    v = torch.stack([r.double().reshape(-1, n1, n1), (c - c.mean()).expand(r.shape[0], n1, n1)], dim=1)
    chans, at = (2, 16, 16, 16, 1), 0
    for i in range(4):
        k = chans[i] * chans[i + 1] * 9
        w = torch.from_numpy(params[at:at + k]).to(DEV).double().reshape(chans[i + 1], chans[i], 3, 3)
        v = torch.nn.functional.conv2d(bf(v), bf(w), padding=1)
        v = torch.relu(v) if i < 3 else v
        at += k
    return v.reshape(r.shape[0], -1)


def exact(case, seed):
    call = case["call"]
    if call == "solve":
        planes, b, _ = _problem(case, seed)
        if case["operator"] == "elasticity":
            diag = torch.stack([planes[27 * a + 13, ..., a] for a in range(3)], dim=-1)
            x = _conjugate_gradients(lambda v: _apply_vector(planes, v), diag, b, (0, 1, 2, 3))
            return x.reshape(-1)
        dims = tuple(range(1, 1 + case["dim"]))
        x = _conjugate_gradients(lambda v: _apply(planes[None], v, case["dim"]), planes[None, 3 ** case["dim"] // 2],
                                 b[None], dims)
        return x.reshape(-1)
    if call == "batch":
        return [_conjugate_gradients(lambda v, p=planes: _apply(p, v, 2), planes[:, 4], b, (1, 2)).reshape(b.shape[0], -1)
                for planes, b in _batch_problems(case, seed).values()]
    if call == "algebraic":
        prob = _fracture(case, seed)
        nx, ny = prob.shape
        planes = torch.from_numpy(prob.stencil).to(DEV).reshape(1, 9, ny, nx)
        b = torch.from_numpy(prob.b).to(DEV).reshape(1, ny, nx)
        return _conjugate_gradients(lambda v: _apply(planes, v, 2), planes[:, 4], b, (1, 2)).reshape(-1)
    if call == "forward":
        gen = _gen(seed, 2)
        nodes = case["nodes"]
        planes = _assemble(2, nodes, pb.q1_stiffness(2, 1.0 / (nodes - 1)), _macro_kappa(2, nodes, gen), 0x3F)
        r, _ = _error_fields(case, planes, gen, case["images"])
        return _exact_forward(case, planes, r, _network(seed))
    return None     # a training epoch: its 64-bit value is not what bfloat16 activations give
