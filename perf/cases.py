"""The work that programs have this library do, as cases that can be timed and compared.

A case is one call (or the few calls that belong together) on one problem: applying the regional
operator, one V-cycle, splitting a composite CSR, the numeric setup, a solve, a whole step of a
time loop or nonlinear iteration (split, setup, solve), and the two halves of the learned
prolongator. Problems are tensor-product tilings of box regions: `x`, `y`, `z` hold the region
sizes (nodes per axis) of the slabs along each axis. All inputs are made on the GPU from the seed.
"""
import itertools
import math

import numpy as np
import torch

from paper_2103_11962_gb300 import rmg

PRECISIONS = {"fp64": 0, "fp32": 1, "bf16coef": 2}
SMOOTHERS = {"jacobi": 0, "chebyshev": 1, "gs": 2}


def _case(op, problem, x, y, z="", **kw):
    c = dict(op=op, problem=problem, x=x, y=y, z=z, sigma=0.0, levels=4, smoother="chebyshev",
             nu=1, precision="fp32")
    c.update(kw)
    return c


def listed():
    return [
        # The smallest call: a matrix-free product inside somebody else's Krylov loop on the
        # 163 x 163 Poisson problem of the benchmark. Launches are all it costs.
        dict(_case("apply", "poisson2d", "82,82", "82,82"), name="apply_poisson2d"),
        # A small solve, all latency: the same problem to 1e-10 with the plain FP64 method and
        # the damped Jacobi smoother (two sweeps each way), as the benchmark runs it.
        dict(_case("solve", "poisson2d", "82,82", "82,82", smoother="jacobi", nu=2,
                   precision="fp64"), name="solve_poisson2d"),
        # The residual operator of the outer CG on the headline operator (3D Q1, 55^3 regions).
        dict(_case("apply", "q1_3d", "55,55,55,55", "55,55,55,55", "55,55,55,55", sigma=0.5),
             name="apply_q1_3d"),
        # One preconditioner application in a caller's own Krylov method: variable-coefficient
        # diffusion on uneven slabs, plain FP64.
        dict(_case("vcycle", "diffusion3d", "82,55,28", "55,28", "28,82", sigma=1.0,
                   precision="fp64"), name="vcycle_diffusion3d"),
        # A new matrix on the same mesh, used matrix-free: split of a 27-point composite CSR
        # and a product with it.
        dict(_case("split", "q1_3d", "55,55,55,55", "55,55,55,55", "55,55,55,55", sigma=0.5),
             name="split_q1_3d"),
        # The numeric setup of the plain method alone (new coefficients, same mesh).
        dict(_case("setup", "diffusion3d", "55,82,28", "82,55", "28,55,55", sigma=1.0,
                   precision="fp64"), name="setup_diffusion3d"),
        # A whole step on the headline family, the largest that fits three times: constant
        # Q1 Laplacian, 216 regions of 55^3, 34 million unknowns, FP32 cycle in FP64 CG.
        dict(_case("step", "q1_3d", "55,55,55,55,55,55", "55,55,55,55,55,55",
                   "55,55,55,55,55,55"), name="step_q1_3d"),
        # A whole step of a variable-coefficient diffusion problem on uneven slabs.
        dict(_case("step", "diffusion3d", "55,28,82,55", "82,55,28", "55,82,28", sigma=1.0),
             name="step_diffusion3d"),
        # A whole step of 3D linear elasticity (3 unknowns per node, clamped at x = 0) with
        # 30 power-method steps, as the benchmark runs it.
        dict(_case("step", "elasticity3d", "55,28,55", "28,55,55", "55,28,28", sigma=0.5),
             name="step_elasticity3d"),
        # The region Gauss-Seidel smoother, a medium problem.
        dict(_case("solve", "diffusion3d", "55,28", "28,55", "55,28", sigma=1.0, smoother="gs"),
             name="solve_gs_diffusion3d"),
        # Learned interpolation weights of the finest level: features, network, weights.
        dict(_case("learn_weights", "diffusion3d", "55,28,55,28", "55,55,28", "28,28,55",
                   sigma=2.0), name="learn_weights"),
        # Training the network: forward and backward over a set of samples.
        dict(op="learn_gradient", samples=65573, name="learn_gradient"),
    ]


def draw(rng):
    op, problem = rng.choice([
        ("apply", "poisson2d"), ("apply", "q1_2d"), ("apply", "q1_3d"), ("apply", "diffusion3d"),
        ("apply", "elasticity3d"), ("solve", "poisson2d"), ("solve", "q1_2d"),
        ("solve", "diffusion3d"), ("vcycle", "q1_2d"), ("vcycle", "diffusion3d"),
        ("vcycle", "q1_3d"), ("split", "q1_3d"), ("split", "diffusion3d"),
        ("split", "elasticity3d"), ("setup", "diffusion3d"), ("setup", "q1_2d"),
        ("step", "q1_3d"), ("step", "q1_3d"), ("step", "diffusion3d"), ("step", "diffusion3d"),
        ("step", "elasticity3d"), ("step", "poisson2d"), ("learn_weights", "diffusion3d"),
        ("learn_gradient", "")])
    if op == "learn_gradient":
        return dict(op=op, samples=int(2.0 ** rng.uniform(7.0, 19.0)) | 1)
    two_d = problem.endswith("2d")
    levels = rng.choice([3, 4])
    if op in ("apply", "split"):
        sizes = list(range(8, 90))
    else:
        sizes = list(range(10, 110, 9)) if levels == 3 else [28, 55, 82, 109]
    # regional nodes: spread over the logarithm, up to the listed cases' sizes and to a coarsest
    # level that is still solved densely in earnest
    ratio = (9 if two_d else 27) ** (levels - 1)
    nodes = 600 if problem == "elasticity3d" else 1800
    most = {"elasticity3d": 1.0e6, "q1_3d": 8.0e6}.get(problem, 5.0e6)
    if op not in ("apply", "split"):
        most = min(most, 0.6 * nodes * ratio)
    target = math.exp(rng.uniform(math.log(min(2.0e4, 0.1 * most)), math.log(most)))
    axes = [[rng.choice(sizes)] for _ in range(2 if two_d else 3)]
    while math.prod(sum(a) for a in axes) < target:
        a = min(axes, key=len)
        a.append(rng.choice(sizes))
        if math.prod(sum(a) for a in axes) > 1.5 * most:
            a[-1] = sizes[0]
        if math.prod(sum(a) for a in axes) > 1.5 * most:
            a.pop()
            break
    text = [",".join(str(v) for v in a) for a in axes] + ([""] if two_d else [])
    if op in ("apply", "split"):
        levels, precision, smoother, nu = 4, "fp32", "chebyshev", 1
    else:
        # results of a cycle or a setup are those of the plain method; solves mostly use the
        # FP32 cycle
        precision = "fp64" if op in ("vcycle", "setup") else rng.choice(
            ["fp32", "fp32", "fp32", "fp64", "bf16coef"])
        if problem == "elasticity3d":
            precision, smoother, nu = "fp32", "chebyshev", 1
        else:
            smoother = rng.choice(["chebyshev", "chebyshev", "chebyshev", "jacobi", "gs"])
            nu = 1 if smoother == "chebyshev" else 2
    return _case(op, problem, *text, sigma=0.0 if problem == "poisson2d" else rng.choice(
        [0.5, 0.75, 1.0]), levels=levels, smoother=smoother, nu=nu, precision=precision)


# ---------------------------------------------------------------------------- geometry
def _axes(case):
    a = [[int(v) for v in case[k].split(",")] for k in ("x", "y", "z") if case[k]]
    return a + [[1]] * (3 - len(a))


def _global_dims(case):
    return [sum(n - 1 for n in a) + 1 for a in _axes(case)]


def _regional_nodes(case):
    return math.prod(sum(a) for a in _axes(case))


def _regions(case):
    """Region sizes (numpy, regions x fastest) and the composite id of every regional node."""
    axes, (Nx, Ny, _) = _axes(case), _global_dims(case)
    origin = [[sum(n - 1 for n in a[:k]) for k in range(len(a))] for a in axes]
    dims, gids = [], []
    for kz, ky, kx in itertools.product(*(range(len(a)) for a in reversed(axes))):
        n = [axes[0][kx], axes[1][ky], axes[2][kz]]
        r = [torch.arange(n[d], dtype=torch.int64, device="cuda") + origin[d][k]
             for d, k in enumerate((kx, ky, kz))]
        dims.append(n)
        gids.append((r[0].view(1, 1, -1) + Nx * (r[1].view(1, -1, 1) +
                                                 Ny * r[2].view(-1, 1, 1))).reshape(-1))
    return np.asarray(dims, dtype=np.int32), torch.cat(gids)


def _mask(case):
    """Dirichlet nodes, [Nz, Ny, Nx]: every face of the domain, or x = 0 for elasticity."""
    Nx, Ny, Nz = _global_dims(case)
    m = torch.zeros((Nz, Ny, Nx), dtype=torch.bool, device="cuda")
    m[:, :, 0] = True
    if case["problem"] != "elasticity3d":
        m[:, :, -1] = True
        m[:, 0] = m[:, -1] = True
        if Nz > 1:
            m[0] = m[-1] = True
    return m


# ---------------------------------------------------------------------------- matrices
def _element_matrix(dim, elastic):
    """Bi-/trilinear element matrix of the unit cube by 2-point Gauss quadrature: Laplacian, or
    linear elasticity with E = 1 and Poisson ratio 0.3 (dof = 3 * corner + component)."""
    corners = np.array([[(a >> d) & 1 for d in range(dim)] for a in range(2 ** dim)], dtype=float)
    g = 0.5 / math.sqrt(3.0)
    nu = 0.3
    lam, mu = nu / ((1 + nu) * (1 - 2 * nu)), 0.5 / (1 + nu)
    K = np.zeros((2 ** dim * (3 if elastic else 1),) * 2)
    for q in itertools.product((0.5 - g, 0.5 + g), repeat=dim):
        f = np.where(corners > 0, np.array(q), 1.0 - np.array(q))           # [corner, axis]
        s = np.where(corners > 0, 1.0, -1.0)
        grad = np.stack([s[:, d] * np.prod(np.delete(f, d, axis=1), axis=1)
                         for d in range(dim)], axis=1)
        if not elastic:
            K += grad @ grad.T / 2 ** dim
            continue
        Bm = np.zeros((6, 24))
        for a in range(8):
            gx, gy, gz = grad[a]
            Bm[:, 3 * a:3 * a + 3] = [[gx, 0, 0], [0, gy, 0], [0, 0, gz],
                                      [gy, gx, 0], [0, gz, gy], [gz, 0, gx]]
        D = np.diag([2 * mu] * 3 + [mu] * 3)
        D[:3, :3] += lam
        K += Bm.T @ D @ Bm / 8
    return 0.5 * (K + K.T)


def _offsets(problem):
    """Stencil offsets (dx, dy, dz) in ascending order of the column they lead to."""
    if problem == "poisson2d":
        return [(0, -1, 0), (-1, 0, 0), (0, 0, 0), (1, 0, 0), (0, 1, 0)]
    if problem == "diffusion3d":
        return [(0, 0, -1), (0, -1, 0), (-1, 0, 0), (0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1)]
    if problem == "q1_2d":
        return [(s % 3 - 1, s // 3 - 1, 0) for s in range(9)]
    return [(s % 3 - 1, s // 3 % 3 - 1, s // 9 - 1) for s in range(27)]


def _edge_means(kappa, axis):
    """Mean of the elements around every edge along `axis` (0: x), [Nz, Ny, Nx] edges from the
    node in the + direction (zero past the last node)."""
    one = torch.ones_like(kappa)
    pad = [0, 0, 0, 0, 0, 0]
    for d in range(3):
        pad[2 * d:2 * d + 2] = [0, 1] if d == axis else [1, 1]
    k, n = (torch.nn.functional.pad(t, pad) for t in (kappa, one))
    for d in range(3):
        if d != axis:
            lo = [slice(None)] * 3
            hi = [slice(None)] * 3
            lo[2 - d], hi[2 - d] = slice(0, -1), slice(1, None)
            k, n = k[tuple(lo)] + k[tuple(hi)], n[tuple(lo)] + n[tuple(hi)]
    return torch.where(n > 0, k / n.clamp(min=1), torch.zeros((), dtype=k.dtype, device=k.device))


def _stencil_planes(case, g):
    """Assembled coefficients [slot, c, c', Nz, Ny, Nx] of the composite operator before the
    boundary condition (B = 1 or 3 components)."""
    Nx, Ny, Nz = _global_dims(case)
    problem, offs = case["problem"], _offsets(case["problem"])
    B = 3 if problem == "elasticity3d" else 1
    v = torch.zeros((len(offs), B, B, Nz, Ny, Nx), dtype=torch.float64, device="cuda")
    if problem == "poisson2d":
        for s, o in enumerate(offs):
            v[s] = 4.0 if o == (0, 0, 0) else -1.0
        return v
    elems = (max(1, Nz - 1), Ny - 1, Nx - 1)
    kappa = torch.exp(case["sigma"] * torch.randn(elems, generator=g, dtype=torch.float64,
                                                  device="cuda"))
    if problem == "diffusion3d":
        h = 1.0 / (Nx - 1)
        for axis, (lo, hi) in enumerate(((2, 4), (1, 5), (0, 6))):
            c = -h * _edge_means(kappa, axis)
            v[hi, 0, 0] = c
            d = 2 - axis
            v[lo, 0, 0].narrow(d, 1, c.shape[d] - 1).copy_(c.narrow(d, 0, c.shape[d] - 1))
        v[3] = -(v[0] + v[1] + v[2] + v[4] + v[5] + v[6])
        return v
    dim = 2 if problem == "q1_2d" else 3
    K = _element_matrix(dim, B == 3) * ((1.0 / (Nx - 1)) if dim == 3 else 1.0)
    for a, c in itertools.product(range(2 ** dim), repeat=2):
        pa, pc = ([(k >> d) & 1 for d in range(3)] for k in (a, c))
        s = offs.index(tuple(pc[d] - pa[d] for d in range(3)))
        for i, j in itertools.product(range(B), repeat=2):
            v[s, i, j, pa[2]:pa[2] + elems[0], pa[1]:pa[1] + elems[1],
              pa[0]:pa[0] + elems[2]] += float(K[B * a + i, B * c + j]) * kappa
    return v


def _matrix(case, g):
    """Composite CSR (rowptr, col, val; dofs node-major): identity rows at Dirichlet nodes, their
    columns removed, columns ascending."""
    Nx, Ny, Nz = _global_dims(case)
    offs, mask = _offsets(case["problem"]), _mask(case)
    v = _stencil_planes(case, g)
    S, B, n = len(offs), v.shape[1], mask.numel()
    keep = torch.zeros((S, Nz, Ny, Nx), dtype=torch.bool, device="cuda")
    free = ~mask
    for s, (dx, dy, dz) in enumerate(offs):
        here = [slice(max(0, -d), N - max(0, d)) for d, N in ((dz, Nz), (dy, Ny), (dx, Nx))]
        there = [slice(max(0, d), N - max(0, -d)) for d, N in ((dz, Nz), (dy, Ny), (dx, Nx))]
        keep[(s, *here)] = free[tuple(here)] & free[tuple(there)]
    centre = offs.index((0, 0, 0))
    for i, j in itertools.product(range(B), repeat=2):
        v[centre, i, j][mask] = 1.0 if i == j else 0.0
    # entries in row order: [node, c, slot, c']
    v = v.reshape(S, B, B, n).permute(3, 1, 0, 2).contiguous()
    keep = keep.reshape(S, n).t().contiguous()
    keep = keep.view(n, 1, S, 1).expand(n, B, S, B).contiguous()
    if B == 1:
        keep[:, 0, centre, 0] = True
    else:
        for i in range(B):
            keep[:, i, centre, i] = True
    count = keep.view(n * B, -1).sum(1)
    rowptr = torch.zeros(n * B + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(count, 0, out=rowptr[1:])
    val = v[keep]
    del v
    step = torch.tensor([dx + Nx * (dy + Ny * dz) for dx, dy, dz in offs], device="cuda")
    col = (torch.arange(n, device="cuda").view(n, 1, 1, 1) + step.view(1, 1, S, 1)) * B + \
        torch.arange(B, device="cuda").view(1, 1, 1, B)
    col = col.expand(n, B, S, B)[keep]
    return rowptr, col, val


def _rhs(case, g):
    """Right-hand side or vector: uniform in [-1, 1), zero at Dirichlet nodes, node-major."""
    B = 3 if case["problem"] == "elasticity3d" else 1
    m = _mask(case).reshape(-1)
    b = 2.0 * torch.rand((m.numel(), B), generator=g, dtype=torch.float64, device="cuda") - 1.0
    b[m] = 0.0
    return b.reshape(-1)


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


# ---------------------------------------------------------------------------- network
def _network(g):
    """He-initialised parameters in the library's order: W1, b1, W2, b2, W3, b3."""
    r = lambda *s: torch.randn(s, generator=g, dtype=torch.float64, device="cuda")  # noqa: E731
    parts = [r(64, 32) * math.sqrt(2 / 27), 0.1 * r(64), r(64, 64) * math.sqrt(2 / 64),
             0.1 * r(64), r(3, 64) / 8, 0.1 * r(3)]
    return torch.cat([p.reshape(-1) for p in parts]).float().cpu().numpy()


def _samples(n, g):
    """Features as the library forms them (log10 ratios, remainder, active flag per axis),
    labels in [0, 1] and the mask of active axes."""
    f = torch.zeros((n, 32), dtype=torch.float32, device="cuda")
    mask = torch.zeros((n, 3), dtype=torch.float32, device="cuda")
    for a in range(3):
        rem = torch.randint(0, 3, (n,), generator=g, device="cuda")
        on = (rem > 0).float()
        f[:, 9 * a:9 * a + 7] = torch.randn((n, 7), generator=g, device="cuda").clamp(-4, 2)
        f[:, 9 * a + 7] = rem.float() / 3
        f[:, 9 * a + 8] = 1.0
        f[:, 9 * a:9 * a + 9] *= on.view(-1, 1)
        mask[:, a] = on
    labels = torch.rand((n, 3), generator=g, device="cuda")
    return f, labels, mask


# ---------------------------------------------------------------------------- the cases
def prepare(case, seed):
    g = _generator(seed)
    ctx = rmg.Context(0)
    op = case["op"]
    if op == "learn_gradient":
        f, labels, mask = _samples(case["samples"], g)
        return dict(op=op, mlp=rmg.MLP(ctx, _network(g)), feats=f, labels=labels, mask=mask)
    problem = case["problem"]
    B = 3 if problem == "elasticity3d" else 1
    rowptr, col, val = _matrix(case, g)
    b = _rhs(case, g)
    dims, gids = _regions(case)
    mask = _mask(case).reshape(-1).to(torch.uint8)
    stencil = len(_offsets(problem))
    lay = rmg.Layout(ctx, 2 if problem.endswith("2d") else 3, dims, gids, mask.numel(), mask)
    s = dict(op=op, lay=lay, stencil=stencil, B=B, levels=case["levels"])
    if op in ("split", "step"):
        s.update(rowptr=rowptr, col=col, val=val)
    _split(lay, stencil, B, rowptr, col, val)
    if op in ("apply", "split"):
        # a consistent regional vector, component-major
        s["u"] = b.view(-1, B)[gids].t().contiguous().reshape(-1)
        s["y"] = torch.empty_like(s["u"])
        return s
    opts = rmg.default_options(levels=case["levels"], smoother=SMOOTHERS[case["smoother"]],
                               nu1=case["nu"], nu2=case["nu"], cheb_degree=3, omega=0.67,
                               power_iters=30 if B == 3 else 10,
                               precision=PRECISIONS[case["precision"]])
    h = s["hier"] = rmg.Hierarchy(lay, opts)
    if op in ("solve", "step", "vcycle"):
        s["b"] = b
        s["x"] = torch.zeros_like(b)
    if op == "setup":
        s["out"] = []
        for l in range(case["levels"]):
            n_r, _, kind = h.level_sizes(l)
            s["out"].append((torch.empty(kind * n_r, dtype=torch.float64, device="cuda")
                             if l else None, torch.empty(n_r, dtype=torch.float64,
                                                         device="cuda")))
    if op == "learn_weights":
        s["mlp"] = rmg.MLP(ctx, _network(g))
        s["w"] = torch.empty(3 * h.level_sizes(0)[0], dtype=torch.float32, device="cuda")
    return s


def _split(lay, stencil, B, rowptr, col, val):
    if B == 1:
        lay.operator_from_csr(stencil, rowptr, col, val)
    else:
        lay.operator_from_block_csr(stencil, B, rowptr, col, val)


def run(s):
    op = s["op"]
    if op == "learn_gradient":
        loss, grad = s["mlp"].gradient(s["feats"], s["labels"], s["mask"])
        return {"loss": loss, "grad": grad}
    if op in ("split", "step"):
        _split(s["lay"], s["stencil"], s["B"], s["rowptr"], s["col"], s["val"])
    if op in ("apply", "split"):
        s["lay"].regional_apply(s["u"], s["y"])
        return {"y": s["y"]}
    h = s["hier"]
    if op == "learn_weights":
        h.mlp_weights(0, s["mlp"], s["w"])
        return {"weights": s["w"]}
    if op == "vcycle":
        h.vcycle(s["b"], s["x"])
        return {"z": s["x"]}
    if op in ("setup", "step"):
        h.setup_numeric()
    if op == "setup":
        # the coarse operators and the inverse diagonals of every level, as a caller's own
        # smoother or coarse solver takes them
        for l, (coef, dinv) in enumerate(s["out"]):
            h.level_export(l, coef, dinv)
        return {"levels": [[c for c in pair if c is not None] for pair in s["out"]],
                "lambda": [h.lam(l) for l in range(s["levels"] - 1)]}
    s["x"].zero_()
    info = h.pcg(s["b"], s["x"], rtol=1e-10, maxit=200, history=False)
    return {"x": s["x"], "iterations": info["iterations"]}


def work(case):
    """Each input read once, each output written once; operations of one application of the
    operator (apply, split), of one cycle with its sweeps (vcycle), of ten cycles and products
    (solve, step), of the Galerkin products (setup) or of the network."""
    if case["op"] == "learn_gradient":
        n, params = case["samples"], 64 * 32 + 64 * 64 + 3 * 64 + 131
        return dict(bytes=n * 4 * (32 + 3 + 3) + 8 * params, flops=6.0 * n * params)
    B = 3 if case["problem"] == "elasticity3d" else 1
    S, n_r, n = len(_offsets(case["problem"])), _regional_nodes(case), math.prod(
        _global_dims(case))
    coef, product = 8.0 * S * B * B * n_r, 2.0 * S * B * B * n_r
    csr = 16.0 * S * B * B * n + 8.0 * B * n
    op = case["op"]
    sweeps = 2 * case["nu"] * (3 if case["smoother"] == "chebyshev" else 1)
    if op == "apply":
        return dict(bytes=coef + 16.0 * B * n_r, flops=product)
    if op == "split":
        return dict(bytes=csr + coef + 16.0 * B * n_r, flops=product)
    if op == "vcycle":
        return dict(bytes=coef + 16.0 * B * n, flops=sweeps * product)
    coarse = 27 if S in (7, 27) else 9
    if op == "setup":
        out = n_r / (27 if coarse == 27 else 9) * coarse * 8.0
        return dict(bytes=coef + out + 16.0 * n_r, flops=2.0 * S * coarse * n_r)
    if op == "learn_weights":
        return dict(bytes=coef + 12.0 * n_r, flops=2.0 * 6336 * n_r)
    return dict(bytes=(csr if op == "step" else coef) + 16.0 * B * n,
                flops=10.0 * (sweeps + 2) * product)


# ---------------------------------------------------------------------------- 64-bit values
def _solve(A, d, b, seconds=18.0):
    """Diagonally scaled conjugate gradients in 64 bits, restarted from the true residual until
    it no longer falls; None when it does not get there in time."""
    import time
    t0 = time.perf_counter()
    x, best = torch.zeros_like(b), math.inf
    bn = float(b.norm())
    for _ in range(6):
        r = b - A @ x
        rn = float(r.norm())
        if rn > 0.1 * best or rn <= 1e-14 * bn:
            return x
        best = rn
        e = torch.zeros_like(b)
        z = r / d
        p, rz = z.clone(), r.dot(z)
        for it in range(1, 20001):
            q = A @ p
            a = rz / p.dot(q)
            e.addcmul_(p, a)
            r.addcmul_(q, a, value=-1)
            torch.div(r, d, out=z)
            rz, old = r.dot(z), rz
            p.mul_(rz / old).add_(z)
            if it % 25 == 0:
                if float(r.norm()) <= 1e-8 * rn:
                    break
                if time.perf_counter() - t0 > seconds:
                    return None
        x = x + e
    return x


def exact(case, seed):
    g = _generator(seed)
    op = case["op"]
    if op == "learn_gradient":
        f, labels, mask = (t.double() for t in _samples(case["samples"], g))
        p = torch.from_numpy(_network(g)).cuda().double().requires_grad_()
        W1, b1, W2, b2, W3, b3 = p.split([64 * 32, 64, 64 * 64, 64, 3 * 64, 3])
        o = torch.relu(f @ W1.view(64, 32).t() + b1)
        o = torch.relu(o @ W2.view(64, 64).t() + b2)
        o = torch.sigmoid(o @ W3.view(3, 64).t() + b3)
        loss = (mask * (o - labels) ** 2).sum() / (3 * case["samples"])
        loss.backward()
        return {"loss": float(loss.detach()), "grad": p.grad}
    if op in ("vcycle", "learn_weights"):
        return None                     # defined by the method itself, not by a closed form
    rowptr, col, val = _matrix(case, g)
    B = 3 if case["problem"] == "elasticity3d" else 1
    N = rowptr.numel() - 1
    row = torch.repeat_interleave(torch.arange(N, device="cuda"), rowptr[1:] - rowptr[:-1])
    d = torch.zeros(N, dtype=torch.float64, device="cuda")
    on = row == col
    d[row[on]] = val[on]
    del row, on
    _, gids = _regions(case)
    if op == "setup":
        levels = [[None, None] for _ in range(case["levels"])]
        levels[0] = [1.0 / d[gids]]     # the coarse operators are the method's own
        return {"levels": levels, "lambda": [None] * (case["levels"] - 1)}
    if col.numel() < 2 ** 31:
        rowptr, col = rowptr.int(), col.int()
    A = torch.sparse_csr_tensor(rowptr, col, val, (N, N))
    b = _rhs(case, g)
    if op in ("apply", "split"):
        return {"y": (A @ b).view(-1, B)[gids].t().contiguous().reshape(-1)}
    x = _solve(A, d, b)
    return None if x is None else {"x": x, "iterations": None}
