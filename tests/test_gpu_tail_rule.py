"""Which levels go to the one-kernel coarse end: the launches of a cycle on either side of each
line, and cycles against the oracle where its forms change."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_common import rel_max

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.filterwarnings("ignore::scipy.sparse.SparseEfficiencyWarning")]


def _hier(p, levels, precision, smoother="CHEBYSHEV", B=1):
    from paper_2103_11962_gb300 import rmg, upload
    dp = upload(p)
    lay = rmg.Layout(rmg.Context(0), p.dim, p.region_dims, dp.gids, p.n_nodes, dp.dirichlet)
    if B == 1:
        lay.operator_from_csr(p.stencil, dp.rowptr, dp.col, dp.val)
    else:
        lay.operator_from_block_csr(27, 3, dp.rowptr, dp.col, dp.val)
    return dp, rmg.Hierarchy(lay, rmg.default_options(
        levels=levels, smoother=getattr(rmg, smoother), nu1=1, nu2=1, cheb_degree=3,
        power_iters=30 if B == 3 else 10, precision=getattr(rmg, precision)))


def _outside(levels, smoother, ncol, B=1):
    """Launches of `levels` levels that are not in the kernel, each with an interface: sweeps are
    two launches, the first one from zero a single one."""
    if smoother == "GAUSS_SEIDEL":             # residual and colours; the mean at the end
        return sum((1 + n) + 2 + 2 + 1 + (2 + n) + (2 if l == 0 else 0)
                   for l, n in enumerate(ncol[:levels]))
    return levels * ((1 + 2 * 2) + 2 + 2 * B + B + 3 * 2)


# problem, levels, and per precision: levels outside and whether the solve is inside (None: no
# level in the kernel)
RULES = {
    # 100 nodes a region on level 1, 16 on level 2: 16,300 / 16,400 nodes, solve above its line
    "16300 nodes": (lambda: W.q1_laplace2d((163, 1), 28), 3, "CHEBYSHEV", dict(FP32=(1, False))),
    "16400 nodes": (lambda: W.q1_laplace2d((164, 1), 28), 3, "CHEBYSHEV", dict(FP32=None)),
    "8100 nodes": (lambda: W.q1_laplace2d((27, 3), 28), 3, "CHEBYSHEV",
                   dict(FP64=(1, False), FP32=(1, False))),
    "8200 nodes": (lambda: W.q1_laplace2d((82, 1), 28), 3, "CHEBYSHEV",
                   dict(FP64=None, FP32=(1, False))),
    # Gauss-Seidel: twice the nodes
    "8200 nodes, gs": (lambda: W.q1_laplace2d((82, 1), 28), 3, "GAUSS_SEIDEL",
                       dict(FP64=(1, False), FP32=(1, False))),
    # coarsest unknowns: 384 / 385 beside a smoothed level, 256 / 258 alone, 48 / 49
    "solve of 384": (lambda: W.q1_laplace2d((25, 17), 10), 3, "CHEBYSHEV",
                     dict(FP64=(1, True), FP32=(1, True), FP32_BF16COEF=(1, True))),
    "solve of 385": (lambda: W.q1_laplace2d((36, 12), 10), 3, "CHEBYSHEV",
                     dict(FP64=(1, False), FP32=(1, False))),
    "256 alone": (lambda: W.q1_laplace2d((17, 17), 4), 2, "CHEBYSHEV",
                  dict(FP64=(1, True), FP32=(1, True))),
    "258 alone": (lambda: W.q1_laplace2d((44, 7), 4), 2, "CHEBYSHEV", dict(FP64=None, FP32=None)),
    "48 alone": (lambda: W.q1_laplace2d((9, 7), 4), 2, "CHEBYSHEV", dict(FP64=(1, True))),
    "49 alone": (lambda: W.q1_laplace2d((8, 8), 4), 2, "CHEBYSHEV", dict(FP64=(1, True))),
}


@pytest.mark.parametrize("case", list(RULES))
def test_levels_inside(case):
    make, levels, smoother, rules = RULES[case]
    p = make()
    for precision, rule in rules.items():
        _, h = _hier(p, levels, precision, smoother)
        ncol = [4] * levels
        n = h.vcycle_launches()
        base = _outside(levels - 1 if rule is None else rule[0], smoother, ncol)
        if rule and rule[1]:
            assert n == base + 1
        else:
            # the solve as its own launches: gather, scatter, scaling, product and three for each
            # of one to eight refinement steps; two parts of the kernel around it
            solve = n - base - (2 if rule else 0)
            assert solve in [4 + 3 * k for k in range(1, 9)]


@pytest.mark.parametrize("case", ["solve of 384", "solve of 385", "256 alone", "258 alone",
                                  "48 alone", "49 alone"])
def test_cycles_on_either_side_match_the_oracle(case):
    from oracle import cycle, hierarchy
    make, levels, _, rules = RULES[case]
    p = make()
    oracle = hierarchy.build(p, levels)
    mg = cycle.RegionalMG(oracle, cycle.Options(smoother="chebyshev", nu1=1, nu2=1, degree=3))
    L0 = oracle[0].layout
    want = L0.average_to_composite(mg.precondition(L0.to_regional(p.b)))
    for precision in rules:
        if precision == "FP32_BF16COEF":
            continue
        dp, h = _hier(p, levels, precision)
        z = torch.empty_like(dp.b)
        h.vcycle(dp.b, z)
        assert rel_max(z.cpu().numpy(), want) <= (1e-10 if precision == "FP64" else 1e-4)


def test_blocks_inside():
    """3-dof blocks: two levels inside, against the block oracle."""
    from oracle import cycle, hierarchy
    p = W.elasticity3d(region_grid=(2, 1, 1), choices=(28,), seed=4)
    oracle = hierarchy.build_block(p, 3)
    mg = cycle.RegionalMG(oracle, cycle.Options(smoother="chebyshev", nu1=1, nu2=1, degree=3,
                                                power_iters=30))
    L0 = oracle[0].layout
    perm = hierarchy.node_major_to_component_major(p.n_nodes, 3)
    want = np.empty(3 * p.n_nodes)
    want[perm] = L0.average_to_composite(mg.precondition(L0.to_regional(p.b[perm])))
    for precision, tol in (("FP64", 1e-10), ("FP32", 1e-4)):
        dp, h = _hier(p, 3, precision, B=3)
        assert h.vcycle_launches() == _outside(1, "CHEBYSHEV", [0], B=3) + 1
        z = torch.empty_like(dp.b)
        h.vcycle(dp.b, z)
        assert rel_max(z.cpu().numpy(), want) <= tol


@pytest.mark.parametrize("precision,tol", [("FP64", 1e-10), ("FP32", 1e-4)])
@pytest.mark.parametrize("dim", [2, 3])
def test_stored_weights_inside(dim, precision, tol):
    """Weights stored on a level that the kernel takes, against the oracle with the same ones."""
    from oracle import cycle, hierarchy
    from paper_2103_11962_gb300 import rmg
    p = W.q1_laplace2d((2, 2), 28) if dim == 2 else W.q1_laplace3d((2, 1, 1), 28)
    dp, h = _hier(p, 3, precision)
    n = h.level_sizes(1)[0]
    wr = torch.empty(3 * n, dtype=torch.float32, device="cuda")
    h.constant_weights(1, wr)
    h.set_transfer_weights(1, wr)
    h.setup_numeric()
    assert h.vcycle_launches() == _outside(1, "CHEBYSHEV", [0]) + 1
    z = torch.empty_like(dp.b)
    h.vcycle(dp.b, z)
    # the same by composite node of level 1 (weight 1 from the right where the remainder is 2)
    N = [(v - 1) // 3 + 1 for v in p.global_dims]
    z1, y1, x1 = np.meshgrid(*(np.arange(v) for v in reversed(N)), indexing="ij")
    w1 = np.stack([(c.reshape(-1) % 3 == 2).astype(np.float32) for c in (x1, y1, z1)])
    oracle = hierarchy.build(p, 3, weights=lambda l, lev: w1 if l == 1 else None)
    mg = cycle.RegionalMG(oracle, cycle.Options(smoother="chebyshev", nu1=1, nu2=1, degree=3))
    L0 = oracle[0].layout
    want = L0.average_to_composite(mg.precondition(L0.to_regional(p.b)))
    assert rel_max(z.cpu().numpy(), want) <= tol
