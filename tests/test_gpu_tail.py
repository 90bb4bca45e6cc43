"""The coarse levels of a cycle in one kernel: cycles against the oracle where its rule changes
(solve inside or outside, several levels, one level, all smoothers)."""
import pytest

import workloads as W
from tests.gpu_common import rel_max

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.filterwarnings("ignore::scipy.sparse.SparseEfficiencyWarning")]

# problem, levels: the coarsest level alone; several levels with the solve inside; a coarsest
# level above 768 unknowns, solved by its own launches between two parts of the kernel
CASES = {
    "coarsest only": (lambda: W.q1_laplace3d(region_grid=(2, 1, 2), n=10), 2),
    "2D, solve inside": (lambda: W.q1_laplace2d(region_grid=(3, 2), n=28), 4),
    "3D, solve inside": (lambda: W.diffusion3d_7pt(region_grid=(2, 2, 1), choices=(10, 28),
                                                   seed=3), 3),
    "2D, solve outside": (lambda: W.q1_laplace2d(region_grid=(11, 10), n=28), 3),
}


@pytest.mark.parametrize("case", list(CASES))
@pytest.mark.parametrize("smoother", ["jacobi", "chebyshev", "gs"])
def test_cycle_matches_oracle(case, smoother):
    from oracle import cycle, hierarchy
    from paper_2103_11962_gb300 import rmg, upload
    make, levels = CASES[case]
    p = make()
    dp = upload(p)
    ctx = rmg.Context(0)
    lay = rmg.Layout(ctx, p.dim, p.region_dims, dp.gids, p.n_nodes, dp.dirichlet)
    lay.operator_from_csr(p.stencil, dp.rowptr, dp.col, dp.val)
    code = dict(jacobi=rmg.JACOBI, chebyshev=rmg.CHEBYSHEV, gs=rmg.GAUSS_SEIDEL)[smoother]
    kw = dict(levels=levels, smoother=code, nu1=1, nu2=2, cheb_degree=3, omega=0.67)
    oracle = hierarchy.build(p, levels)
    mg = cycle.RegionalMG(oracle, cycle.Options(smoother=smoother, nu1=1, nu2=2, degree=3,
                                                omega=0.67))
    L0 = oracle[0].layout
    want = L0.average_to_composite(mg.precondition(L0.to_regional(p.b)))
    z = torch.empty_like(dp.b)
    for precision, tol in ((rmg.FP64, 1e-10), (rmg.FP32, 1e-4)):
        h = rmg.Hierarchy(lay, rmg.default_options(precision=precision, **kw))
        h.vcycle(dp.b, z)
        assert rel_max(z.cpu().numpy(), want) <= tol
