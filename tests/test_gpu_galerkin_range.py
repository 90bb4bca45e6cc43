"""The FP32 Galerkin product holds whatever coarse coefficients FP32 holds: scaling an operator by a
power of two scales every coarse stencil by it, bit for bit, up to the end of the range."""
import math

import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.filterwarnings("ignore::scipy.sparse.SparseEfficiencyWarning")]

PROBLEMS = {
    "5-point": lambda: W.poisson2d_5pt(region_grid=(2, 1), n=28),
    "9-point": lambda: W.q1_laplace2d(region_grid=(2, 1), n=10),
    "7-point": lambda: W.diffusion3d_7pt(region_grid=(2, 1, 1), choices=(10, 19), seed=3),
    "27-point": lambda: W.q1_laplace3d(region_grid=(1, 2, 1), n=10),
}


@pytest.mark.parametrize("problem", list(PROBLEMS))
@pytest.mark.parametrize("precision", ["FP32", "FP64"])
def test_coarse_stencils_scale_with_the_operator(problem, precision):
    from paper_2103_11962_gb300 import rmg, upload
    p = PROBLEMS[problem]()
    dp = upload(p)
    ctx = rmg.Context(0)

    def coarse(scale):
        lay = rmg.Layout(ctx, p.dim, p.region_dims, dp.gids, p.n_nodes, dp.dirichlet)
        lay.operator_from_csr(p.stencil, dp.rowptr, dp.col, dp.val * scale)
        h = rmg.Hierarchy(lay, rmg.default_options(levels=2, smoother=rmg.JACOBI,
                                                   precision=getattr(rmg, precision)))
        n, _, kind = h.level_sizes(1)
        c = torch.empty(kind * n, dtype=torch.float64, device="cuda")
        h.level_export(1, c)
        return c

    one = coarse(1.0)
    kept = coarse(2.0) == one                  # identity rows of masked coarse nodes, and zeros
    # the largest coarse coefficient between 2^122 and 2^123 (FP32 ends at 2^128): room for the
    # partial sums of a product, which are a few times its result
    scale = 2.0 ** (122 - math.floor(math.log2(float(one[~kept].abs().max()))))
    got = coarse(scale)
    assert torch.equal(got[kept], one[kept])
    assert torch.equal(got[~kept], one[~kept] * scale)
    assert 2.0 ** 122 <= float(got.abs().max()) < 2.0 ** 123
