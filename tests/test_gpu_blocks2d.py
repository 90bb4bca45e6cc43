"""Block operators on a 9-point stencil (3 dofs per node in 2D): the split, the Galerkin product,
the cycle with its coarse end in one kernel, and the half planes."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_common import matrix_rel_diff, rel_max, stencils_to_matrix

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.filterwarnings("ignore::scipy.sparse.SparseEfficiencyWarning")]


def _problem(region_grid, n, seed):
    """Bilinear elements whose coefficient is a 3 x 3 symmetric positive definite matrix of the
    element's own, zero at the boundary."""
    slabs = ([n] * region_grid[0], [n] * region_grid[1], [1])
    gdims, rdims, gids = W.region_map(slabs)
    Nx, Ny, _ = gdims
    rng = np.random.default_rng(seed)
    kappa = rng.uniform(-0.3, 0.3, (3, 3, 1, Ny - 1, Nx - 1))
    kappa += kappa.transpose(1, 0, 2, 3, 4)
    kappa[np.arange(3), np.arange(3)] += 2.5      # diagonally dominant: off-diagonals below 0.6
    Ke = np.array([[4, -1, -1, -2], [-1, 4, -2, -1], [-1, -2, 4, -1], [-2, -1, -1, 4]]) / 6.0
    corners = [(0, 0), (1, 0), (0, 1), (1, 1)]
    vals = np.zeros((9, 3, 3, 1, Ny, Nx))
    for a, (ax, ay) in enumerate(corners):
        for c, (cx, cy) in enumerate(corners):
            s = (cx - ax + 1) + 3 * (cy - ay + 1)
            vals[s, :, :, :, ay:ay + Ny - 1, ax:ax + Nx - 1] += Ke[a, c] * kappa
    mask = W.boundary_mask(gdims)
    A = W._csr_from_block_stencil(gdims, W.OFFS9, vals, mask, 3)
    b = rng.uniform(-1.0, 1.0, A.shape[0]) * np.repeat(mask == 0, 3)
    return W.Problem("blocks2d", 2, 3, gdims, slabs, rdims, gids, mask, A, b, 9)


def _layout(ctx, p, dp, val=None):
    from paper_2103_11962_gb300 import rmg
    lay = rmg.Layout(ctx, 2, p.region_dims, dp.gids, p.n_nodes, dp.dirichlet)
    lay.operator_from_block_csr(9, 3, dp.rowptr, dp.col, dp.val if val is None else val)
    return lay


# one level below the finest, two; regions of one run of 256 nodes and of several
@pytest.mark.parametrize("grid,n,levels", [((2, 2), 10, 2), ((3, 2), 10, 3), ((2, 1), 28, 3)])
def test_operators_and_cycle_match_oracle(grid, n, levels):
    import scipy.sparse as sp
    from oracle import cycle, hierarchy
    from paper_2103_11962_gb300 import rmg, upload
    p = _problem(grid, n, seed=n)
    dp = upload(p)
    oracle = hierarchy.build_block(p, levels)
    mg = cycle.RegionalMG(oracle, cycle.Options(smoother="chebyshev", nu1=1, nu2=1, degree=3,
                                                power_iters=30))
    L0 = oracle[0].layout
    perm = hierarchy.node_major_to_component_major(p.n_nodes, 3)
    want = np.empty(3 * p.n_nodes)
    want[perm] = L0.average_to_composite(mg.precondition(L0.to_regional(p.b[perm])))
    ctx = rmg.Context(0)
    lay = _layout(ctx, p, dp)
    for precision, tol in ((rmg.FP64, 1e-10), (rmg.FP32, 1e-4)):
        h = rmg.Hierarchy(lay, rmg.default_options(levels=levels, smoother=rmg.CHEBYSHEV, nu1=1,
                                                   nu2=1, cheb_degree=3, power_iters=30,
                                                   precision=precision))
        z = torch.empty_like(dp.b)
        h.vcycle(dp.b, z)
        assert rel_max(z.cpu().numpy(), want) <= tol
        if precision != rmg.FP64:
            continue
        for l, lev in enumerate(oracle):
            n_r, _, kind = h.level_sizes(l)
            coef = torch.empty(9 * kind * n_r, dtype=torch.float64, device="cuda")
            h.level_export(l, coeffs=coef)
            c = coef.cpu().numpy().reshape(3, 3, kind * n_r)
            M = sp.bmat([[stencils_to_matrix(lev.layout.region_dims, c[i, j], kind)
                          for j in range(3)] for i in range(3)], format="csr")
            assert matrix_rel_diff(M, lev.Ar) <= 1e-12, l


@pytest.mark.parametrize("symmetric", [True, False])
@pytest.mark.parametrize("tile_shape", [-1, 0, 4])
def test_half_planes_give_the_same_bits(symmetric, tile_shape):
    from paper_2103_11962_gb300 import rmg, upload
    p = _problem((2, 2), 19, seed=4)
    dp = upload(p)
    val = dp.val.clone()
    if not symmetric:
        row = 3 * int(np.flatnonzero(np.bincount(p.region_gids) == 1)[150]) + 1
        k = int(dp.rowptr[row])
        k += int(torch.nonzero(dp.col[k:int(dp.rowptr[row + 1])] // 3 != row // 3)[0])
        val[k] *= 1.0 + 2.0 ** -20
    ctx = rmg.Context(0)
    lay = _layout(ctx, p, dp, val)
    z, regions = [], []
    for storage in (1, 0):
        h = rmg.Hierarchy(lay, rmg.default_options(
            levels=3, smoother=rmg.CHEBYSHEV, nu1=1, nu2=1, power_iters=10, precision=rmg.FP32,
            symmetric_storage=storage, tile_shape=tile_shape))
        regions.append(h.half_regions(0)[0])
        out = torch.empty_like(dp.b)
        h.vcycle(dp.b, out)
        z.append(out)
    assert regions == [4 if symmetric else 3, 0]
    assert torch.equal(z[0], z[1])


def test_split_takes_rows_in_any_order():
    """Rows in column order go to their slots by position, the same rows the other way round entry
    by entry: the same bits in single-copy rows, sums in another order in shared ones (a row has
    27 entries)."""
    from paper_2103_11962_gb300 import rmg, upload
    p = _problem((2, 2), 13, seed=7)
    dp = upload(p)
    rp = dp.rowptr.cpu().numpy()
    row = np.repeat(np.arange(rp.size - 1), np.diff(rp))
    col, val = dp.col.cpu().numpy(), dp.val.cpu().numpy()
    o = np.lexsort((-col, row))
    back = [torch.from_numpy(np.ascontiguousarray(a[o])).cuda() for a in (col, val)]
    ctx = rmg.Context(0)
    got = []
    for c, v in ((dp.col, dp.val), back):
        lay = rmg.Layout(ctx, 2, p.region_dims, dp.gids, p.n_nodes, dp.dirichlet)
        lay.operator_from_block_csr(9, 3, dp.rowptr, c, v)
        h = rmg.Hierarchy(lay, rmg.default_options(levels=1))
        coef = torch.empty(81 * p.n_regional_nodes, dtype=torch.float64, device="cuda")
        h.level_export(0, coef)
        got.append(coef.cpu().numpy().reshape(81, -1))
    single = np.bincount(p.region_gids)[p.region_gids] == 1
    assert np.array_equal(got[0][:, single], got[1][:, single])
    assert np.abs(got[0] - got[1]).max() <= 27 * 2.0 ** -52 * np.abs(val).max()
