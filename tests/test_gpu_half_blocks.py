"""Half planes of block operators: bit for bit the full planes, and given up when the operator is
not symmetric."""
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.filterwarnings("ignore::scipy.sparse.SparseEfficiencyWarning")]


# regions at the edge of one tile (7^3 nodes are one run and a remainder), several runs, ragged
@pytest.mark.parametrize("grid,choices", [((1, 1, 1), (7,)), ((2, 1, 2), (10,)),
                                          ((2, 2, 1), (10, 19))])
@pytest.mark.parametrize("symmetric", [True, False])
@pytest.mark.parametrize("tile_shape", [-1, 0, 8])
def test_block_half_planes(grid, choices, symmetric, tile_shape):
    from paper_2103_11962_gb300 import rmg, upload
    p = W.elasticity3d(region_grid=grid, choices=choices, seed=3)
    dp = upload(p)
    val = dp.val.clone()
    if not symmetric:
        # one coupling of a free node to another
        row = 3 * (p.n_nodes // 2 + 3) + 1
        k = int(dp.rowptr[row])
        k += int(torch.nonzero(dp.col[k:int(dp.rowptr[row + 1])] // 3 != row // 3)[0])
        val[k] *= 1.0 + 2.0 ** -20
    ctx = rmg.Context(0)
    lay = rmg.Layout(ctx, 3, p.region_dims, dp.gids, p.n_nodes, dp.dirichlet)
    lay.operator_from_block_csr(27, 3, dp.rowptr, dp.col, val)
    z, lam = [], []
    for storage in (1, 0):
        h = rmg.Hierarchy(lay, rmg.default_options(
            levels=2, smoother=rmg.CHEBYSHEV, nu1=1, nu2=1, cheb_degree=3, power_iters=10,
            precision=rmg.FP32, symmetric_storage=storage, tile_shape=tile_shape))
        assert h.coef_planes(0) == 9 * (14 if storage and symmetric else 27)
        out = torch.empty_like(dp.b)
        h.vcycle(dp.b, out)
        z.append(out)
        lam.append(h.lam(0))
    assert lam[0] == lam[1]
    assert torch.equal(z[0], z[1])


def test_half_regions_are_counted_one_by_one():
    """One region with a coupling of its own: the others stay on the half form, and are counted."""
    import numpy as np
    from paper_2103_11962_gb300 import rmg, upload
    p = W.elasticity3d(region_grid=(2, 1, 1), choices=(7, 10), seed=5)
    dp = upload(p)
    sizes = np.prod(np.asarray(p.region_dims), axis=1)
    inner = np.bincount(p.region_gids, minlength=p.n_nodes) == 1
    last = p.region_gids[sizes[0]:]
    ctx = rmg.Context(0)
    lay = rmg.Layout(ctx, 3, p.region_dims, dp.gids, p.n_nodes, dp.dirichlet)

    def numbers(val, precision=rmg.FP32):
        lay.operator_from_block_csr(27, 3, dp.rowptr, dp.col, val)
        h = rmg.Hierarchy(lay, rmg.default_options(levels=2, precision=precision))
        return h.half_regions(0), h.half_regions(1), h.coef_planes(0)

    assert numbers(dp.val) == ((2, int(sizes.sum())), (0, 0), 126)
    val = dp.val.clone()
    rp = dp.rowptr.cpu().numpy()
    for g in last[inner[last]]:                # a row of the second region alone
        cols = dp.col[int(rp[3 * g]):int(rp[3 * g + 1])].cpu().numpy()
        k = np.flatnonzero(inner[cols // 3] & (cols // 3 != g))
        if k.size:
            val[int(rp[3 * g]) + int(k[0])] *= 1.0 + 2.0 ** -20
            break
    assert numbers(val) == ((1, int(sizes[0])), (0, 0), 243)
    assert numbers(dp.val, rmg.FP64) == ((0, 0), (0, 0), 243)
