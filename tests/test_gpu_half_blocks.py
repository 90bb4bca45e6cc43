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


def _asymmetric(p, dp, regions):
    """The matrix with one coupling inside each of the regions moved in its last bits."""
    import numpy as np
    val = dp.val.clone()
    rp = dp.rowptr.cpu().numpy()
    inner = np.bincount(p.region_gids, minlength=p.n_nodes) == 1
    off = np.concatenate([[0], np.cumsum(np.prod(np.asarray(p.region_dims), axis=1))])
    for r in regions:
        own = p.region_gids[off[r]:off[r + 1]]
        for g in own[inner[own]]:
            cols = dp.col[int(rp[3 * g]):int(rp[3 * g + 1])].cpu().numpy()
            k = np.flatnonzero(inner[cols // 3] & (cols // 3 != g))
            if k.size:
                val[int(rp[3 * g]) + int(k[0])] *= 1.0 + 2.0 ** -20
                break
    return val


def test_half_planes_go_when_no_region_uses_them():
    """A hierarchy whose operator turns asymmetric in every region gives the memory of its half
    planes back, and takes it again when a region turns symmetric; the cycle stays that of the
    full planes."""
    from paper_2103_11962_gb300 import rmg, upload
    p = W.elasticity3d(region_grid=(2, 1, 1), choices=(28,), seed=5)
    dp = upload(p)
    ctx = rmg.Context(0)
    lay = rmg.Layout(ctx, 3, p.region_dims, dp.gids, p.n_nodes, dp.dirichlet)
    lay.operator_from_block_csr(27, 3, dp.rowptr, dp.col, dp.val)
    opts = dict(levels=2, smoother=rmg.CHEBYSHEV, nu1=1, nu2=1, precision=rmg.FP32)
    h = rmg.Hierarchy(lay, rmg.default_options(symmetric_storage=1, **opts))
    full = rmg.Hierarchy(lay, rmg.default_options(symmetric_storage=0, **opts))
    size = 4 * 126 * p.n_regional_nodes
    steps = [(0, 1), (0, 1), (1,), (), (0, 1)]
    vals = [_asymmetric(p, dp, moved) for moved in steps]
    z = [torch.empty_like(dp.b) for _ in range(2)]
    free = torch.cuda.mem_get_info()[0]        # with the planes, and all tensors of this test
    for moved, val in zip(steps, vals):
        lay.operator_from_block_csr(27, 3, dp.rowptr, dp.col, val)
        h.setup_numeric()
        full.setup_numeric()
        assert h.half_regions(0)[0] == 2 - len(moved)
        # device memory comes in granules of up to 2 MB; the planes take 22
        gained = torch.cuda.mem_get_info()[0] - free
        assert abs(gained - (size if len(moved) == 2 else 0)) <= 2 ** 23
        h.vcycle(dp.b, z[0])
        full.vcycle(dp.b, z[1])
        assert torch.equal(z[0], z[1])


def test_no_half_planes_where_memory_is_short():
    """Half planes of a block operator that would not leave as much memory free as they take are
    not made: what fits without them still does, with the same results."""
    from paper_2103_11962_gb300 import rmg, upload
    p = W.elasticity3d(region_grid=(2, 2, 1), choices=(28,), seed=6)
    dp = upload(p)
    ctx = rmg.Context(0)
    lay = rmg.Layout(ctx, 3, p.region_dims, dp.gids, p.n_nodes, dp.dirichlet)
    lay.operator_from_block_csr(27, 3, dp.rowptr, dp.col, dp.val)
    opts = rmg.default_options(levels=2, smoother=rmg.CHEBYSHEV, nu1=1, nu2=1, precision=rmg.FP32)
    size = 4 * 126 * p.n_regional_nodes
    want, got = torch.empty_like(dp.b), torch.empty_like(dp.b)
    for _ in range(2):                         # the first time loads kernels as well
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        before = torch.cuda.mem_get_info()[0]
        h = rmg.Hierarchy(lay, opts)
        assert h.half_regions(0)[0] == 4
        h.vcycle(dp.b, want)
        torch.cuda.synchronize()
        took = before - torch.cuda.mem_get_info()[0]
        h.close()
    # all but what the hierarchy takes and half of its half planes
    left = torch.cuda.mem_get_info()[0] - took - size // 2
    held = torch.empty(left, dtype=torch.uint8, device="cuda")
    h = rmg.Hierarchy(lay, opts)
    assert h.half_regions(0) == (0, 0) and h.coef_planes(0) == 243
    h.vcycle(dp.b, got)
    assert torch.equal(got, want)
    h.setup_numeric()                          # decided once: later setups change nothing
    assert h.half_regions(0) == (0, 0)
    h.vcycle(dp.b, got)
    assert torch.equal(got, want)
    del held
    torch.cuda.empty_cache()
