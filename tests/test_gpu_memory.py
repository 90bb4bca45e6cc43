"""Device memory that calls keep."""
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.filterwarnings("ignore::scipy.sparse.SparseEfficiencyWarning")]


def test_split_keeps_the_operator_only():
    """Between calls a layout holds the coefficients of the split and the region of every node; the
    list of rows that the direct pass leaves has its place in the apply's scratch vector."""
    from paper_2103_11962_gb300 import rmg, upload
    from workloads import device
    ctx = rmg.Context(0)
    small = upload(W.diffusion3d_7pt(region_grid=(2, 1, 1), choices=(10,), seed=1))

    def layout(p, gids, mask):
        return rmg.Layout(ctx, 3, p.region_dims, gids, p.n_nodes, mask)

    q = W.diffusion3d_7pt(region_grid=(2, 1, 1), choices=(10,), seed=1)
    warm = layout(q, small.gids, small.dirichlet)      # the kernels are loaded
    warm.operator_from_csr(7, small.rowptr, small.col, small.val)
    p = device.diffusion3d_7pt(region_grid=(2, 2, 2), choices=(82,))
    gids = torch.from_numpy(p.region_gids).cuda()
    mask = torch.from_numpy(p.dirichlet).cuda()
    lay = layout(p, gids, mask)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    lay.operator_from_csr(7, p.rowptr, p.col, p.val)
    n = p.n_regional_nodes
    took = free - torch.cuda.mem_get_info()[0]
    # 4.4M nodes: 60 bytes each; granules of 2 MB for each of a few arrays
    assert took <= 60 * n + 2 ** 24
