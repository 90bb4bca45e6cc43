"""The split's direct pass: rows in column order go by position, every other form of the same row
goes entry by entry with the same result."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.filterwarnings("ignore::scipy.sparse.SparseEfficiencyWarning")]

PROBLEMS = {
    "5-point": (lambda: W.poisson2d_5pt(region_grid=(2, 3), n=10), 5, 1),
    "9-point": (lambda: W.q1_laplace2d(region_grid=(3, 2), n=10), 9, 1),
    "7-point": (lambda: W.diffusion3d_7pt(region_grid=(2, 2, 1), choices=(10, 19), seed=2), 7, 1),
    "27-point": (lambda: W.q1_laplace3d(region_grid=(2, 1, 2), n=10), 27, 1),
    "27-point blocks": (lambda: W.elasticity3d(region_grid=(2, 1, 1), choices=(10,), seed=2), 27, 3),
}


def _split(ctx, p, kind, B, rowptr, col, val, gids):
    from paper_2103_11962_gb300 import rmg
    lay = rmg.Layout(ctx, p.dim, p.region_dims, gids, p.n_nodes, None)
    t = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (rowptr, col, val)]
    if B == 1:
        lay.operator_from_csr(kind, *t)
    else:
        lay.operator_from_block_csr(kind, B, *t)
    h = rmg.Hierarchy(lay, rmg.default_options(levels=1))
    n = h.level_sizes(0)[0]
    coef = torch.empty(B * B * kind * n, dtype=torch.float64, device="cuda")
    h.level_export(0, coef)
    return coef.view(B, B, kind, n).cpu().numpy()


@pytest.mark.parametrize("name", list(PROBLEMS))
def test_forms_of_a_row(name):
    from paper_2103_11962_gb300 import rmg
    make, kind, B = PROBLEMS[name]
    p = make()
    A = p.A.tocsr()
    A.sort_indices()
    rp, col, val = A.indptr.astype(np.int64), A.indices.astype(np.int64), A.data.copy()
    # every entry its own value (and the matrix still positive definite)
    val *= 1.0 + 1e-6 * np.random.default_rng(1).uniform(-1.0, 1.0, val.size)
    gids = torch.from_numpy(np.asarray(p.region_gids, dtype=np.int64)).cuda()
    ctx = rmg.Context(0)
    want = _split(ctx, p, kind, B, rp, col, val, gids)
    copies = np.bincount(p.region_gids, minlength=p.n_nodes)
    single = copies[p.region_gids] == 1
    # the matrix entries themselves at single-copy rows (centre included)
    full = np.flatnonzero((np.diff(rp).reshape(-1, B).min(1) == B * kind) & (copies == 1))
    where = {int(g): n for n, g in enumerate(p.region_gids)}
    for g in full[:: max(1, full.size // 50)]:
        for c in range(B):
            row = val[rp[g * B + c]:rp[g * B + c + 1]].reshape(kind, B)
            assert np.array_equal(want[c, :, :, where[int(g)]].T, row)
    # entries of every row in another order: the same bits in single-copy rows, sums in another
    # order in shared ones (a row has at most 81 entries)
    rng = np.random.default_rng(2)
    col2, val2 = col.copy(), val.copy()
    for r in range(rp.size - 1):
        o = rp[r] + rng.permutation(rp[r + 1] - rp[r])
        col2[rp[r]:rp[r + 1]], val2[rp[r]:rp[r + 1]] = col[o], val[o]
    got = _split(ctx, p, kind, B, rp, col2, val2, gids)
    assert np.array_equal(got[..., single], want[..., single])
    assert np.abs(got - want).max() <= 81 * 2.0 ** -52 * np.abs(val).max()
    # one full row whose first column appears twice and whose second is missing
    g = int(full[full.size // 2])
    k = rp[g * B]
    col3 = col.copy()
    col3[k + B] = col3[k]
    got = _split(ctx, p, kind, B, rp, col3, val, gids)
    expect = want.copy()
    expect[0, 0, 0, where[g]] = val[k] + val[k + B]
    expect[0, 0, 1, where[g]] = 0.0
    assert np.array_equal(got, expect)


@pytest.mark.parametrize("name", list(PROBLEMS))
def test_orders_of_a_row(name):
    """Orders that programs write rows in: the same bits in single-copy rows, whose entries each
    have a slot of their own, and sums in another order in shared ones."""
    from paper_2103_11962_gb300 import rmg
    make, kind, B = PROBLEMS[name]
    p = make()
    A = p.A.tocsr()
    A.sort_indices()
    rp, col, val = A.indptr.astype(np.int64), A.indices.astype(np.int64), A.data.copy()
    val *= 1.0 + 1e-6 * np.random.default_rng(3).uniform(-1.0, 1.0, val.size)
    gids = torch.from_numpy(np.asarray(p.region_gids, dtype=np.int64)).cuda()
    ctx = rmg.Context(0)
    want = _split(ctx, p, kind, B, rp, col, val, gids)
    single = np.bincount(p.region_gids, minlength=p.n_nodes)[p.region_gids] == 1
    row = np.repeat(np.arange(rp.size - 1), np.diff(rp))
    swap = col.copy()                          # the last two entries of a row change places
    swap[rp[1:] - 1], swap[rp[1:] - 2] = col[rp[1:] - 2], col[rp[1:] - 1]
    orders = {"diagonal first": col != row, "diagonal last": col == row, "descending": -col,
              "by component": col % B, "last two": swap}
    for order, key in orders.items():
        o = np.lexsort((col, key, row)) if order != "last two" else np.lexsort((swap, row))
        got = _split(ctx, p, kind, B, rp, np.ascontiguousarray(col[o]), val[o], gids)
        assert np.array_equal(got[..., single], want[..., single]), order
        assert np.abs(got - want).max() <= 81 * 2.0 ** -52 * np.abs(val).max(), order


# sizes that the direct pass takes, with the rows it lists and the regions it leaves
LARGE = {
    "5-point": (lambda: W.poisson2d_5pt(region_grid=(14, 14), n=91), 5, 1, 8000000),
    "9-point": (lambda: W.q1_laplace2d(region_grid=(10, 11), n=91), 9, 1, 8000000),
    "7-point": (lambda: W.diffusion3d_7pt(region_grid=(4, 4, 3), choices=(31,), seed=2), 7, 1,
                8000000),
    "27-point": (lambda: W.q1_laplace3d(region_grid=(2, 3, 2), n=25), 27, 1, 4000000),
    "27-point blocks": (lambda: W.elasticity3d(region_grid=(2, 2, 2), choices=(25,), seed=2), 27, 3,
                        24000000),
}


@pytest.mark.parametrize("name", list(LARGE))
def test_direct_pass_against_the_general_one(name):
    """Rows in column order go by position; with rows the other way round the same regions go entry
    by entry, and with a few rows of that kind, or with a column twice, those go through the list.
    The same bits in single-copy rows, sums in another order in shared ones."""
    from paper_2103_11962_gb300 import rmg
    make, kind, B, line = LARGE[name]
    p = make()
    assert p.n_regional_nodes * kind * B * B >= line
    A = p.A.tocsr()
    A.sort_indices()
    rp, col, val = A.indptr.astype(np.int64), A.indices.astype(np.int64), A.data.copy()
    rng = np.random.default_rng(5)
    val *= 1.0 + 1e-6 * rng.uniform(-1.0, 1.0, val.size)
    gids = torch.from_numpy(np.asarray(p.region_gids, dtype=np.int64)).cuda()
    ctx = rmg.Context(0)
    want = _split(ctx, p, kind, B, rp, col, val, gids)
    copies = np.bincount(p.region_gids, minlength=p.n_nodes)
    single = copies[p.region_gids] == 1
    row = np.repeat(np.arange(rp.size - 1), np.diff(rp))
    at = np.arange(col.size)
    back = rp[row] + rp[row + 1] - 1 - at      # the entries of every row the other way round
    for some in (np.ones(rp.size - 1, bool), rng.uniform(size=rp.size - 1) < 0.01):
        o = np.where(some[row], back, at)
        got = _split(ctx, p, kind, B, rp, col[o], val[o], gids)
        assert np.array_equal(got[..., single], want[..., single])
        assert np.abs(got - want).max() <= 81 * 2.0 ** -52 * np.abs(val).max()
    full = np.flatnonzero((np.diff(rp).reshape(-1, B).min(1) == B * kind) & (copies == 1))
    g = int(full[full.size // 3])
    col[rp[g * B] + B] = col[rp[g * B]]
    got = _split(ctx, p, kind, B, rp, col, val, gids)
    n = int(np.flatnonzero(p.region_gids == g)[0])
    want[0, 0, 0, n] = val[rp[g * B]] + val[rp[g * B] + B]
    want[0, 0, 1, n] = 0.0
    assert np.array_equal(got, want)
