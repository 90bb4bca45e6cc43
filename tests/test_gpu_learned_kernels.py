"""Edges of the learned prolongator's kernels: the one-pass weights against features, network and
masking as separate calls, and the gradient's tiles of 128 samples and remainders."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.filterwarnings("ignore::scipy.sparse.SparseEfficiencyWarning")]


@pytest.fixture(scope="module")
def ctx():
    from paper_2103_11962_gb300 import rmg
    return rmg.Context(0)


PROBLEMS = {
    "5-point": lambda: W.poisson2d_5pt(region_grid=(3, 2), n=28),
    "9-point": lambda: W.q1_laplace2d(region_grid=(2, 2), n=10),
    "7-point": lambda: W.highcontrast3d_7pt(region_grid=(3, 2, 2), choices=(10, 19), seed=4),
    "27-point": lambda: W.q1_laplace3d(region_grid=(2, 2, 2), n=10),
}


@pytest.mark.parametrize("problem", list(PROBLEMS))
def test_weights_are_features_then_network(ctx, problem):
    from paper_2103_11962_gb300 import learned, rmg, upload
    p = PROBLEMS[problem]()
    dp = upload(p)
    lay = rmg.Layout(ctx, p.dim, p.region_dims, dp.gids, p.n_nodes, dp.dirichlet)
    lay.operator_from_csr(p.stencil, dp.rowptr, dp.col, dp.val)
    h = rmg.Hierarchy(lay, learned._options(3, "chebyshev"))
    net = rmg.MLP(ctx, learned.init_params(5))
    for level in (0, 1):
        n = h.level_sizes(level)[0]
        feats = torch.full((n, 32), float("nan"), device="cuda")
        off = torch.full((n * 32 + 1,), float("nan"), device="cuda")
        out = torch.empty((n, 3), device="cuda")
        wr = torch.full((3 * n,), float("nan"), device="cuda")
        h.mlp_features(level, feats)
        h.mlp_features(level, off[1:])             # rows that are only 4-byte aligned
        assert torch.equal(off[1:].view(n, 32), feats)
        net.forward(feats, out)
        h.mlp_weights(level, net, wr)
        active = feats[:, 8:27:9] > 0.5
        want = torch.where(active, out, torch.zeros_like(out)).t().reshape(-1)
        # the same operations in the same order: equal bits
        assert torch.equal(wr, want)


@pytest.mark.parametrize("n", [1, 127, 128, 129, 152 * 128 + 5, 2 * 152 * 128 + 127])
def test_gradient_tiles_and_remainders(ctx, n):
    """Only a few rows carry a nonzero mask: first, last, and around every tile edge. They must
    give the gradient of those rows alone (times the ratio of the normalisations); the forward
    values of a row do not depend on its place, so only the FP32 order of the sums differs
    (a few dozen terms: 64 units of 2^-24 of the largest entry)."""
    from paper_2103_11962_gb300 import learned, rmg
    rng = np.random.default_rng(n)
    rows = sorted({r for r in (0, 1, 63, 126, 127, 128, n // 2, n - 129, n - 2, n - 1)
                   if 0 <= r < n})
    feats = torch.from_numpy(rng.normal(size=(n, 32)).astype(np.float32)).cuda()
    labels = torch.from_numpy(rng.uniform(size=(n, 3)).astype(np.float32)).cuda()
    mask = torch.zeros((n, 3), device="cuda")
    mask[rows] = 1.0
    net = rmg.MLP(ctx, learned.init_params(3))
    loss, g = net.gradient(feats, labels, mask)
    loss1, g1 = net.gradient(feats[rows].contiguous(), labels[rows].contiguous(),
                             mask[rows].contiguous())
    scale = len(rows) / n
    tol = 64 * 2.0 ** -24
    assert abs(loss - loss1 * scale) <= tol * loss1 * scale
    assert np.abs(g - g1 * scale).max() <= tol * np.abs(g1).max() * scale


@pytest.mark.parametrize("problem", ["9-point", "7-point"])
def test_features_beside_a_cycle_on_another_stream(ctx, problem):
    """Features and weights only read what a cycle reads: formed on another stream while FP64
    cycles are queued, they change neither the cycles' results nor their own."""
    from paper_2103_11962_gb300 import learned, rmg, upload
    p = PROBLEMS[problem]()
    dp = upload(p)
    own = rmg.Context(0)
    lay = rmg.Layout(own, p.dim, p.region_dims, dp.gids, p.n_nodes, dp.dirichlet)
    lay.operator_from_csr(p.stencil, dp.rowptr, dp.col, dp.val)
    h = rmg.Hierarchy(lay, rmg.default_options(levels=3, smoother=rmg.CHEBYSHEV, nu1=1, nu2=1,
                                               precision=rmg.FP64))
    net = rmg.MLP(own, learned.init_params(5))
    n = [h.level_sizes(l)[0] for l in range(3)]
    want_z = torch.empty_like(dp.b)
    h.vcycle(dp.b, want_z)
    want = []
    for l in range(3):
        want.append((torch.empty(n[l], 32, device="cuda"), torch.empty(3 * n[l], device="cuda")))
        h.mlp_features(l, want[l][0])
        h.mlp_weights(l, net, want[l][1])
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    z = [torch.empty_like(dp.b) for _ in range(8)]
    got = [[torch.empty_like(t) for t in w] for w in want]
    torch.cuda.synchronize()
    for k in range(8):
        own.set_stream(a.cuda_stream)
        h.vcycle(dp.b, z[k])
        own.set_stream(b.cuda_stream)
        for l in range(3):
            h.mlp_features(l, got[l][0])
            h.mlp_weights(l, net, got[l][1])
    torch.cuda.synchronize()
    for k in range(8):
        assert torch.equal(z[k], want_z)
    for w, g in zip(want, got):
        assert torch.equal(w[0], g[0]) and torch.equal(w[1], g[1])
