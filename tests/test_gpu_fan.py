"""Regions around a vertex of high valence: m square regions share one node, and each shares an
edge with the next. Nodes with more than eight copies take the loops behind the unrolled sums of
the interface phases; the cycle is compared with the same cycle in dense matrices."""
import numpy as np
import pytest

from tests.gpu_common import OFFSETS, rel_max, stencils_to_matrix

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _fan(m, n):
    """Region sizes and composite ids: node 0 is the vertex, region k's edge i = 0 is region
    (k + 1)'s edge j = 0."""
    edge = lambda k, s: 1 + (k % m) * (n - 1) + s - 1                       # noqa: E731
    inner = lambda k, i, j: 1 + m * (n - 1) + k * (n - 1) ** 2 + (i - 1) + (n - 1) * (j - 1)  # noqa: E731
    gids = []
    for k in range(m):
        for j in range(n):
            for i in range(n):
                if i == 0 and j == 0:
                    gids.append(0)
                elif j == 0:
                    gids.append(edge(k, i))
                elif i == 0:
                    gids.append(edge(k + 1, j))
                else:
                    gids.append(inner(k, i, j))
    return np.array([[n, n, 1]] * m, dtype=np.int32), np.array(gids, dtype=np.int64)


def _stencils(dims, seed):
    """9-point region stencils, symmetric and diagonally dominant, another coupling at every pair."""
    rng = np.random.default_rng(seed)
    out = []
    for nx, ny, _ in dims:
        c = np.zeros((9, ny, nx))
        for s, (dx, dy, _) in enumerate(OFFSETS[9]):
            if s <= 4:
                continue
            v = -rng.uniform(0.5, 1.0, (ny, nx))
            lo = (slice(max(0, -dy), ny - max(0, dy)), slice(max(0, -dx), nx - max(0, dx)))
            hi = (slice(max(0, dy), ny - max(0, -dy)), slice(max(0, dx), nx - max(0, -dx)))
            c[s][lo] = v[lo]
            c[8 - s][hi] = v[lo]
        c[4] = 0.05 - c.sum(0)
        out.append(c.reshape(9, -1))
    return np.concatenate(out, axis=1)


class _Dense:
    """The regional cycle (damped Jacobi) in dense matrices."""

    def __init__(self, dims, gids, A, levels, omega, nu):
        self.omega, self.nu, self.lev = omega, nu, []
        for l in range(levels):
            Psi = np.zeros((gids.max() + 1, gids.size))
            Psi[gids, np.arange(gids.size)] = 1.0
            used = np.flatnonzero(Psi.sum(1))
            Psi = Psi[used]
            S = Psi.T @ Psi
            L = dict(Psi=Psi, S=S, A=A, mult=S.sum(1), Dinv=1.0 / (S @ np.diag(A)))
            self.lev.append(L)
            if l + 1 == levels:
                break
            P, cg, off = [], [], 0
            for n in dims:
                nc = (n - 1) // 3 + 1
                p1 = np.maximum(0.0, 1.0 - np.abs(np.arange(n)[:, None] / 3.0 - np.arange(nc)))
                P.append(np.kron(p1, p1))
                g = gids[off:off + n * n].reshape(n, n)
                cg.append(g[::3, ::3].reshape(-1))
                off += n * n
            L["P"] = np.zeros((sum(p.shape[0] for p in P), sum(p.shape[1] for p in P)))
            r = c = 0
            for p in P:
                L["P"][r:r + p.shape[0], c:c + p.shape[1]] = p
                r, c = r + p.shape[0], c + p.shape[1]
            A = L["P"].T @ A @ L["P"]
            gids = np.concatenate(cg)
            dims = [(n - 1) // 3 + 1 for n in dims]

    def cycle(self, b, l=0):
        L = self.lev[l]
        if l + 1 == len(self.lev):
            M = L["Psi"] @ L["A"] @ L["Psi"].T
            bc = (L["Psi"] @ b) / L["Psi"].sum(1)
            return L["Psi"].T @ np.linalg.solve(M, bc)
        u = np.zeros_like(b)
        for _ in range(self.nu):
            u = u + self.omega * L["Dinv"] * (b - L["S"] @ (L["A"] @ u))
        r = (b - L["S"] @ (L["A"] @ u)) / L["mult"]
        C = self.lev[l + 1]
        u = u + L["P"] @ self.cycle(C["S"] @ (L["P"].T @ r), l + 1)
        for _ in range(self.nu):
            u = u + self.omega * L["Dinv"] * (b - L["S"] @ (L["A"] @ u))
        return u


@pytest.mark.parametrize("m", [5, 8, 9, 13])
@pytest.mark.parametrize("n,levels", [(4, 2), (10, 3)])
def test_cycle_around_a_vertex(m, n, levels):
    from paper_2103_11962_gb300 import rmg
    dims, gids = _fan(m, n)
    ncomp = int(gids.max()) + 1
    coef = _stencils(dims, seed=m)
    dense = _Dense([n] * m, gids, stencils_to_matrix(dims, coef, 9).toarray(), levels, 0.67, 2)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()        # noqa: E731
    ctx = rmg.Context(0)
    lay = rmg.Layout(ctx, 2, dims, dev(gids), ncomp, None)
    lay.operator_from_region_stencils(9, dev(coef.reshape(-1)))
    u = np.random.default_rng(1).standard_normal(ncomp)[gids]
    y = torch.empty(gids.size, dtype=torch.float64, device="cuda")
    lay.regional_apply(dev(u), y)
    L0 = dense.lev[0]
    assert rel_max(y.cpu().numpy(), L0["S"] @ (L0["A"] @ u)) <= 1e-13
    b = np.random.default_rng(2).standard_normal(ncomp)[gids]
    want = dense.cycle(b)
    for precision, tol in ((rmg.FP64, 1e-10), (rmg.FP32, 1e-4)):
        h = rmg.Hierarchy(lay, rmg.default_options(levels=levels, smoother=rmg.JACOBI, nu1=2, nu2=2,
                                                   omega=0.67, precision=precision))
        z = torch.empty(gids.size, dtype=torch.float64, device="cuda")
        h.vcycle(dev(b), z, regional=True)
        assert rel_max(z.cpu().numpy(), want) <= tol
