"""Regions that hold a composite node more than once (closed on themselves along an axis): the
coarsest composite matrix sums every entry of a row, also those of one copy that meet in a
column."""
import itertools

import numpy as np
import pytest

from tests.gpu_common import OFFSETS

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# region sizes, axes along which the last node is the first again
@pytest.mark.parametrize("kind,dims,closed", [(5, (3, 4, 1), (0,)), (9, (2, 3, 1), (0, 1)),
                                              (7, (3, 3, 4), (1,)), (27, (3, 2, 3), (0, 1, 2))])
def test_coarse_matrix_of_a_closed_region(kind, dims, closed):
    from paper_2103_11962_gb300 import rmg
    size = [n - (a in closed) for a, n in enumerate(dims)]
    nodes = [(i, j, l) for l, j, i in itertools.product(*(range(n) for n in reversed(dims)))]
    gid = [(i % size[0]) + size[0] * ((j % size[1]) + size[1] * (l % size[2]))
           for i, j, l in nodes]
    w = np.random.default_rng(kind).uniform(0.1, 1.0, len(nodes))
    coef = np.zeros((kind, len(nodes)))
    at = {p: n for n, p in enumerate(nodes)}
    for n, p in enumerate(nodes):
        for s, d in enumerate(OFFSETS[kind]):
            q = tuple(a + b for a, b in zip(p, d))
            if q in at:
                coef[s, n] = 60.0 + w[n] if n == at[q] else -(w[n] + w[at[q]])
    ncomp = int(np.prod(size))
    want = np.zeros((ncomp, ncomp))
    for n, p in enumerate(nodes):              # the copies in order, the slots of one in order
        for s, d in enumerate(OFFSETS[kind]):
            q = tuple(a + b for a, b in zip(p, d))
            if q in at:
                want[gid[n], gid[at[q]]] += coef[s, n]
    ctx = rmg.Context(0)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    lay = rmg.Layout(ctx, 2 if dims[2] == 1 else 3, np.array([dims], dtype=np.int32),
                     dev(np.array(gid, dtype=np.int64)), ncomp, None)
    lay.operator_from_region_stencils(kind, dev(coef.reshape(-1)))
    for _ in range(3):
        h = rmg.Hierarchy(lay, rmg.default_options(levels=1))
        got, ids = h.coarse_matrix()
        assert np.array_equal(ids, np.arange(ncomp))
        assert np.array_equal(got, want)
