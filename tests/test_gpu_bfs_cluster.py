"""BFS on both sides of the one-launch form's limits (tile_dim 4 and 8, at most
2^18 vertices and as many chunks of tiles as the cluster's warps hold): rows
over many blocks, long searches, isolated and unreached vertices, many
sources, ragged sizes.  Levels equal the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2201_08560_gb300 import graphs
from tests.gpu_util import csr_dev, to_np

pytestmark = pytest.mark.gpu


def _graphs():
    gaps = graphs.disjoint_union(graphs.from_dense(np.zeros((70, 70))), graphs.complete(300), graphs.path(500),
                                 graphs.from_dense(np.zeros((41, 41))))
    thin = graphs.rmat(18, 1, seed=7)
    past = graphs.CSR(thin.n + 5, np.concatenate([thin.rowptr, np.full(5, thin.nnz, np.int32)]), thin.colind)
    return {"rmat16": graphs.rmat(16, 16, seed=3), "rmat14perm": graphs.rmat(14, 32, seed=4, permute_seed=5),
            "star": graphs.star(200_001), "grid": graphs.grid2d(301, 299), "gaps": gaps,
            "one": graphs.from_dense(np.ones((1, 1))), "directed": graphs.random_directed(1501, 0.004, seed=6),
            "at_n": graphs.cycle(1 << 18), "past_n": past}


GRAPHS = _graphs()


@pytest.mark.parametrize("k", [4, 8])
@pytest.mark.parametrize("name", list(GRAPHS))
def test_levels(name, k):
    from paper_2201_08560_gb300 import binding as B
    g = GRAPHS[name]
    with B.b2sr_from_csr(g.n, *csr_dev(g), k) as m:
        for src in {0, g.n // 2, g.n - 1} if name != "at_n" else {5}:
            np.testing.assert_array_equal(to_np(B.b2sr_bfs(m, int(src))), oracle.bfs(g, int(src)))
        if g.n > 64 and name != "at_n":
            srcs = [int(v) for v in np.random.default_rng(1).choice(g.n, 9, replace=False)]
            want = np.stack([oracle.bfs(g, s) for s in srcs])
            want = np.where(want < 0, np.iinfo(np.int32).max, want).min(axis=0)
            want[want == np.iinfo(np.int32).max] = -1
            np.testing.assert_array_equal(to_np(B.b2sr_bfs_sources(m, srcs)), want)


def _row_of_blobs(n, blob, seed):
    """Random graphs of `blob` vertices, six neighbours each, in a row; ids permuted."""
    rng = np.random.default_rng(seed)
    m = n // blob
    base = np.repeat(np.arange(m) * blob, 3 * blob)
    u, v = base + rng.integers(0, blob, base.size), base + rng.integers(0, blob, base.size)
    first = np.arange(m - 1) * blob
    p = rng.permutation(n)
    return graphs.from_edges(n, p[np.concatenate([u, first])], p[np.concatenate([v, first + blob])])


@pytest.mark.parametrize("k", [4, 8])
@pytest.mark.parametrize("n,blob", [(5 << 15, 640), (3 << 16, 1024), (1 << 18, 4096)])
def test_long_searches_of_large_graphs(n, blob, k):
    """Eight to twelve chunks a warp: the rounds after the first launch's are launched
    one by one, with the same levels and the same limit."""
    from paper_2201_08560_gb300 import binding as B
    g = _row_of_blobs(n, blob, seed=n)
    want = oracle.bfs(g, 3)
    rounds = int(want.max()) + 1  # the last finds nothing
    assert rounds > 68
    with B.b2sr_from_csr(g.n, *csr_dev(g), k) as m:
        np.testing.assert_array_equal(to_np(B.b2sr_bfs(m, 3)), want)
        np.testing.assert_array_equal(to_np(B.b2sr_bfs(m, 3, max_iters=rounds - 1)), want)
        for short in (15, 16, 63, 64, rounds - 5):
            with pytest.raises(Exception, match="max_iters"):
                B.b2sr_bfs(m, 3, max_iters=short)
