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
