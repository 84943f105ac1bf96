"""B2SR -> CSR by chunks of tiles: rows that cross no, one or many chunks, empty
rows and ragged sizes give back the CSR they came from, at every tile size."""
import numpy as np
import pytest

from paper_2201_08560_gb300 import graphs
from tests.gpu_util import csr_dev, to_np

pytestmark = pytest.mark.gpu


def _graphs():
    dense = graphs.random_directed(200, 0.4, seed=2)
    gaps = graphs.disjoint_union(graphs.from_dense(np.zeros((75, 75))), graphs.complete(60),
                                 graphs.from_dense(np.zeros((500, 500))), graphs.star(1000),
                                 graphs.from_dense(np.zeros((33, 33))))
    rows = np.repeat(np.arange(3), 70_001)  # three full rows: a tile-row of 70,001 / k tiles
    wide = graphs.from_edges(70_001, rows, np.tile(np.arange(70_001), 3), symmetric=False, drop_self_loops=False)
    return {"dense": dense, "gaps": gaps, "wide": wide, "rmat": graphs.rmat(13, 16, seed=4),
            "grid": graphs.grid2d(61, 67), "one": graphs.from_dense(np.ones((1, 1))),
            "none": graphs.from_dense(np.zeros((5, 5)))}


GRAPHS = _graphs()


@pytest.mark.parametrize("k", [4, 8, 16, 32])
@pytest.mark.parametrize("name", list(GRAPHS))
def test_rows_come_back(name, k):
    from paper_2201_08560_gb300 import binding as B
    g = GRAPHS[name]
    rp, ci = csr_dev(g)
    with B.b2sr_from_csr(g.n, rp, ci, k) as m:
        rowptr, colind = B.b2sr_to_csr(m)
        np.testing.assert_array_equal(to_np(rowptr), g.rowptr)
        np.testing.assert_array_equal(to_np(colind), g.colind)
