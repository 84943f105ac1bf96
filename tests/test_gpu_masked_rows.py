"""The masked count over row lists: rows shorter and longer than the list form
takes (32 columns), runs of mask entries inside one row and over many, distinct
asymmetric operands, a matrix too long for the bitmap, and a mask of few tiles
(the tile form).  Whole numbers: equal to the dense product or a closed form."""
import numpy as np
import pytest
import torch

from paper_2201_08560_gb300 import graphs
from tests.gpu_util import csr_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2201_08560_gb300 import binding
    return binding


@pytest.mark.parametrize("k", [4, 8, 16, 32])
@pytest.mark.parametrize("density", [0.01, 0.08, 0.5])
def test_distinct_operands(B, k, density):
    n = 401
    gs = [graphs.random_directed(n, d, seed=i + k) for i, d in enumerate((density, 0.3, 0.1))]
    a, b, m = (graphs.to_dense(g) for g in gs)
    hs = [B.b2sr_from_csr(n, *csr_dev(g), k) for g in gs]
    assert int(B.b2sr_spgemm_masked_count(*hs).item()) == int(((a @ b.T) * m).sum())
    count, pairs = B.b2sr_spgemm_masked_count_work(*hs)  # the tile form
    assert int(count.item()) == int(((a @ b.T) * m).sum())
    for h in hs:
        h.close()


@pytest.mark.parametrize("n", [70_001, 1_700_003], ids=["bitmap", "lists"])
def test_long_rows(B, n):
    """Rows 0 .. 2 hold every column and the mask has rows 0 .. 2 by columns
    0 .. 2: nine entries of n common columns each.  A second mask adds single
    entries (i, 0) of rows with one column."""
    full = np.arange(n)
    diag = np.arange(3, n, 997)
    g = graphs.from_edges(n, np.concatenate([np.repeat(np.arange(3), n), diag]),
                          np.concatenate([np.tile(full, 3), diag]), symmetric=False, drop_self_loops=False)
    rows3 = np.repeat(np.arange(3), 3)
    mask = graphs.from_edges(n, np.concatenate([rows3, diag]), np.concatenate([np.tile(np.arange(3), 3), 0 * diag]),
                             symmetric=False, drop_self_loops=False)
    h, hm = B.b2sr_from_csr(n, *csr_dev(g), 4), B.b2sr_from_csr(n, *csr_dev(mask), 4)
    want = 9 * n + diag.size
    assert int(B.b2sr_spgemm_masked_count(h, h, hm).item()) == want
    # the whole matrix as its own mask: row i < 3 against row j is full with 3 rows and one column with the others
    own = 9 * n + 3 * diag.size + diag.size
    assert int(B.b2sr_spgemm_masked_count(h, h, h).item()) == own
    h.close()
    hm.close()


def test_triangles_of_a_complete_graph(B):
    g = graphs.complete(700)
    with B.b2sr_from_csr(g.n, *csr_dev(g), 8) as m:
        assert int(B.b2sr_tc(m).item()) == 700 * 699 * 698 // 6
        torch.cuda.synchronize()
