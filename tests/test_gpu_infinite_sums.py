"""Plus-times sums with infinite inputs: an infinite sum stays infinite, and
infinities of both signs give NaN, in short rows and in rows that cross many
chunks, at every k and schedule, as the plain sum gives them."""
import numpy as np
import pytest
import torch

from paper_2201_08560_gb300 import graphs
from tests.gpu_util import csr_dev, to_dev, to_np

pytestmark = pytest.mark.gpu

N = 40_000


@pytest.fixture(scope="module")
def B():
    from paper_2201_08560_gb300 import binding
    return binding


@pytest.fixture(scope="module")
def graph():
    """Rows 0 .. 3 hold every column, rows 4 .. 7 every third, the others their neighbours."""
    i = np.arange(N)
    return graphs.from_edges(N, np.concatenate([np.repeat(np.arange(4), N), np.repeat(np.arange(4, 8), len(i[::3])), i]),
                             np.concatenate([np.tile(i, 4), np.tile(i[::3], 4), (i + 1) % N]), symmetric=False,
                             drop_self_loops=False)


def _inputs():
    ones = np.ones(N, dtype=np.float32)
    some = ones.copy()
    some[12_345] = np.inf  # a column of rows 0 .. 7 (12,345 = 3 * 4,115)
    last = ones.copy()
    last[N - 1] = -np.inf
    both = some.copy()
    both[30_001] = -np.inf
    nan = ones.copy()
    nan[77] = np.nan
    return [ones, some, last, both, nan]


def _expect(g, x, weights=1.0):
    rows = np.repeat(np.arange(g.n), np.diff(g.rowptr))
    out = np.zeros(g.n, dtype=np.float64)
    with np.errstate(invalid="ignore"):
        np.add.at(out, rows, weights * x[g.colind].astype(np.float64))
    return out.astype(np.float32)  # whole numbers below 2^24, infinities, NaN: exact


@pytest.mark.parametrize("schedule", [0, 1, 2])
@pytest.mark.parametrize("k", [4, 8, 16, 32])
def test_plus_times(B, graph, k, schedule):
    xs = _inputs()
    with B.b2sr_from_csr(N, *csr_dev(graph), k) as m:
        B.b2sr_set_schedule(m, schedule)
        for x in xs:
            y = torch.full((N,), -1.0, device="cuda")
            B.b2sr_spmv(m, B.PLUS_TIMES, B.VEC_F32, to_dev(x), B.VEC_F32, y)
            np.testing.assert_array_equal(to_np(y), _expect(graph, x))
        X4 = np.stack(xs[1:], axis=1)
        Y4 = torch.full((N, 4), -1.0, device="cuda")
        B.b2sr_spmm_f32x4(m, to_dev(X4), Y4)
        for c in range(4):
            np.testing.assert_array_equal(to_np(Y4)[:, c], _expect(graph, X4[:, c]))


@pytest.mark.parametrize("k", [4, 8, 16, 32])
def test_bit_plane_weights(B, graph, k):
    rp, ci = csr_dev(graph)
    w = np.random.default_rng(k).integers(1, 8, graph.nnz)
    with B.b2sr_from_csr(N, rp, ci, k) as m:
        planes = B.b2sr_planes_from_csr(m, rp, ci, to_dev(w.astype(np.uint32)), 3)
        for x in _inputs():
            y = torch.full((N,), -1.0, device="cuda")
            B.b2sr_spmv_planes(m, planes, 3, B.VEC_F32, to_dev(x), B.VEC_F32, y)
            np.testing.assert_array_equal(to_np(y), _expect(graph, x, w))
