"""B2SR to CSR where the kernels change: tiles of one entry and full ones, rows
that end anywhere in a chunk and cross several, a chunk whose tile-rows are
mostly empty, ragged sizes, at every k.  The arrays equal the ones the matrix
was built from."""
import time

import numpy as np
import pytest
import torch

from paper_2201_08560_gb300 import graphs
from tests.gpu_util import csr_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2201_08560_gb300 import binding
    return binding


def _band(n, half):
    i = np.repeat(np.arange(n), 2 * half + 1)
    j = i + np.tile(np.arange(-half, half + 1), n)
    ok = (j >= 0) & (j < n)
    return graphs.from_edges(n, i[ok], j[ok], symmetric=False, drop_self_loops=False)


def _hubs(n):
    """Rows 5 and 70 hold every column, row n - 1 every second; column 3 in every row."""
    i = np.arange(n)
    src = np.concatenate([np.full(n, 5), np.full(n, 70), np.full(len(i[::2]), n - 1), i])
    return graphs.from_edges(n, src, np.concatenate([i, i, i[::2], np.full(n, 3)]), symmetric=False,
                             drop_self_loops=False)


def _scattered():
    """Entries 1,023 to 70,000 tile-rows of 4 apart, a short dense part, an empty tail."""
    at = np.cumsum([1023 * 4, 1024 * 4, 1025 * 4, 280_000, 3, 40_000, 120_001])
    dense = np.arange(40)
    return graphs.from_edges(at[-1] + 200_000, np.concatenate([at, at[2] + np.repeat(dense, 40)]),
                             np.concatenate([at // 3, np.tile(dense, 40)]), symmetric=False)


GRAPHS = {"band1": lambda: _band(5003, 1), "band40": lambda: _band(3001, 40), "full": lambda: graphs.complete(517),
          "hubs": lambda: _hubs(20_011), "scattered": _scattered, "rmat": lambda: graphs.rmat(13, 16, seed=4),
          "one_a_tile": lambda: graphs.random_directed(4099, 0.002, seed=3)}


@pytest.mark.parametrize("k", [4, 8, 16, 32])
@pytest.mark.parametrize("name", list(GRAPHS))
def test_arrays_come_back(B, name, k):
    g = GRAPHS[name]()
    with B.b2sr_from_csr(g.n, *csr_dev(g), k) as m:
        rp, ci = B.b2sr_to_csr(m)
    np.testing.assert_array_equal(to_np(rp), g.rowptr)
    np.testing.assert_array_equal(to_np(ci), g.colind)


@pytest.mark.parametrize("k", [4, 8, 16, 32])
def test_empty_rows_cost_little(B, k):
    """1,000 edges over 2^24 rows: 11 ms at k = 4 when a warp went through a
    chunk's empty tile-rows 31 at a time; a pass over the row pointers takes
    under 0.1 ms."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    n = 1 << 24
    key = torch.unique(torch.randint(0, n * n, (2000,), generator=gen, device="cuda"))
    rp = torch.searchsorted(key, torch.arange(n + 1, device="cuda") * n).to(torch.int32)
    ci = (key % n).to(torch.int32)
    best = 1e9
    with B.b2sr_from_csr(n, rp, ci, k) as m:
        for _ in range(6):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            got = B.b2sr_to_csr(m)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
    assert torch.equal(got[0], rp) and torch.equal(got[1], ci)
    assert best < 0.004
