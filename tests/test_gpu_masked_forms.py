"""The masked count's forms by sizes: rows found by search, rows as bitmaps in the
first launch and in one of their own, entries grouped by column with distinct
operands, and full tiles (the tile form).  Whole numbers: equal to a sparse
product."""
import time

import numpy as np
import pytest
import torch

from paper_2201_08560_gb300 import graphs
from tests.gpu_util import csr_dev

sp = pytest.importorskip("scipy.sparse")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2201_08560_gb300 import binding
    return binding


def _scipy(g):
    return sp.csr_matrix((np.ones(g.nnz, dtype=np.int64), g.colind, g.rowptr), shape=(g.n, g.n))


def _rows(n, lengths, seed):
    """Row lengths by (row, length), drawn columns."""
    rng = np.random.default_rng(seed)
    src, dst = [], []
    for row, length in lengths:
        cols = rng.choice(n, min(length, n), replace=False) if length < n else np.arange(n)
        src.append(np.full(cols.size, row))
        dst.append(cols)
    return graphs.from_edges(n, np.concatenate(src), np.concatenate(dst), symmetric=False, drop_self_loops=False)


@pytest.mark.parametrize("n", [70_001, 300_001, 1_200_007, 1_700_003])
def test_rows_of_all_lengths(B, n):
    """Rows of 3 to n columns against each other: bitmaps beside the lists, in a
    launch of their own, and none."""
    rng = np.random.default_rng(n)
    sizes = [3, 31, 32, 33, 40, 300, 511, 512, 513, 700, 5000, n // 3, n]
    a = _rows(n, [(i * 37 % 1000, s) for i, s in enumerate(sizes * 3)], 1)
    b = _rows(n, [(i * 53 % 1000, s) for i, s in enumerate(sizes[::-1] * 3)], 2)
    rows = np.array([i * 37 % 1000 for i in range(len(sizes) * 3)] + [999])
    m = graphs.from_edges(n, np.repeat(rows, 1300), np.concatenate([rng.permutation(1300) for _ in rows]),
                          symmetric=False, drop_self_loops=False)
    want = int((_scipy(a) @ _scipy(b).T).multiply(_scipy(m)).sum())
    hs = [B.b2sr_from_csr(n, *csr_dev(g), 4) for g in (a, b, m)]
    assert int(B.b2sr_spgemm_masked_count(*hs).item()) == want
    assert int(B.b2sr_spgemm_masked_count(hs[1], hs[0], hs[2]).item()) == int(
        (_scipy(b) @ _scipy(a).T).multiply(_scipy(m)).sum())
    for h in hs:
        h.close()


@pytest.mark.parametrize("k", [8, 32])
def test_distinct_operands_by_column(B, k):
    """2.2 M mask entries, rows of A shorter and longer than those of B."""
    n = 3000
    rng = np.random.default_rng(7)

    def dense(density):  # a density a row
        return rng.random((n, n)) < density[:, None]
    a, b, m = dense(rng.uniform(0.0, 0.12, n)), dense(rng.uniform(0.0, 0.3, n)), dense(np.full(n, 0.25))
    assert m.sum() >= 1 << 21
    want = int((a.astype(np.float32) @ b.T.astype(np.float32))[m].astype(np.int64).sum())
    hs = [B.b2sr_from_csr(n, *csr_dev(graphs.from_dense(x)), k) for x in (a, b, m)]
    assert int(B.b2sr_spgemm_masked_count(*hs).item()) == want
    for h in hs:
        h.close()


@pytest.mark.parametrize("k", [4, 8, 16, 32])
@pytest.mark.parametrize("cliques,size", [(300, 64), (5000, 64), (9, 500)])
def test_triangles_of_cliques(B, k, cliques, size):
    """Tiles a quarter full and more, n on both sides of 2^18."""
    i = torch.arange(cliques * size, device="cuda")
    rp = (torch.arange(cliques * size + 1, device="cuda") * (size - 1)).to(torch.int32)
    cols = (i // size * size)[:, None] + torch.arange(size, device="cuda")[None, :]
    ci = cols[cols != i[:, None]].to(torch.int32)
    with B.b2sr_from_csr(cliques * size, rp, ci, k) as m:
        assert int(B.b2sr_tc(m).item()) == cliques * size * (size - 1) * (size - 2) // 6


def test_hubs_past_the_bitmap(B):
    """A vertex joined to all of 2^21, and 2 M entries below it: 0.3 ms; the list
    form walked the hub's million columns once an entry."""
    n, hub = 1 << 21, 1 << 20
    i = torch.arange(n, device="cuda")
    leaves = i[i != hub]
    key = torch.unique(torch.cat([leaves * n + hub, hub * n + leaves]))
    rp = torch.searchsorted(key, torch.arange(n + 1, device="cuda") * n).to(torch.int32)
    best = 1e9
    with B.b2sr_from_csr(n, rp, (key % n).to(torch.int32), 4) as m:
        for _ in range(3):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            assert int(B.b2sr_tc(m).item()) == 0
            best = min(best, time.perf_counter() - t0)
    assert best < 0.05
