"""CSR -> B2SR by pieces (rows in column order without repeats, k = 4 and 8):
tile-rows shorter and longer than a window, long ones cut into slices at
columns where up to k * k entries meet, empty windows, many empty tile-rows,
ragged sizes.  The arrays equal the oracle's; a repeated entry takes the other
path and gives the same arrays."""
import time

import numpy as np
import pytest
import torch

import oracle
from paper_2201_08560_gb300 import graphs
from tests.gpu_util import csr_dev, to_np

pytestmark = pytest.mark.gpu


def _rows(n, rows, density, seed):
    """n columns; the given rows hold each column with the given density."""
    rng = np.random.default_rng(seed)
    src, dst = [], []
    for r in rows:
        c = np.flatnonzero(rng.random(n) < density)
        src.append(np.full(c.size, r))
        dst.append(c)
    return graphs.from_edges(n, np.concatenate(src), np.concatenate(dst), symmetric=False, drop_self_loops=False)


def _graphs():
    n = 30_011
    return {
        "full_rows": _rows(n, range(16, 32), 1.0, 1),           # every tile full: slices are cut between full tiles
        "half_rows": _rows(n, list(range(8)) + [12_345, n - 1], 0.5, 2),
        "one_long_row": _rows(200_003, [77], 0.9, 3),            # one run of many slices
        "window_edges": graphs.disjoint_union(*[graphs.complete(m) for m in (32, 33, 64, 129, 7)]),
        "sparse": graphs.from_edges(1_000_000, np.array([0, 5, 999_999]), np.array([999_999, 3, 0]), symmetric=False),
        "rmat": graphs.rmat(14, 16, seed=6),
        "dense": graphs.random_directed(700, 0.6, seed=7),
        "single": graphs.from_dense(np.ones((1, 1))),
    }


GRAPHS = _graphs()


@pytest.mark.parametrize("k", [4, 8])
@pytest.mark.parametrize("name", list(GRAPHS))
def test_pieces_give_the_arrays(name, k):
    from paper_2201_08560_gb300 import binding as B
    g = GRAPHS[name]
    trp, tci, tiles = oracle.b2sr(g, k)
    rep = graphs.CSR(g.n, g.rowptr.copy(), g.colind, None, "")
    rows = np.repeat(np.arange(g.n), np.diff(g.rowptr))
    at = int(g.rowptr[rows[g.nnz // 2]])  # the first entry of a row, twice
    rep.colind = np.insert(g.colind, at, g.colind[at])
    rep.rowptr[rows[at] + 1:] += 1
    for h in (g, rep):
        with B.b2sr_from_csr(h.n, *csr_dev(h), k) as m:
            got = [to_np(t) for t in B.b2sr_export(m)]
            assert m.nnz == g.nnz
        np.testing.assert_array_equal(got[0], trp)
        np.testing.assert_array_equal(got[1], tci)
        np.testing.assert_array_equal(got[2], np.ascontiguousarray(tiles).view(np.uint8).ravel())


@pytest.mark.parametrize("k", [4, 8])
@pytest.mark.parametrize("tail", [0, 1, 4095, 4096, 4097, 20000])
def test_stretches_of_empty_rows(k, tail):
    """Runs of 4,094 to 12,289 empty tile-rows before, between and after single
    entries, a short dense part and a long row."""
    from paper_2201_08560_gb300 import binding as B
    at, rows, cols = 0, [], []
    for gap in (4096, 0, 4094, 4095, 4097, 8191, 8192, 12289):
        at += gap * k
        rows += [at + k - 1]
        cols += [at // 2]
        at += k
    dense = np.arange(64)
    rows += list(np.repeat(at + dense, 64)) + [at + 100] * 1500
    cols += list(np.tile(dense, 64)) + list(range(0, 3000, 2))
    n = at + 101 + tail * k
    g = graphs.from_edges(n, np.array(rows), np.array(cols), symmetric=False)
    trp, tci, tiles = oracle.b2sr(g, k)
    with B.b2sr_from_csr(n, *csr_dev(g), k) as m:
        got = [to_np(t) for t in B.b2sr_export(m)]
    np.testing.assert_array_equal(got[0], trp)
    np.testing.assert_array_equal(got[1], tci)
    np.testing.assert_array_equal(got[2], np.ascontiguousarray(tiles).view(np.uint8).ravel())


@pytest.mark.parametrize("k", [4, 8])
def test_empty_rows_are_shared(k):
    """2^24 rows of which the first 1,000 hold entries: 37 ms when one block
    filled in the empty tile-rows' pointers; the other passes over them take
    under 1 ms."""
    from paper_2201_08560_gb300 import binding as B
    g = graphs.rmat(10, 2, seed=3)
    n = 1 << 24
    rp = np.full(n + 1, g.nnz, dtype=np.int32)
    rp[: g.n + 1] = g.rowptr
    rp, ci = torch.from_numpy(rp).cuda(), csr_dev(g)[1]
    best = 1e9
    for _ in range(6):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        B.b2sr_from_csr(n, rp, ci, k).close()
        best = min(best, time.perf_counter() - t0)
    assert best < 0.012
