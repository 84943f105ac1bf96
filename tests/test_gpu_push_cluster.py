"""Push SSSP where its rounds change hands: the thread-block cluster's launches
of 128 rounds and the launched rounds it leaves a wide round or a wide search
to.  Distances are the same as those of the SpMV SSSP, bit for bit."""
import time

import numpy as np
import pytest
import torch

from tests.gpu_util import to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2201_08560_gb300 import binding
    return binding


def _csr(n, u, v):
    rows, cols = np.concatenate([u, v]), np.concatenate([v, u])
    order = np.lexsort((cols, rows))
    rows, cols = rows[order], cols[order]
    return to_dev(np.searchsorted(rows, np.arange(n + 1)).astype(np.int32)), to_dev(cols.astype(np.int32)), cols.size


def _path(n):
    return n, np.arange(n - 1), np.arange(1, n)


def _broom():
    """A path, its end joined to 60000 leaves, the leaves to a second path."""
    a, leaves = 700, np.arange(700, 60700)
    b = 60700
    u = np.concatenate([np.arange(a - 1), np.full(leaves.size, a - 1), leaves, np.arange(b, b + 700)])
    v = np.concatenate([np.arange(1, a), leaves, np.full(leaves.size, b), np.arange(b + 1, b + 701)])
    return b + 701, u, v


def _grid(rows, cols):
    i = np.arange(rows * cols).reshape(rows, cols)
    return rows * cols, np.concatenate([i[:, :-1].ravel(), i[:-1].ravel()]), np.concatenate([i[:, 1:].ravel(), i[1:].ravel()])


SHAPES = {"path": lambda: _path(1500), "broom": _broom, "grid": lambda: _grid(400, 900)}


@pytest.mark.parametrize("delta", [0.0, 7.0, 300.0])
@pytest.mark.parametrize("k", [4, 8, 16, 32])
@pytest.mark.parametrize("shape", SHAPES)
def test_same_as_spmv_sssp(B, shape, k, delta):
    n, u, v = SHAPES[shape]()
    rp, ci, nnz = _csr(n, u, v)
    rows = np.repeat(np.arange(n), np.diff(to_np(rp)))
    lo, hi = np.minimum(rows, to_np(ci)), np.maximum(rows, to_np(ci))
    w = (1.0 + ((lo * 7919 + hi * 104729) % 997) / 32.0).astype(np.float32)  # the same both ways
    assert w.size == nnz
    with B.b2sr_from_csr(n, rp, ci, k) as m:
        wb = B.b2sr_weights_from_csr(m, rp, ci, to_dev(w))
        for weights in (wb, None):
            want = to_np(B.b2sr_sssp(m, 3, weights)).view(np.int32)
            got = to_np(B.b2sr_sssp_push(m, 3, weights, delta=delta)).view(np.int32)
            np.testing.assert_array_equal(got, want)


@pytest.mark.parametrize("k", [4, 32])
def test_round_limit(B, k):
    n, u, v = _path(1000)
    rp, ci, _ = _csr(n, u, v)
    with B.b2sr_from_csr(n, rp, ci, k) as m:
        with pytest.raises(Exception, match="max_iters"):
            B.b2sr_sssp_push(m, 0, max_iters=900)
        assert to_np(B.b2sr_sssp_push(m, 0, max_iters=1024))[-1] == 999.0


def _layers(layers, width):
    """Paths side by side, all begun by the last vertex."""
    n = layers * width + 1
    i = np.arange((layers - 1) * width)
    return n, np.concatenate([i, np.full(width, n - 1)]), np.concatenate([i + width, np.arange(width)])


@pytest.mark.parametrize("shape,k", [("path", 4), ("path", 32), ("layers", 4)])
def test_last_allowed_round(B, shape, k):
    """A limit of 32 m - 1 allows 32 m rounds with work, in the cluster (the
    path) and in launched rounds (500 tile-rows a round)."""
    (n, u, v), src, rounds = (_path(1024), 0, 1024) if shape == "path" else (_layers(639, 2000), 639 * 2000, 640)
    rp, ci, _ = _csr(n, u, v)
    with B.b2sr_from_csr(n, rp, ci, k) as m:
        far = to_np(B.b2sr_sssp_push(m, src, max_iters=rounds - 1)).max()
        assert far == rounds - 1
        assert B.b2sr_sssp_push_rounds() == rounds
        with pytest.raises(Exception, match="max_iters"):
            B.b2sr_sssp_push(m, src, max_iters=rounds - 33)


def _random(n, m, seed):
    rng = np.random.default_rng(seed)
    u, v = rng.integers(0, n, (2, m))
    key = np.unique(np.minimum(u, v) * n + np.maximum(u, v))
    key = key[key // n != key % n]
    return n, key // n, key % n


def _skewed(n, m, seed):
    """A few vertices with most of the edges."""
    rng = np.random.default_rng(seed)
    u, v = (n * rng.random((2, m)) ** 4).astype(np.int64)
    key = np.unique(np.minimum(u, v) * n + np.maximum(u, v))
    key = key[key // n != key % n]
    return n, key // n, key % n


SKEWED = {"random": lambda: _random(20_001, 160_000, 1), "skewed": lambda: _skewed(30_003, 200_000, 2),
          "dense": lambda: _random(700, 60_000, 3), "star": lambda: (9000, np.zeros(8999, np.int64), np.arange(1, 9000)),
          "wide": lambda: _random(300_000, 900_000, 4)}


@pytest.mark.parametrize("delta", [0.0, 20.0])
@pytest.mark.parametrize("k", [4, 8, 16, 32])
@pytest.mark.parametrize("shape", SKEWED)
def test_irregular_graphs(B, shape, k, delta):
    """Tile-rows of none to thousands of tiles, tiles of one entry and of many,
    rounds with every row of a tile active."""
    n, u, v = SKEWED[shape]()
    rp, ci, nnz = _csr(n, u, v)
    rows = np.repeat(np.arange(n), np.diff(to_np(rp)))
    lo, hi = np.minimum(rows, to_np(ci)), np.maximum(rows, to_np(ci))
    w = (1.0 + ((lo * 7919 + hi * 104729) % 997) / 32.0).astype(np.float32)
    src = int(u[0])
    with B.b2sr_from_csr(n, rp, ci, k) as m:
        wb = B.b2sr_weights_from_csr(m, rp, ci, to_dev(w))
        for weights in (wb, None):
            want = to_np(B.b2sr_sssp(m, src, weights)).view(np.int32)
            got = to_np(B.b2sr_sssp_push(m, src, weights, delta=delta)).view(np.int32)
            np.testing.assert_array_equal(got, want)


def test_rounds_of_full_tile_rows(B):
    """A random graph of 2^15 vertices, k = 16, one entry a tile: 6.3 ms when every
    (tile, active row) pair had a lane of 16 SMs; 1.1 ms."""
    n, u, v = _random(1 << 15, 1 << 18, 5)
    rp, ci, nnz = _csr(n, u, v)
    w = torch.rand(nnz, device="cuda") * 99.0 + 1.0
    best = 1e9
    with B.b2sr_from_csr(n, rp, ci, 16) as m:
        wb = B.b2sr_weights_from_csr(m, rp, ci, w)
        for _ in range(6):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            B.b2sr_sssp_push(m, 0, wb)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
    assert best < 0.004
