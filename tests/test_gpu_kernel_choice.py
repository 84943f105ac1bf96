"""Matrices at which the SpMV's kernel changes: one tile-row holding most of the
tiles (a star, whose centre's tiles are full rows), a hub holding less, and
counts over many short rows.  Whole-number inputs: all results exact."""
import numpy as np
import pytest
import torch

from paper_2201_08560_gb300 import graphs
from tests.gpu_util import csr_dev, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2201_08560_gb300 import binding
    return binding


def _hub_and_ring(n):
    i = np.arange(n)
    return graphs.from_edges(n, np.concatenate([i, i, i]), np.concatenate([np.zeros(n, np.int64), (i + 1) % n, i * 7 % n]))


GRAPHS = {"star": lambda: graphs.star(30_011), "hub": lambda: _hub_and_ring(20_003), "ring": lambda: graphs.cycle(700_003)}


@pytest.mark.parametrize("schedule", [0, 1, 2])
@pytest.mark.parametrize("k", [4, 8, 16, 32])
@pytest.mark.parametrize("name", list(GRAPHS))
def test_all_schemes(B, name, k, schedule):
    g = GRAPHS[name]()
    n, rng = g.n, np.random.default_rng(k)
    rows, cols = np.repeat(np.arange(n), np.diff(g.rowptr)), g.colind
    xf = rng.integers(0, 16, n).astype(np.float32)
    xi = rng.permutation(n).astype(np.int32)
    xb = rng.random(n) < 0.3
    X = rng.integers(0, 2**63, n, dtype=np.int64).astype(np.uint64)
    w = rng.integers(1, 16, g.nnz).astype(np.float32)
    keep = rng.random(n) < 0.5
    mask = to_dev(graphs.pack_bits(keep))

    def fold(ufunc, ident, values, dtype):
        out = np.full(n, ident, dtype=dtype)
        ufunc.at(out, rows, values)
        return out

    plus = fold(np.add, 0, xf[cols], np.float32)
    rp, ci = csr_dev(g)
    with B.b2sr_from_csr(n, rp, ci, k) as m:
        B.b2sr_set_schedule(m, schedule)
        y = torch.full((n,), -1.0, device="cuda")
        yi = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        Y = torch.full((n,), -1, dtype=torch.int64, device="cuda")
        B.b2sr_spmv(m, B.PLUS_TIMES, B.VEC_F32, to_dev(xf), B.VEC_F32, y)
        np.testing.assert_array_equal(to_np(y), plus)
        B.b2sr_spmv(m, B.MAX_TIMES, B.VEC_F32, to_dev(xf), B.VEC_F32, y)
        np.testing.assert_array_equal(to_np(y), fold(np.maximum, -np.inf, xf[cols], np.float32))
        wb = B.b2sr_weights_from_csr(m, rp, ci, to_dev(w))
        B.b2sr_spmv(m, B.MIN_PLUS, B.VEC_F32, to_dev(xf), B.VEC_F32, y, weights=wb)
        np.testing.assert_array_equal(to_np(y), np.minimum(xf, fold(np.minimum, np.inf, xf[cols] + w, np.float32)))
        B.b2sr_spmv(m, B.MIN_PLUS, B.VEC_I32, to_dev(xi), B.VEC_I32, yi)
        np.testing.assert_array_equal(to_np(yi), np.minimum(xi, fold(np.minimum, np.iinfo(np.int32).max, xi[cols], np.int32)))
        B.b2sr_spmv(m, B.PLUS_TIMES, B.VEC_BITS, to_dev(graphs.pack_bits(xb)), B.VEC_I32, yi, mask, True)
        np.testing.assert_array_equal(to_np(yi), np.where(keep, 0, fold(np.add, 0, xb[cols].astype(np.int32), np.int32)))
        B.b2sr_spmm_bits64(m, to_dev(X), Y)
        np.testing.assert_array_equal(to_np(Y, np.uint64), fold(np.bitwise_or, 0, X[cols], np.uint64))
        X4 = rng.random((n, 4)).astype(np.float32)
        Y4 = torch.full((n, 4), -1.0, device="cuda")
        B.b2sr_spmm_f32x4(m, to_dev(X4), Y4)
        for c in range(4):
            B.b2sr_spmv(m, B.PLUS_TIMES, B.VEC_F32, to_dev(X4[:, c]), B.VEC_F32, y)
            np.testing.assert_array_equal(to_np(Y4)[:, c], to_np(y))
