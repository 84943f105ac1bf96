"""The row-lane SpMV kernel (value schemes at k = 8, 16 and 32) where tile-rows
end anywhere in a step, a group or a segment: every tile-row length from none to
40 tiles in a mixed order, one tile-row over several chunks, full and one-bit
tiles, a ragged order, with and without a mask and weights.  Every input is a
whole number small enough that fp32 sums are exact, so all results are exact;
the four-column product is checked column by column against the single-column
one on fractions too, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2201_08560_gb300 import graphs
from tests.gpu_util import to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2201_08560_gb300 import binding
    return binding


def _matrix(k, ragged):
    """Rows, columns: tile-row R holds (R * 17) % 41 tiles, tile-row 3 holds 700."""
    rng = np.random.default_rng(k + ragged)
    ntr = 720
    n = ntr * k - ragged
    keys = []
    for R in range(ntr):
        tiles = 700 if R == 3 else (R * 17) % 41
        for J in rng.choice(ntr, tiles, replace=False):
            bits = k * k if rng.random() < 0.01 else rng.choice([1, 1, 1, 2, k])
            at = rng.choice(k * k, bits, replace=False)
            keys.append((R * k + at // k) * (ntr * k) + J * k + at % k)
    key = np.unique(np.concatenate(keys))
    rows, cols = key // (ntr * k), key % (ntr * k)
    keep = (rows < n) & (cols < n)
    return n, rows[keep], cols[keep]


@pytest.mark.parametrize("ragged", [0, 3, 7])
@pytest.mark.parametrize("k", [8, 16, 32])
def test_row_ends_anywhere(B, k, ragged):
    n, rows, cols = _matrix(k, ragged)
    rng = np.random.default_rng(100 * k + ragged)
    rp = to_dev(np.searchsorted(rows, np.arange(n + 1)).astype(np.int32))
    ci = to_dev(cols.astype(np.int32))
    xi = rng.permutation(n).astype(np.int32)
    xf = rng.integers(0, 64, n).astype(np.float32)
    w = rng.integers(1, 16, rows.size).astype(np.float32)
    X = rng.integers(0, 2**63, n, dtype=np.int64).astype(np.uint64)
    X4 = rng.random((n, 4)).astype(np.float32)
    keep = rng.random(n) < 0.5
    mask = to_dev(graphs.pack_bits(keep))

    def reduce_rows(ufunc, ident, values, dtype):
        out = np.full(n, ident, dtype=dtype)
        ufunc.at(out, rows, values)
        return out

    plus = reduce_rows(np.add, 0, xf[cols], np.float32)
    xinf = np.where(rng.random(n) < 0.05, np.float32(np.inf), xf)
    plus_inf = reduce_rows(np.add, 0, xinf[cols], np.float32)
    low = np.minimum(reduce_rows(np.minimum, np.iinfo(np.int32).max, xi[cols], np.int32), xi)
    far = np.minimum(reduce_rows(np.minimum, np.inf, xf[cols] + w, np.float32), xf)
    near = np.minimum(reduce_rows(np.minimum, np.inf, xf[cols] + np.float32(1), np.float32), xf)
    ors = reduce_rows(np.bitwise_or, 0, X[cols], np.uint64)
    with B.b2sr_from_csr(n, rp, ci, k) as m:
        wb = B.b2sr_weights_from_csr(m, rp, ci, to_dev(w))
        for schedule in (0, 2):
            B.b2sr_set_schedule(m, schedule)
            y = torch.full((n,), float("nan"), device="cuda")
            B.b2sr_spmv(m, B.PLUS_TIMES, B.VEC_F32, to_dev(xf), B.VEC_F32, y)
            np.testing.assert_array_equal(to_np(y), plus)
            B.b2sr_spmv(m, B.PLUS_TIMES, B.VEC_F32, to_dev(xf), B.VEC_F32, y, mask, True)
            np.testing.assert_array_equal(to_np(y), np.where(keep, 0, plus))
            B.b2sr_spmv(m, B.PLUS_TIMES, B.VEC_F32, to_dev(xinf), B.VEC_F32, y)
            np.testing.assert_array_equal(to_np(y)[: 3 * k], plus_inf[: 3 * k])  # tile-rows inside one chunk
            B.b2sr_spmv(m, B.MIN_PLUS, B.VEC_F32, to_dev(xf), B.VEC_F32, y, weights=wb)
            np.testing.assert_array_equal(to_np(y), far)
            B.b2sr_spmv(m, B.MIN_PLUS, B.VEC_F32, to_dev(xf), B.VEC_F32, y)
            np.testing.assert_array_equal(to_np(y), near)
            yi = torch.full((n,), -7, dtype=torch.int32, device="cuda")
            B.b2sr_spmv(m, B.MIN_PLUS, B.VEC_I32, to_dev(xi), B.VEC_I32, yi)
            np.testing.assert_array_equal(to_np(yi), low)
            Y = torch.full((n,), -1, dtype=torch.int64, device="cuda")
            B.b2sr_spmm_bits64(m, to_dev(X), Y)
            np.testing.assert_array_equal(to_np(Y, np.uint64), ors)
            Y4 = torch.full((n, 4), float("nan"), device="cuda")
            B.b2sr_spmm_f32x4(m, to_dev(X4), Y4)
            for c in range(4):
                B.b2sr_spmv(m, B.PLUS_TIMES, B.VEC_F32, to_dev(X4[:, c]), B.VEC_F32, y)
                np.testing.assert_array_equal(to_np(Y4)[:, c], to_np(y))
