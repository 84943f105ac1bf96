"""64-lane OR SpMM at k = 4 where whole chunks of 256 tiles add nothing because
every row they touch is masked out: rows inside one chunk, rows over several,
empty tile-rows between them, ragged orders, and an output that held something
else.  Exact against numpy."""
import numpy as np
import pytest
import torch

from tests.gpu_util import to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2201_08560_gb300 import binding
    return binding


@pytest.mark.parametrize("n", [4096, 4097, 4099])
@pytest.mark.parametrize("degree", [12, 40, 400])
@pytest.mark.parametrize("seed", [0, 1])
def test_masked_out_chunks(B, n, degree, seed):
    rng = np.random.default_rng(1000 * seed + degree)
    rows = np.repeat(np.arange(n), rng.poisson(degree, n))
    rows = rows[(rows // 4) % 11 != 5]  # empty tile-rows
    rows = rows[(rows < 2000) | (rows >= 2048)]
    key = np.unique(rows * n + rng.integers(0, n, rows.size))
    rows, cols = key // n, key % n
    rp = to_dev(np.searchsorted(rows, np.arange(n + 1)).astype(np.int32))
    ci = to_dev(cols.astype(np.int32))
    X = rng.integers(0, 2**63, n, dtype=np.int64).astype(np.uint64)
    full = np.uint64(2**64 - 1)
    want = np.zeros(n, np.uint64)
    np.bitwise_or.at(want, rows, X[cols])
    with B.b2sr_from_csr(n, rp, ci, 4) as m:
        B.b2sr_set_schedule(m, 2)
        for run in (1, 16, 64, 700, n):  # rows masked out one after another
            M = rng.integers(0, 2**63, n, dtype=np.int64).astype(np.uint64)
            M[(np.arange(n) // run) % 2 == seed] = full
            Y = torch.full((n,), -1, dtype=torch.int64, device="cuda")
            B.b2sr_spmm_bits64(m, to_dev(X), Y, to_dev(M), True)
            np.testing.assert_array_equal(to_np(Y, np.uint64), want & ~M)
