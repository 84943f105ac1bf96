"""The small-tile SpMV kernels at the edges of their dispatch.  Value schemes at
k = 4: whole 4-value segments (aligned input, n a multiple of 4) against one
value per column (misaligned input, ragged n).  Bit schemes at k = 4 and 8: the
input bitset copied to shared memory (many chunks, a bitset that fits) against
read from global memory (few chunks, or too long a bitset), with a bitset that
is not 16-byte aligned.  Boolean, count, min, max and OR results are exact;
plus-times sums in an order that does not depend on how the input is read, so
both forms are equal bit for bit, and within 1e-5 of the fp64 oracle (the bound
derived in test_gpu_spmv.py)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2201_08560_gb300 import graphs
from tests.gpu_util import csr_dev, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2201_08560_gb300 import binding
    return binding


def _shifted(a):
    """The same vector, one element past an aligned address."""
    t = torch.empty(a.size + 1, dtype=to_dev(a[:1]).dtype, device="cuda")
    t[1:] = to_dev(a)
    return t[1:]


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 1000, 1001, 1002, 1003, 4096])
def test_value_schemes_read_any_input(B, n):
    rng = np.random.default_rng(n)
    g = graphs.random_directed(n, min(1.0, 40.0 / n), seed=n) if n < 2000 else graphs.rmat(12, 16, seed=5)
    rp, ci = csr_dev(g)
    xf, xi = rng.random(n).astype(np.float32), rng.permutation(n).astype(np.int32)
    X = rng.integers(0, 2**63, n, dtype=np.int64).astype(np.uint64)
    with B.b2sr_from_csr(n, rp, ci, 4) as m:
        B.b2sr_set_schedule(m, 2)
        plus = []
        for place in (to_dev, _shifted):
            y = torch.full((n,), float("nan"), device="cuda")
            plus.append(to_np(B.b2sr_spmv(m, B.PLUS_TIMES, B.VEC_F32, place(xf), B.VEC_F32, y)).copy())
            B.b2sr_spmv(m, B.MAX_TIMES, B.VEC_F32, place(xf), B.VEC_F32, y)
            np.testing.assert_array_equal(to_np(y), oracle.spmv_max(g, xf.astype(np.float64)).astype(np.float32))
            yi = torch.full((n,), -7, dtype=torch.int32, device="cuda")
            B.b2sr_spmv(m, B.MIN_PLUS, B.VEC_I32, place(xi), B.VEC_I32, yi)
            np.testing.assert_array_equal(to_np(yi), oracle.spmv_min_i32(g, xi))
            Y = torch.full((n,), -1, dtype=torch.int64, device="cuda")
            B.b2sr_spmm_bits64(m, place(X), Y)
            np.testing.assert_array_equal(to_np(Y, np.uint64), oracle.spmm_or64(g, X))
        ref = oracle.spmv_plus(g, xf.astype(np.float64))
        np.testing.assert_array_less(np.abs(plus[0] - ref), 1e-5 * np.abs(ref) + 1e-30)
        np.testing.assert_array_equal(plus[0], plus[1])


@pytest.mark.parametrize("k", [4, 8])
@pytest.mark.parametrize("n", [1_000_003, 1_700_001], ids=["fits", "too_long"])
def test_bit_schemes_with_many_chunks(B, k, n):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nnz = 256 * 4 * 32 * (sms + 8)  # enough chunks for the shared copy: nearly every entry has its own tile
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n + k)
    key = torch.unique(torch.randint(0, n * n, (nnz + nnz // 50,), generator=gen, device="cuda"))
    rows, cols = key // n, key % n
    rp = torch.searchsorted(key, torch.arange(n + 1, device="cuda") * n).to(torch.int32)
    bits = torch.rand(n, generator=gen, device="cuda") < 0.3
    keep = torch.rand(n, generator=gen, device="cuda") < 0.5
    x, mask = graphs.pack_bits(bits.cpu().numpy()), to_dev(graphs.pack_bits(keep.cpu().numpy()))
    want = torch.zeros(n, dtype=torch.int64, device="cuda").index_add_(0, rows, bits[cols].long())
    with B.b2sr_from_csr(n, rp, cols.to(torch.int32), k) as m:
        assert m.n_tiles >= 256 * 4 * 32 * sms
        for place in (to_dev, _shifted):
            y = torch.full((B.bitset_words(n),), -1, dtype=torch.int32, device="cuda")
            B.b2sr_spmv(m, B.BOOL_OR_AND, B.VEC_BITS, place(x), B.VEC_BITS, y, mask, True)
            got = graphs.unpack_bits(to_np(y, np.uint32), n)
            np.testing.assert_array_equal(got, ((want > 0) & ~keep).cpu().numpy())
            yc = torch.full((n,), -7, dtype=torch.int32, device="cuda")
            B.b2sr_spmv(m, B.PLUS_TIMES, B.VEC_BITS, place(x), B.VEC_I32, yc)
            np.testing.assert_array_equal(to_np(yc), want.cpu().numpy())
