"""Two host threads, each with its own stream and graph, on kernels whose
dynamic shared memory grows with the graph: neither thread's calls may change
what the other's launches are allowed."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2201_08560_gb300 import binding
    return binding


def _csr(n, u, v):
    key = torch.unique(torch.cat([u * n + v, v * n + u]))
    rowptr = torch.searchsorted(key, torch.arange(n + 1, device="cuda") * n).to(torch.int32)
    return rowptr, (key % n).to(torch.int32)


def _ring(n):
    i = torch.arange(n, device="cuda")
    return _csr(n, i, (i + 1) % n)


def _side_by_side(bodies, rounds):
    """Runs every body `rounds` times in a thread and stream of its own; the errors."""
    errors, start = [], threading.Barrier(len(bodies))

    def work(body):
        stream = torch.cuda.Stream()
        try:
            with torch.cuda.stream(stream):
                start.wait()
                for _ in range(rounds):
                    body()
                stream.synchronize()
        except Exception as e:  # noqa: BLE001 -- reported by the caller
            errors.append(e)

    threads = [threading.Thread(target=work, args=(b,)) for b in bodies]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return errors


def test_triangle_counts_of_two_sizes(B):
    """A bitmap of 1.4 M bits in two launches beside one of 96 bits."""
    mats = [B.b2sr_from_csr(n, *_ring(n), 8) for n in (1_400_000, 96)]
    counts = [torch.full((1,), -1, dtype=torch.int64, device="cuda") for _ in mats]
    torch.cuda.synchronize()
    errors = _side_by_side([lambda m=m, c=c: B.b2sr_tc(m, c) for m, c in zip(mats, counts)], 200)
    assert not errors, errors[0]
    assert [int(c.item()) for c in counts] == [0, 0]
    for m in mats:
        m.close()


def _random(n, m, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    u, v = torch.randint(0, n, (2, m), generator=gen, device="cuda")
    return _csr(n, u, v)


@pytest.mark.parametrize("k", [4, 8])
def test_boolean_and_count_spmv_of_two_sizes(B, k):
    """Inputs of 1.4 M and of 0.3 M bits, each copied to a block's shared memory."""
    sizes = [(1_400_000, 4_500_000), (300_000, 4_500_000)]
    mats = [B.b2sr_from_csr(n, *_random(n, m, 5), k) for n, m in sizes]
    bodies, got, want = [], [], []
    for m, (n, _) in zip(mats, sizes):
        x = torch.randint(-2**31, 2**31 - 1, (B.bitset_words(n),), device="cuda").to(torch.int32)
        for out, size in ((B.VEC_BITS, B.bitset_words(n)), (B.VEC_I32, n)):
            sr = B.BOOL_OR_AND if out == B.VEC_BITS else B.PLUS_TIMES
            want.append(B.b2sr_spmv(m, sr, B.VEC_BITS, x, out, torch.empty(size, dtype=torch.int32, device="cuda")))
            got.append(torch.full((size,), -1, dtype=torch.int32, device="cuda"))
            bodies.append(lambda m=m, sr=sr, x=x, out=out, y=got[-1]: B.b2sr_spmv(m, sr, B.VEC_BITS, x, out, y))
    torch.cuda.synchronize()
    errors = _side_by_side(bodies, 300)
    assert not errors, errors[0]
    for g, w in zip(got, want):
        assert torch.equal(g, w)
    for m in mats:
        m.close()


def test_batched_bfs_of_two_sizes(B):
    """Live columns of 2^20 and of 2^18 groups of four vertices."""
    sizes = [(1 << 22, 24_000_000), (1 << 20, 24_000_000)]
    mats = [B.b2sr_from_csr(n, *_random(n, m, 6), 4) for n, m in sizes]
    want = [B.b2sr_bfs_multi(m, [1, 2, 3]) for m in mats]
    got = [torch.full_like(w, -2) for w in want]
    torch.cuda.synchronize()
    errors = _side_by_side([lambda m=m, g=g: B.b2sr_bfs_multi(m, [1, 2, 3], g) for m, g in zip(mats, got)], 20)
    assert not errors, errors[0]
    for g, w in zip(got, want):
        assert torch.equal(g, w)
    for m in mats:
        m.close()
