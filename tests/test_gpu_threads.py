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
