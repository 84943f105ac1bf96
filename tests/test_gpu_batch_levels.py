"""Batched BFS levels where a search ends in any round of a batch of four:
paths of 1 to 10 vertices and of 41, between isolated vertices, one to 64
sources with repeats, 32- and 64-lane words, a reused levels array.  The level
of a path's vertex is its distance from the source; exact."""
import numpy as np
import pytest
import torch

from tests.gpu_util import to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2201_08560_gb300 import binding
    return binding


@pytest.mark.parametrize("k", [4, 8, 32])
@pytest.mark.parametrize("nsrc", [1, 31, 32, 33, 64])
@pytest.mark.parametrize("length", [1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 41])
def test_levels_of_paths(B, length, nsrc, k):
    before, after = 37, 70 + length % 3
    n = before + length + after
    a = np.arange(before, before + length - 1)
    rows, cols = np.concatenate([a, a + 1]), np.concatenate([a + 1, a])
    order = np.lexsort((cols, rows))
    rp = to_dev(np.searchsorted(rows[order], np.arange(n + 1)).astype(np.int32))
    ci = to_dev(cols[order].astype(np.int32))
    srcs = [before - 1, before, before + length - 1, before + length // 2, n - 1, before][:nsrc]
    srcs = (srcs * 11)[:nsrc]
    at = np.arange(n)
    on_path = (at >= before) & (at < before + length)
    with B.b2sr_from_csr(n, rp, ci, k) as m:
        levels = torch.full((nsrc, n), 7777, dtype=torch.int32, device="cuda")
        for _ in range(2):
            got = to_np(B.b2sr_bfs_multi(m, srcs, levels)).reshape(nsrc, n)
            for lane, v in enumerate(srcs):
                inside = on_path if on_path[v] else at == v
                np.testing.assert_array_equal(got[lane], np.where(inside, np.abs(at - v), -1))
