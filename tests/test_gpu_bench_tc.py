"""The triangle-count figures of the benchmark: the AND-popc rate is that of the
kernel that does the AND-popcs, over its own time."""
import numpy as np
import pytest
import torch

import bench
import oracle
from paper_2201_08560_gb300 import binding as B
from paper_2201_08560_gb300 import graphs

pytestmark = pytest.mark.gpu


def test_rate_and_time_are_of_one_kernel():
    g = graphs.rmat(12, 16, seed=2)
    out = bench.tc_extra(B, torch.device("cuda", 0), (g.n, g.rowptr.astype(np.int32), g.colind.astype(np.int32)))
    assert out["triangles"] == oracle.triangle_count(g)
    r = out["roofline"]
    assert r["kernel"].startswith("masked_count_kernel")
    assert r["achieved"] * 1e12 * out["tile_form_ms"] / 1e3 == pytest.approx(r["algorithmic_ops_per_launch"])
