"""Which curves bench.py takes to be ranked by one CTA, in plans that mix them
with fused and sample-sorted ones."""
import pytest

import bench
from paper_1909_06374_gb300 import workloads


@pytest.mark.parametrize("esize,top,want", [(4, 12, 0), (4, 11, 1 << 12), (4, 9, (1 << 10) + (1 << 11) + (1 << 12)),
                                            (4, 14, 0), (8, 9, sum(1 << l for l in range(10, 15)))])
def test_rank_cta_elements(esize, top, want):
    jobs = [workloads.job(l, 5, seed=l, curve_id=l) for l in (8, 10, 11, 12, 13, 14, 15)]
    fused = sum(1 << j["log2n"] for j in jobs if esize == 4 and 10 <= j["log2n"] <= top)
    assert bench.rank_cta_elements(jobs, esize, fused) == want
