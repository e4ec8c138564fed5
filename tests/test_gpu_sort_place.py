"""The two-step last pass of the long curves' argsort (2^26 samples on): the
new values bucketed by position, then stored.  Twice on one plan (the bucket
cursors start from zero each time), beside a shorter curve that takes the
direct pass, bit for bit against the oracle's stable argsort."""
import numpy as np
import pytest

import oracle
from paper_1909_06374_gb300 import LC_FP32, LC_FP64, Plan, workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,dt", [(LC_FP32, np.float32), (LC_FP64, np.float64)])
def test_long_argsort_by_position_buckets(prec, dt):
    rng = np.random.default_rng(8)
    jobs = [workloads.job(26, 1, seed=3, curve_id=0), workloads.job(21, 1, seed=4, curve_id=1)]
    with Plan(jobs, prec) as p:
        p.setup()
        s = p.buffer(2).cpu().numpy()
        for call in range(2 if prec == LC_FP32 else 1):
            xa = rng.standard_normal(p.total)
            xa = np.where(rng.random(p.total) < 0.5, np.round(xa * 8.0), xa).astype(dt)  # half of them ties
            got = p.rank_replace(torch.tensor(xa, device="cuda")).cpu().numpy()
            for c in range(2):
                seg = slice(p.offsets[c], p.offsets[c + 1])
                perm = oracle.argsort(xa[seg].astype(np.float64))
                want = np.empty_like(s[seg])
                want[perm] = s[seg]
                assert np.array_equal(got[seg], want), (call, c)
