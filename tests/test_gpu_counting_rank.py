"""The fused one-CTA kernel's ranking where its bins go wrong: many equal
values, values far outside the bounds of the iteration before, and values
that no comparison orders.  Whatever the state, the new iterate is a
permutation of the draws; a state of distinct values keeps the oracle's order
(test_gpu_parity.py)."""
import numpy as np
import pytest

from paper_1909_06374_gb300 import LC_FP32, Plan, workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _states(n, rng):
    spike = np.zeros(n)
    spike[n // 3] = 1e6
    return {"constant": np.full(n, 0.25), "zero": np.zeros(n), "spike": spike, "nan": np.full(n, np.nan),
            "inf": np.where(np.arange(n) == 5, np.inf, 1.0), "period_2": np.tile([1.0, 2.0], n // 2),
            "tiny": rng.standard_normal(n) * 1e-38, "normal": rng.standard_normal(n)}


@pytest.mark.parametrize("conv", [False, True])
@pytest.mark.parametrize("log2n", [10, 11, 12, 13, 14])
def test_every_state_gives_a_permutation_of_the_draws(log2n, conv, monkeypatch):
    monkeypatch.setenv("LC_PATH", "resident")
    n = 1 << log2n
    states = _states(n, np.random.default_rng(log2n))
    jobs = [workloads.job(log2n, 3, seed=40 + c, curve_id=c) for c in range(len(states))]
    with Plan(jobs, LC_FP32) as p:
        if conv:
            p.set_convergence()
        p.setup()
        s = p.buffer(2).cpu().numpy()
        x = torch.tensor(np.concatenate(list(states.values())).astype(np.float32), device="cuda")
        for iters in (1, 3):  # the bounds from a sample, then from the ranks
            p.set_state(x)
            p.iterate(iters)
            got = p.get_state().cpu().numpy()
            for c, name in enumerate(states):
                seg = slice(p.offsets[c], p.offsets[c + 1])
                assert np.array_equal(np.sort(got[seg]), s[seg]), (name, iters)
