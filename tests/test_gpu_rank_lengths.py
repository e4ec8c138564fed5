"""One CTA per curve (FP32 2^10..2^12, FP64 2^10..2^14) outside the fused
kernel: its lengths against the oracle's argsort, bounds carried between
iterations over tied and crowded states, and graphs of several iterations
with a remainder."""
import numpy as np
import pytest

from paper_1909_06374_gb300 import LC_FP32, LC_FP64, Plan, workloads
from tests.test_gpu_counting_rank import _states
from tests.test_gpu_rank import _check

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,log2ns", [(LC_FP32, [10, 11, 12]), (LC_FP64, [10, 11, 12, 14])])
def test_rank_replace_every_length(prec, log2ns):
    _check(prec, log2ns, seed=11)


@pytest.mark.parametrize("prec,log2ns", [(LC_FP32, [10, 12]), (LC_FP64, [10, 11, 13, 14])])
def test_every_state_gives_a_permutation_of_the_draws(prec, log2ns, monkeypatch):
    monkeypatch.setenv("LC_PATH", "multi")
    rng = np.random.default_rng(12)
    states = [(l, name, x) for l in log2ns for name, x in _states(1 << l, rng).items()]
    jobs = [workloads.job(l, 3, seed=40 + c, curve_id=c) for c, (l, _, _) in enumerate(states)]
    with Plan(jobs, prec) as p:
        p.setup()
        s = p.buffer(2).cpu().numpy()
        with np.errstate(over="ignore"):
            x = torch.tensor(np.concatenate([v for _, _, v in states])).to(p.dtype).cuda()
        for iters in (1, 3):
            p.set_state(x)
            p.iterate(iters)
            got = p.get_state().cpu().numpy()
            for c, (l, name, _) in enumerate(states):
                seg = slice(p.offsets[c], p.offsets[c + 1])
                assert np.array_equal(np.sort(got[seg]), s[seg]), (l, name, iters)


@pytest.mark.parametrize("prec,log2ns", [(LC_FP32, [10, 11, 12, 14]), (LC_FP64, [10, 11, 12, 13, 14])])
def test_sorted_draws_of_a_narrow_range(prec, log2ns):
    """Draws that are equal in float, so that every bin is crowded: sorted whole."""
    jobs = [workloads.job(l, 1, seed=60 + c, curve_id=c, log_lmin=-1.0, log_lmax=-1.0 + 1e-9, log_lbreak=-1.0 + 5e-10)
            for c, l in enumerate(log2ns)]
    with Plan(jobs, prec) as p:
        p.setup()
        x, s = p.get_state().cpu().numpy(), p.buffer(2).cpu().numpy()
        for c in range(len(jobs)):
            seg = slice(p.offsets[c], p.offsets[c + 1])
            assert np.array_equal(np.sort(x[seg]), s[seg])


@pytest.mark.parametrize("prec", [LC_FP32, LC_FP64])
@pytest.mark.parametrize("iters", [7, 8, 11, 32, 101])
def test_graphs_with_a_remainder(prec, iters):
    """One call of many iterations as many calls of one, with the convergence
    test switched on in between."""
    jobs = [workloads.job(l, iters, seed=5 + l, curve_id=l) for l in (9, 13, 14)]
    with Plan(jobs, prec) as p:
        p.setup()
        x0 = p.get_state()
        p.iterate(iters)
        whole = p.get_state()
        p.set_state(x0)
        for _ in range(iters):
            p.iterate(1)
        assert torch.equal(whole, p.get_state())
        p.set_convergence()
        for _ in range(2):
            p.set_state(x0)
            p.iterate(iters)
            assert torch.equal(whole, p.get_state())
