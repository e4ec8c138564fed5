"""A curve's bits do not depend on the plan it is in: the setup and the
transforms take other kernels and tile sizes for a few curves than for many,
for classes with PSD-target curves, and for launches over several lengths."""
import numpy as np
import pytest

from paper_1909_06374_gb300 import LC_FP32, LC_FP64, Plan, workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _jobs(log2ns, **over):
    rng = np.random.default_rng(sum(log2ns))
    return [workloads.job(l, 6, seed=70 + c, curve_id=c, f_br=float(np.exp(rng.uniform(-9.0, -3.0))),
                          alpha_high=float(rng.uniform(2.0, 3.0)), **over) for c, l in enumerate(log2ns)]


def _results(jobs, prec, c):
    """TK95 series, amplitudes, sorted draws and final state of curve c."""
    offh = sum((1 << j["log2n"]) // 2 + 1 for j in jobs[:c])
    nh = (1 << jobs[c]["log2n"]) // 2 + 1
    with Plan(jobs, prec) as p:
        seg = slice(p.offsets[c], p.offsets[c + 1])
        tk = p.empty()
        x = p.generate(out_tk=tk)
        return [v.cpu().numpy() for v in (tk[seg], p.buffer(1)[offh:offh + nh], p.buffer(2)[seg], x[seg])]


def _same(jobs, prec, curves):
    for c in curves:
        for got, want, what in zip(_results(jobs, prec, c), _results([jobs[c]], prec, 0), ("tk", "A", "s", "x")):
            assert np.array_equal(got, want), (what, c)


@pytest.mark.parametrize("prec", [LC_FP32, LC_FP64])
@pytest.mark.parametrize("log2n,curves", [(4, 400), (10, 700), (13, 400), (16, 60), (19, 8)])
def test_alone_as_among_many(log2n, curves, prec):
    _same(_jobs([log2n] * curves), prec, (0, curves - 1))


@pytest.mark.parametrize("prec", [LC_FP32, LC_FP64])
@pytest.mark.parametrize("log2n", [11, 14, 17])
def test_beside_a_psd_target_curve(log2n, prec):
    jobs = _jobs([log2n] * 3)
    jobs[1]["tk_targets"] = 1
    jobs[2]["tk_coeffs"] = 1
    _same(jobs, prec, (0, 2))


@pytest.mark.parametrize("prec", [LC_FP32, LC_FP64])
def test_alone_as_among_other_lengths(prec):
    _same(_jobs([13, 14, 15, 16, 17, 18, 20, 21]), prec, range(8))
