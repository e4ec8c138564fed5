"""Float ERDF draws where the single-precision path can go wrong, bit for bit
against the oracle: steep and nearly flat slopes, zero slopes, narrow and very
wide ranges, values at the edges of the float range, and both sides of the
table's ends."""
import numpy as np
import pytest

import oracle
from paper_1909_06374_gb300 import LC_FP32, Plan, workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = {
    "steep": dict(log_lmin=-3.0, log_lmax=2.0, log_lbreak=-0.5, slope_low=30.0, slope_high=-30.0),
    "steep_outwards": dict(log_lmin=-2.0, log_lmax=2.0, log_lbreak=0.3, slope_low=-12.0, slope_high=9.0),
    "nearly_flat": dict(slope_low=1e-5, slope_high=-1e-5),
    "zero_below": dict(slope_low=0.0),
    "zero_above_linear": dict(slope_high=-1.0, linear_space=1),
    "narrow": dict(log_lmin=-1.0001, log_lmax=-0.9999, log_lbreak=-1.0),
    "wide": dict(log_lmin=-30.0, log_lmax=30.0, log_lbreak=4.0, slope_low=0.05, slope_high=-0.04),
    "below_float_normal": dict(log_lmin=-46.0, log_lmax=-36.0, log_lbreak=-40.0),
    "above_float": dict(log_lmin=30.0, log_lmax=45.0, log_lbreak=38.0),
    "smooth": workloads.ERDF_SHAPES["smooth_eq1"],
    "smooth_steep": dict(erdf_kind=1, log_lmin=-5.0, log_lmax=5.0, log_lbreak=0.0, slope_low=-0.1, slope_high=-40.0),
    "lognormal_narrow": dict(erdf_kind=2, log_lmin=-4.0, log_lmax=1.0, log_lbreak=-1.0, sigma=5.0 / 1024),
    "lognormal_outside": dict(erdf_kind=2, log_lmin=-4.0, log_lmax=1.0, log_lbreak=4.0, sigma=0.7),
}


@pytest.mark.parametrize("log2n", [4, 11, 16])
def test_float_draws_keep_the_oracle_bits(log2n):
    jobs = [workloads.job(log2n, 0, seed=500 + c, curve_id=c, **over) for c, over in enumerate(SHAPES.values())]
    with Plan(jobs, LC_FP32) as p:
        p.setup()
        x = p.buffer(0).cpu().numpy()
    for c, (name, j) in enumerate(zip(SHAPES, jobs)):
        with np.errstate(over="ignore"):
            d = oracle.erdf_draws(oracle.job_params(j)[4:], 1 << log2n, j["seed"], j["curve_id"], prec=0,
                                  linear_space=j["linear_space"], kind=j["erdf_kind"]).astype(np.float32)
        assert np.array_equal(x[p.offsets[c]:p.offsets[c + 1]], d), name
