"""Structure function and periodogram of FP32 plans over the range of float:
large and infinite samples, bin powers at both ends, and the batches whose
blocks take all lags of a curve."""
import numpy as np
import pytest

import oracle
from paper_1909_06374_gb300 import LC_FP32, Plan, workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# a run of 64 float squares: a difference (2^-24), its square and 63 additions (64 x 2^-24)
SF_TOL = 66 * 2.0 ** -24


def _plan(log2n, curves=1):
    return Plan([workloads.job(log2n, 0, seed=1 + c, curve_id=c) for c in range(curves)], LC_FP32)


@pytest.mark.parametrize("log2n", [8, 12, 14, 16])
@pytest.mark.parametrize("scale", [1e-17, 1e16, 2e17, 5e17, "spread"])
def test_structure_function_stays_finite(log2n, scale):
    """A lag's squares add up to more than the largest float, no run of 64 does
    (2e17, 5e17); runs far apart in size (spread)."""
    n = 1 << log2n
    rng = np.random.default_rng(log2n)
    x = rng.standard_normal(n) * (10.0 ** rng.uniform(-16, 16, n) if scale == "spread" else scale)
    x = x.astype(np.float32)
    lags = [1, 3, n // 4, n - 1]
    with _plan(log2n) as p:
        got = p.structure_function(torch.tensor(x, device="cuda"), lags).cpu().numpy()[0]
    np.testing.assert_allclose(got, oracle.structure_function(x.astype(np.float64), lags), rtol=SF_TOL)


@pytest.mark.parametrize("log2n", [8, 14, 16])
def test_structure_function_of_infinite_samples(log2n):
    """A lag is infinite where a pair holds the infinite sample, NaN where a
    pair holds two of them, and the other curves of the batch keep theirs."""
    n = 1 << log2n
    x = np.random.default_rng(3).standard_normal((4, n)).astype(np.float32)
    x[1, n // 2] = np.inf
    x[2, [0, 5]] = -np.inf
    lags = [1, 5, n // 2 + 1, n - 1]
    with _plan(log2n, 4) as p:
        got = p.structure_function(torch.tensor(x.reshape(-1), device="cuda"), lags).cpu().numpy()
    with np.errstate(invalid="ignore"):
        want = np.array([[np.mean((xc[:-l] - xc[l:]) ** 2) for l in lags] for xc in x.astype(np.float64)])
    assert np.isinf(want).any() and np.isnan(want).any()
    np.testing.assert_allclose(got, want, rtol=SF_TOL)


@pytest.mark.parametrize("curves,log2n,nlags", [(1, 11, 3), (1, 12, 40), (640, 11, 50), (640, 12, 33), (640, 14, 17),
                                                (160, 16, 50), (1, 20, 20), (10, 20, 40)])
def test_structure_function_by_blocks_of_many_lags(curves, log2n, nlags):
    n = 1 << log2n
    rng = np.random.default_rng(nlags)
    x = rng.standard_normal((curves, n)).astype(np.float32)
    lags = np.unique(np.append(np.geomspace(1, n - 1, nlags).astype(np.int64), [n // 2 - 1, n // 2, n // 2 + 1]))
    with _plan(log2n, curves) as p:
        got = p.structure_function(torch.tensor(x.reshape(-1), device="cuda"), [int(l) for l in lags]).cpu().numpy()
    for c in {0, curves // 2, curves - 1}:
        np.testing.assert_allclose(got[c], oracle.structure_function(x[c].astype(np.float64), lags), rtol=SF_TOL)


def test_bin_powers_keep_their_precision():
    """x = (a, b, 0, 0, ...) has X_{N/4} = a - i b exactly (the transform's two
    additions are of zeros), so that bin's power is (a^2 + b^2) 2 / N^2 to the
    rounding of one FP64 addition."""
    rng = np.random.default_rng(5)
    ab = (rng.standard_normal((400, 2)) * 10.0 ** rng.uniform(-30, 30, (400, 1))).astype(np.float32)
    ab = np.concatenate([ab, np.float32([[2.0 ** -46, 0], [0, 2.0 ** -46], [1, 0], [0, 0], [3, 4], [1e-40, 1e-42],
                                         [2.0 ** -43, 2.0 ** -62], [1, 2.0 ** -12], [1, np.nan]])])
    n = 16
    x = np.zeros((len(ab), n), dtype=np.float32)
    x[:, :2] = ab
    with _plan(4, len(ab)) as p:
        P = p.periodogram(torch.tensor(x.reshape(-1), device="cuda")).cpu().numpy().reshape(len(ab), n // 2 + 1)
    a, b = ab.astype(np.float64).T
    np.testing.assert_allclose(P[:, n // 4], (a * a + b * b) * (2.0 / n ** 2), rtol=2.0 ** -52)
