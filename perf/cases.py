"""Performance cases of the light-curve generator: the calls that its users make.

A case is a dict of plain values: ``kind`` says which public entry point runs,
``curves`` x 2^``log2n`` samples (``log2n`` .. ``log2n_hi`` for ragged batches)
say how much, ``prec`` is the sample type.  Kinds:

  generate     Plan.generate: the whole generator (TK95, ERDF draws, ``iters``
               amplitude-adjustment iterations), the result left on the device;
  host         lc_generate_host: the same with the result copied to pinned host
               memory inside the call;
  converge     Plan.generate with the Eq. 4 convergence test on, then the
               record of the run that says where each curve stopped;
  iterate      Plan.set_state, Plan.iterate(``iters``), Plan.get_state: the
               iterations alone, from the draws in draw order;
  setup        Plan.setup with the TK95 series asked for: realisation, target
               amplitudes, draws and their sort;
  periodogram  Plan.periodogram of a generated batch;
  structure    Plan.structure_function of a generated batch at ``lags`` lags.

Curve parameters follow the repository's workloads: ``base`` is the uniform
batch's PSD and ERDF, ``varied`` the per-curve PSD and ERDF of the ragged
batch, ``shapes`` the varied PSD with the paper's smooth and log-normal ERDFs
and the sharp form in turn.
"""
import math

import numpy as np
import torch

from paper_1909_06374_gb300 import LC_FP32, LC_FP64, Plan, lc_generate_host, workloads

DEV = "cuda:0"
LN10 = math.log(10.0)


def _case(name, kind, curves, log2n, iters=0, prec="fp32", hi=None, params="base", lags=0, rms=False, threshold=0.0):
    c = dict(kind=kind, curves=curves, log2n=log2n, log2n_hi=log2n if hi is None else hi, iters=iters, prec=prec,
             params=params, lags=lags, rms=rms, threshold=threshold)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one short curve, as an interactive user asks for it: latency of the
        # setup launches and of the on-chip iterations
        _case("one_2p10", "generate", 1, 10, 100),
        # one curve from the middle of the serving range: a chain of short kernels
        _case("one_2p17", "generate", 1, 17, 100, params="varied"),
        # the repository's single-curve workload, in double precision
        _case("single_fp64_2p14", "generate", 1, 14, 100, prec="fp64"),
        # a large ensemble of short curves
        _case("batch_4096x2p12", "generate", 4096, 12, 100),
        # the benchmark's batch: its iterations, which are nearly all of its time
        _case("uniform_4096x2p16", "iterate", 4096, 16, 8),
        # the benchmark's curves, whole call with all iterations and the copy to the host
        _case("host_512x2p16", "host", 512, 16, 200),
        # curves of uneven length with their own PSD and ERDF
        _case("ragged_1000_2p10_2p20", "generate", 1000, 10, 20, hi=20, params="varied"),
        # survey-length curves: far above any cache
        _case("long_4x2p26", "iterate", 4, 26, 3, params="varied"),
        # the paper's ERDF shapes with the TK95 series returned: setup alone
        _case("setup_1021x2p16", "setup", 1021, 16, params="shapes"),
        # an ensemble that stops curve by curve once it has converged
        _case("converge_1000x2p15", "converge", 1000, 15, 100, params="varied", threshold=4e-3),
        # ensemble checks of Sec. 3.2.5: periodograms and structure functions
        _case("periodogram_2048x2p16", "periodogram", 2048, 16, params="base"),
        _case("structure_256x2p16", "structure", 256, 16, lags=58),
    ]


#: Most samples of a drawn batch, and most sample-iterations by sample type
#: (the listed cases' largest are 2^28 and 6.7e9).
MAX_SAMPLES = 1 << 27
MAX_WORK = {"fp32": 2.5e9, "fp64": 2.5e8}


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["generate", "generate", "generate", "iterate", "iterate", "host", "converge", "setup",
                       "periodogram", "structure"])
    prec = "fp64" if rng.random() < 0.2 else "fp32"
    params = rng.choice(["base", "varied", "shapes"])
    log2n = rng.randint(10, 24 if kind in ("iterate", "generate") else 20)
    hi = min(log2n + rng.randint(1, 8), 20) if log2n < 19 and rng.random() < 0.3 else log2n
    most = MAX_SAMPLES >> (2 if kind in ("structure", "setup") or prec == "fp64" else 0)
    mean = sum(1 << k for k in range(log2n, hi + 1)) // (hi - log2n + 1)
    curves = min(_logint(rng, 1, max(1, most // mean)), 4096)
    if curves > 2:
        curves |= 1
    samples = curves * mean
    iters = max(1, min(_logint(rng, 3, 200), int(MAX_WORK[prec] // samples)))
    if kind == "iterate":
        iters = min(iters, 12)
    if kind in ("setup", "periodogram", "structure"):
        iters = 0
    lags = 0
    if kind == "structure":
        lags = max(1, min(_logint(rng, 5, 400), int(1.2e9 // samples)))
    thr = 10.0 ** rng.uniform(-3.0, -2.0) if kind == "converge" else 0.0
    return _case(None, kind, curves, log2n, iters, prec=prec, hi=hi, params=params, lags=lags,
                 rms=kind == "periodogram" and rng.random() < 0.5, threshold=thr)


# ------------------------------------------------------------------ inputs
def _jobs(case, seed):
    rng = np.random.default_rng([seed, 17])
    shapes = ["smooth_eq1", "lognormal", None, "table2"]
    base_id = int(rng.integers(0, 1 << 40))
    # a batch's lengths are the case's own; its parameters and random streams the seed's
    lengths = np.random.default_rng([case["curves"], case["log2n"]]).integers(case["log2n"], case["log2n_hi"] + 1,
                                                                              case["curves"])
    jobs = []
    for c in range(case["curves"]):
        over = {}
        if case["params"] != "base":
            over = dict(f_br=float(np.exp(rng.uniform(np.log(1e-4), np.log(1e-1)))),
                        alpha_high=float(rng.uniform(2.0, 3.0)),
                        log_lbreak=float(rng.uniform(-2.5, -0.5)), slope_high=float(rng.uniform(-3.0, -1.5)))
        if case["params"] == "shapes" and shapes[c % 4]:
            over.update(workloads.ERDF_SHAPES[shapes[c % 4]])
        jobs.append(workloads.job(int(lengths[c]), case["iters"], seed=base_id + c, curve_id=c, **over))
    return jobs


def _lags(case, nmin):
    """Distinct lags spread over the logarithm of [1, nmin/2], as an ensemble check takes them."""
    want = np.unique(np.round(np.geomspace(1, nmin // 2, case["lags"])).astype(np.int64))
    return [int(v) for v in want]


def prepare(case, seed):
    jobs = _jobs(case, seed)
    prec = LC_FP32 if case["prec"] == "fp32" else LC_FP64
    p = Plan(jobs, prec, device=0)
    st = {"case": case, "plan": p}
    kind = case["kind"]
    if kind == "host":
        st["host"] = torch.empty(p.total, dtype=p.dtype, pin_memory=True)
    elif kind == "converge":
        p.set_convergence([case["threshold"]] * len(jobs))
    elif kind == "iterate":
        p.setup()
        st["x0"] = p.get_state()
    elif kind in ("periodogram", "structure"):
        # the series that Sec. 3.2.5 checks: a generated batch after a few iterations
        p.setup()
        p.iterate(2)
        st["x"] = p.get_state()
        if kind == "structure":
            st["lags"] = _lags(case, 1 << min(j["log2n"] for j in jobs))
    return st


def run(state):
    p, kind = state["plan"], state["case"]["kind"]
    if kind == "generate":
        return p.generate()
    if kind == "host":
        lc_generate_host(p.handle, state["host"], None, torch.cuda.current_stream(0))
        return state["host"]
    if kind == "converge":
        x = p.generate()
        deltas, iters_run = p.convergence()
        return [x, deltas, iters_run]
    if kind == "iterate":
        p.set_state(state["x0"])
        p.iterate(state["case"]["iters"])
        return p.get_state()
    if kind == "setup":
        tk = p.empty()
        p.setup(out_tk=tk)
        return [tk, p.get_state()]
    if kind == "periodogram":
        return p.periodogram(state["x"], rms=state["case"]["rms"])
    return p.structure_function(state["x"], state["lags"])


def work(case):
    """Bytes: the state or series read once where the call takes one, with the
    targets and draws it is matched to, and the results written once.  Flops:
    two real transforms of 2.5 N log2 N per iteration, and what the estimators
    sum."""
    es = 4 if case["prec"] == "fp32" else 8
    ks = range(case["log2n"], case["log2n_hi"] + 1)
    share = case["curves"] / len(ks)
    n = share * sum(1 << k for k in ks)
    fft = share * sum(2.5 * k * (1 << k) for k in ks)
    kind, it = case["kind"], case["iters"]
    if kind in ("generate", "host", "converge"):
        return {"bytes": es * n, "flops": 2 * fft * it}
    if kind == "iterate":
        return {"bytes": 3.5 * es * n, "flops": 2 * fft * it}
    if kind == "setup":
        return {"bytes": 2 * es * n, "flops": fft}
    if kind == "periodogram":
        return {"bytes": (es + 4) * n, "flops": fft}
    pairs = case["curves"] * sum((1 << case["log2n"]) - l for l in _lags(case, 1 << case["log2n"]))
    return {"bytes": es * n, "flops": 3.0 * pairs}


# ------------------------------------------------------------ 64-bit results
def _mulhilo(a, b):
    """High and low 32 bits of a * b (a a Python int, b an int64 tensor below 2^32)."""
    a0, a1 = a & 0xFFFF, a >> 16
    b0, b1 = b & 0xFFFF, b >> 16
    m = a1 * b0 + ((a0 * b0) >> 16)
    k = a0 * b1 + (m & 0xFFFF)
    return a1 * b1 + (m >> 16) + (k >> 16), ((k & 0xFFFF) << 16) | ((a0 * b0) & 0xFFFF)


def _uniforms(idx, curve_id, tag, seed):
    """Two uniforms per Philox4x32-10 block: (2u + 1) 2^-53 with u the top 52 bits of a word pair."""
    c0, c1 = idx & 0xFFFFFFFF, idx >> 32
    c2, c3 = torch.full_like(idx, curve_id & 0xFFFFFFFF), torch.full_like(idx, tag)
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        hi_a, lo_a = _mulhilo(0xD2511F53, c0)
        hi_b, lo_b = _mulhilo(0xCD9E8D57, c2)
        c0, c1, c2, c3 = hi_b ^ c1 ^ k0, lo_b, hi_a ^ c3 ^ k1, lo_a
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return [(2 * ((w1 << 20) | (w0 >> 12)) + 1).double() * 2.0 ** -53 for w0, w1 in ((c0, c1), (c2, c3))]


def _spectrum(j):
    """TK95 spectrum X_0..X_{N/2} over its standard deviation (C2R of it has unit variance)."""
    n = 1 << j["log2n"]
    k = torch.arange(1, n // 2 + 1, device=DEV)
    u1, u2 = _uniforms(k, j["curve_id"], 0, j["seed"])
    y = k.double() / (n * j["dt"] * j["f_br"])
    pw = 1.0 / (y ** j["alpha_low"] + y ** j["alpha_high"])
    rad = torch.sqrt(-torch.log(u1) * pw)
    X = torch.zeros(n // 2 + 1, dtype=torch.complex128, device=DEV)
    X[1:] = torch.complex(rad * torch.cos(2 * math.pi * u2), rad * torch.sin(2 * math.pi * u2))
    X[-1] = math.sqrt(2.0) * X[-1].real
    var = 2.0 * (X[1:-1].abs() ** 2).sum() + X[-1].abs() ** 2
    return X / torch.sqrt(var)


def _density(j, u):
    d = u - j["log_lbreak"]
    if j["erdf_kind"] == 1:
        return 1.0 / (np.exp(-j["slope_low"] * LN10 * d) + np.exp(-j["slope_high"] * LN10 * d))
    return np.exp(-0.5 * (d / j["sigma"]) ** 2)


def _draws(j):
    """ERDF draws in draw order: the inverse CDF in closed form (sharp break) or
    through the 4096-interval Simpson table with linear interpolation."""
    n = 1 << j["log2n"]
    U = torch.stack(_uniforms(torch.arange(n // 2, device=DEV), j["curve_id"], 1, j["seed"]), 1).reshape(-1)
    lo, hi, ub = j["log_lmin"], j["log_lmax"], j["log_lbreak"]
    if j["erdf_kind"] == 0:
        c1, c2 = j["slope_low"] * LN10, j["slope_high"] * LN10
        m1 = (1.0 - math.exp(c1 * (lo - ub))) / c1
        m2 = (math.exp(c2 * (hi - ub)) - 1.0) / c2
        v = U * (m1 + m2)
        below = torch.log(math.exp(c1 * (lo - ub)) + c1 * torch.clamp(v, max=m1)) / c1
        above = torch.log1p(c2 * torch.clamp(v - m1, min=0.0)) / c2
        u = ub + torch.where(v < m1, below, above)
    else:
        K = 4096
        h = (hi - lo) / K
        g = lo + h * np.arange(K + 1)
        F = np.concatenate([[0.0], np.cumsum((_density(j, g[:-1]) + 4.0 * _density(j, g[:-1] + 0.5 * h) +
                                              _density(j, g[1:])) * h / 6.0)])
        F = torch.tensor(F, device=DEV)
        v = U * F[-1]
        a = torch.clamp(torch.searchsorted(F, v, right=True) - 1, 0, K - 1)
        u = lo + a * h + (v - F[a]) / (F[a + 1] - F[a]) * h
    return torch.exp(LN10 * u)


def _iterate(x, A, iters, threshold=None):
    """Amplitude adjustment in 64 bits; with a threshold also Eq. 4's record."""
    s, n = torch.sort(x)[0], x.numel()
    deltas = []
    for _ in range(iters):
        X = torch.fft.rfft(x)
        m = X.abs()
        Y = torch.where(m > 0, X / torch.where(m > 0, m, 1.0), 1.0 + 0j) * A
        Y[-1] = torch.where(X[-1].real < 0, -A[-1], A[-1]) + 0j
        Y[0] = A[0] + 0j
        order = torch.sort(torch.fft.irfft(Y, n=n), stable=True)[1]
        new = torch.empty_like(x)
        new[order] = s
        if threshold is not None:
            deltas.append(float(torch.sqrt(torch.mean(torch.log10(new / x) ** 2))))
        x = new
        if threshold is not None and deltas[-1] < threshold:
            break
    return x, deltas


def exact(case, seed):
    kind = case["kind"]
    total = case["curves"] * sum(1 << k for k in range(case["log2n"], case["log2n_hi"] + 1)) / \
        (case["log2n_hi"] - case["log2n"] + 1)
    # a 64-bit transform and sort per iteration, and some launches per curve
    if total * (case["iters"] + 8) * 6e-10 + case["curves"] * (case["iters"] * 6e-4 + 4e-3) > 15.0:
        return None
    jobs = _jobs(case, seed)
    if kind in ("periodogram", "structure"):
        st = prepare(case, seed)
        x, p = st["x"].double(), st["plan"]
        outs = []
        for c, j in enumerate(jobs):
            xc, n = x[p.offsets[c]:p.offsets[c + 1]], 1 << j["log2n"]
            if kind == "periodogram":
                pw = torch.fft.rfft(xc).abs() ** 2
                outs.append(pw * (2.0 * j["dt"] * n / pw[0] if case["rms"] else 2.0 / (float(n) * n)))
            else:
                outs.append(torch.stack([torch.mean((xc[l:] - xc[:-l]) ** 2) for l in st["lags"]])[None])
        p.close()
        return torch.cat(outs)
    xs, tks, deltas, runs = [], [], [], []
    for j in jobs:
        X = _spectrum(j)
        x = _draws(j)
        if case["prec"] == "fp32" and kind == "iterate":
            x = x.float().double()  # the state that the call is given
        if kind == "setup":
            tks.append(torch.fft.irfft(X, n=x.numel()) * x.numel())
        else:
            x, d = _iterate(x, X.abs(), case["iters"], case["threshold"] if kind == "converge" else None)
            deltas.append(d + [math.nan] * (case["iters"] - len(d)))
            runs.append(len(d))
        xs.append(x)
    x = torch.cat(xs)
    if kind == "setup":
        return [torch.cat(tks), x]
    if kind == "converge":
        return [x, np.array(deltas), None]
    return x
