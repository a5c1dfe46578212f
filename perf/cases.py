"""The work that a user of this framework has it do, as cases that can be timed.

Five kinds of use, each through the public entry points of
``paper_1905_10252_gb300.native``:

* ``step``  a standing sampler advanced by K iterations of Algorithm 2 in one
            call (``Sampler.step``), its particles read afterwards,
* ``loop``  the user's own iteration out of the separate calls (move, reweight,
            estimate with the covariance, resample and redistribute when the
            last statistics asked for it),
* ``job``   a whole run, from creating the sampler to its posterior (what a
            server does for each request),
* ``raw``   stateless resampling and redistribution of the caller's own
            log-weights and rows,
* ``batch`` many small samplers stepped together (``Batch``).

A case names its kind and sizes; inputs are drawn from the seed alone.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1905_10252_gb300 import inputs, native

_MODES = {"ess": native.RESAMPLE_ESS, "always": native.RESAMPLE_ALWAYS}
_DTYPES = {"f32": torch.float32, "f64": torch.float64}
_STEP, _SCALE, _PRIOR = 0.5, 2.0, 4.0  # proposal, q0 and the logistic prior of the repository's workloads
_L2 = 128e6  # bytes of state that stay on the chip from one iteration to the next


def listed():
    return [
        # the headline workload: a large sampler that resamples in every iteration, its copy left to the next move
        dict(name="step_large", kind="step", target="gauss", dtype="f32", n=1 << 24, d=16, mode="always", defer=True,
             k=4, m=0, cov=False),
        # an ordinary sampler of a ragged size that resamples when N_eff asks for it
        dict(name="step_ess", kind="step", target="gauss", dtype="f32", n=1_000_003, d=8, mode="ess", defer=False,
             k=10, m=0, cov=False),
        # the widest state, with the posterior covariance after the last iteration
        dict(name="step_wide", kind="step", target="gauss", dtype="f32", n=1 << 20, d=32, mode="ess", defer=False,
             k=5, m=0, cov=True),
        # double precision throughout
        dict(name="step_fp64", kind="step", target="gauss", dtype="f64", n=1 << 18, d=8, mode="ess", defer=False,
             k=5, m=0, cov=False),
        # the tensor-core likelihood at its full data size
        dict(name="logistic_large", kind="step", target="logistic", dtype="f32", n=1 << 18, d=32, mode="ess",
             defer=False, k=2, m=8192, cov=False),
        # a user's own loop over the separate calls, mean and covariance in every iteration
        dict(name="loop_moments", kind="loop", target="gauss", dtype="f32", n=2_000_003, d=12, mode="ess", m=0),
        # the same over a small regression: few data rows, a ragged number of particles
        dict(name="loop_logistic", kind="loop", target="logistic", dtype="f32", n=30_011, d=7, mode="ess", m=1000),
        # the plain double-precision sampler, from creation to its posterior
        dict(name="job_fp64", kind="job", target="gauss", dtype="f64", n=1024, d=4, mode="ess", defer=False, k=20,
             m=0, cov=False),
        # one request of the serving stream
        dict(name="job_wide", kind="job", target="gauss", dtype="f32", n=20_011, d=32, mode="ess", defer=False, k=50,
             m=0, cov=True),
        # resampling and redistribution of the caller's own rows: the largest, and a small odd one
        dict(name="raw_large", kind="raw", dtype="f32", n=1 << 24, d=16, weights="2"),
        dict(name="raw_small", kind="raw", dtype="f32", n=65_537, d=3, weights="0.5"),
        # many samplers of different sizes in one launch per stage
        dict(name="batch", kind="batch", members=60, k=10, lo=10, hi=18),
    ]


def _size(rng, lo, hi):
    """A size spread over the logarithm of [lo, hi], odd ones among them."""
    n = int(math.exp(rng.uniform(math.log(lo), math.log(hi))))
    return max(lo, min(hi, n | 1 if rng.random() < 0.5 else n))


def draw(rng):
    kind = rng.choice(["step", "step", "loop", "loop", "job", "job", "raw", "raw", "batch"])
    if kind == "raw":
        d = rng.choice([1, 2, 3, 4, 5, 8, 12, 16, 31, 32])
        return dict(kind="raw", dtype=rng.choice(["f32", "f64"]), n=_size(rng, 1 << 10, (1 << 26) // max(d, 4)), d=d,
                    weights=rng.choice(["0.5", "2", "8", "one_hot"]))
    if kind == "batch":
        return dict(kind="batch", members=_size(rng, 8, 60), k=2 * rng.randint(1, 5), lo=rng.randint(8, 12),
                    hi=rng.randint(15, 18))
    target = rng.choice(["gauss", "gauss", "gauss", "student_t", "logistic"])
    dtype = rng.choice(["f32", "f32", "f64"]) if target != "logistic" else "f32"
    d = 1 if target == "student_t" else rng.randint(2, 32)
    m = _size(rng, 200, 8192) if target == "logistic" else 0
    k = rng.randint(1, 10) if kind == "step" else (rng.choice([20, 50]) if kind == "job" else 1)
    most = 1 << (24 if dtype == "f32" else 20)
    if target == "logistic":
        most = min(1 << 18, (1 << 31) // (m * k))
    elif kind == "job":
        most = 1 << 18 if dtype == "f32" else 1 << 14
    else:
        most = min(most, (1 << (28 if dtype == "f32" else 24)) // (d * k))
    n = _size(rng, 1 << 10, max(most, 1 << 11))
    case = dict(kind=kind, target=target, dtype=dtype, n=n, d=d, m=m, mode=rng.choice(["ess", "ess", "always"]))
    if kind != "loop":
        case.update(k=k, defer=rng.random() < 0.3, cov=rng.random() < 0.3)
    return case


def _target(case, seed):
    """The target's parameters as Sampler takes them, on the GPU."""
    d = case["d"]
    if case["target"] == "student_t":
        return dict(target="student_t", mu=torch.tensor([1.5], dtype=torch.float64, device="cuda"), nu=5.0)
    if case["target"] == "logistic":
        X, y, _ = inputs.logistic_data(case["m"], d, seed)
        return dict(target="logistic", X=torch.from_numpy(X).cuda(), y=torch.from_numpy(y).cuda(), prior_var=_PRIOR)
    mu, sigma = inputs.gaussian_target(d, seed)
    return dict(target="gauss", mu=torch.from_numpy(mu).cuda(), sigma=torch.from_numpy(sigma).cuda())


def _arguments(case, seed):
    return dict(n=case["n"], d=case["d"], dtype=_DTYPES[case["dtype"]], seed=seed, step=_STEP, init_scale=_SCALE,
                resample_mode=_MODES[case["mode"]],
                flags=native.FLAG_DEFER_REDISTRIBUTE if case.get("defer") else 0, **_target(case, seed))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "job":
        return dict(case=case, args=_arguments(case, seed))
    if kind == "raw":
        g = torch.Generator(device="cuda").manual_seed(seed)
        n = case["n"]
        x = torch.randn(n, case["d"], generator=g, device="cuda", dtype=torch.float32).to(_DTYPES[case["dtype"]])
        if case["weights"] == "one_hot":
            logw = torch.full((n,), -math.inf, dtype=torch.float64, device="cuda")
            logw[int(torch.randint(n, (1,), generator=g, device="cuda"))] = 0.0
        else:
            logw = float(case["weights"]) * torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
        return dict(case=case, seed=seed, x=x, logw=logw, out=torch.empty_like(x),
                    ncopies=torch.empty(n, dtype=torch.int32, device="cuda"),
                    stats=torch.zeros(native.STATS_WORDS, dtype=torch.float64, device="cuda"),
                    ws=torch.empty(native.smc_redistribute_ws_bytes(n), dtype=torch.uint8, device="cuda"))
    if kind == "batch":
        # ragged sizes spread over the logarithm of the range, the largest among them
        span = case["hi"] - case["lo"]
        ns = [int(2.0 ** (case["hi"] - span * (i * 0.6180339887498949 % 1.0))) for i in range(case["members"])]
        ds = [(2, 8, 32)[i % 3] for i in range(case["members"])]
        members = []
        for i, (n, d) in enumerate(zip(ns, ds)):
            mu, sigma = inputs.gaussian_target(d, seed + i)
            members.append(native.Sampler(n, d, seed=seed + i, mu=mu, sigma=sigma, step=_STEP, init_scale=_SCALE,
                                          resample_mode=native.RESAMPLE_ALWAYS))
        means = torch.zeros(len(members), 32, dtype=torch.float64, device="cuda")
        trace = torch.zeros(len(members), case["k"], native.STATS_WORDS, dtype=torch.float64, device="cuda")
        return dict(case=case, members=members, batch=native.Batch(members), means=means, trace=trace)
    return dict(case=case, sampler=native.Sampler(**_arguments(case, seed)), resample=0)


def _records(trace):
    """smc_iter_stats records: the numbers, and the whole numbers behind them."""
    return dict(stats=trace[..., :4], counts=trace.view(torch.int64)[..., 4:])


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "raw":
        w = case["n"], state["ws"]
        native.smc_resample_raw(state["logw"], state["seed"], 1, ncopies=state["ncopies"], ws=w[1],
                                stats=state["stats"])
        native.smc_redistribute_raw(state["ncopies"], state["x"], state["out"], w[1])
        return dict(ncopies=state["ncopies"], x=state["out"], **_records(state["stats"]))
    if kind == "batch":
        # every member resamples in each of an even number of iterations: its particles are in its first buffer
        ms = state["members"]
        state["batch"].step_raw(case["k"], means=[state["means"][i, : m.d] for i, m in enumerate(ms)],
                                traces=[state["trace"][i] for i in range(len(ms))])
        return dict(x=[m.x for m in ms], mean=state["means"], **_records(state["trace"]))
    if kind == "loop":
        s = state["sampler"]
        if state["resample"]:
            ncopies, _ = s.resample()
            s.redistribute(ncopies)
        s.move()
        s.reweight()
        mean, cov = s.estimate(cov=True)
        state["resample"] = s.stats()["resampled"]
        x, logpi = s.current()
        return dict(x=x, logpi=logpi, logw=s.logw, mean=mean, cov=cov)
    s = state["sampler"] if kind == "step" else native.Sampler(**state["args"])
    out = s.step(case["k"], cov=case["cov"], trace=True, fhat=True)
    x, logpi = s.current()
    got = dict(x=x, logpi=logpi, logw=s.logw, mean=out["mean"], fhat=out["fhat"], **_records(out["trace"]))
    if case["cov"]:
        got["cov"] = out["cov"]
    return got


def _iteration(n, d, es, m):
    """(bytes, flops) of one iteration: the state read and written; the normals, the target, the weights."""
    target = m * (2.0 * d + 8.0) if m else d * (d + 1.0)
    return n * (2.0 * d * es + 2.0 * es + 16.0), n * (30.0 * d + target + 40.0)


def work(case):
    kind = case["kind"]
    if kind == "raw":
        n, row = case["n"], case["d"] * (4 if case["dtype"] == "f32" else 8)
        # expected share of rows with a copy, from which each is read once
        alive = {"0.5": 0.63, "2": 0.4, "8": 0.05, "one_hot": 0.0}[case["weights"]]
        return dict(bytes=n * (8.0 + 4.0 + row * (1.0 + alive)), flops=n * 20.0)
    if kind == "batch":
        lo, hi = case["lo"], case["hi"]
        n = case["members"] * (2.0**hi - 2.0**lo) / (math.log(2.0) * (hi - lo))
        b, f = (sum(v) / 3.0 for v in zip(*(_iteration(n, d, 4, 0) for d in (2, 8, 32))))
        return dict(bytes=b * (case["k"] if b > _L2 else 1), flops=f * case["k"])
    k = case.get("k", 1)
    n, d, es = case["n"], case["d"], 4 if case["dtype"] == "f32" else 8
    b, f = _iteration(n, d, es, case["m"])
    cov = n * (d * (d + 1.0) + 2.0 * d) if kind == "loop" or case["cov"] else 0.0
    return dict(bytes=b * (k if b > _L2 else 1), flops=f * k + cov)


# ------------------------------------------------------------------ 64-bit values
def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 (Salmon et al., SC'11) on 32-bit words held in int64 tensors."""
    low = 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & low) ^ c1 ^ k0, p1 & low, ((p0 >> 32) & low) ^ c3 ^ k1, p0 & low
        k0, k1 = (k0 + 0x9E3779B9) & low, (k1 + 0xBB67AE85) & low
    return c0, c1, c2, c3


def _normals(n, d, seed, t, purpose, dtype):
    """The n x d standard normals of a sampler's stream, in 64 bits."""
    i = torch.arange(n, dtype=torch.int64, device="cuda")
    z = torch.empty(n, d + 1, dtype=torch.float64, device="cuda")
    zero = torch.zeros_like(i)
    pairs = (d + 1) // 2
    for p in range(pairs):
        block = p // 2 if dtype == "f32" else p
        w = _philox(i, zero + t, zero + ((purpose << 24) | block), zero, seed & 0xFFFFFFFF, seed >> 32)
        if dtype == "f32":
            a, b = ((v >> 8).double() * 2.0**-24 for v in w[2 * (p % 2): 2 * (p % 2) + 2])
        else:
            a, b = (((u << 21) | (v >> 11)).double() * 2.0**-53 for u, v in (w[:2], w[2:]))
        r = torch.sqrt(-2.0 * torch.log1p(-a))
        z[:, 2 * p] = r * torch.cos(2.0 * math.pi * b)
        if 2 * p + 1 < d:
            z[:, 2 * p + 1] = r * torch.sin(2.0 * math.pi * b)
    return z[:, :d]


def _logpi(case, seed, x):
    if case["target"] == "student_t":
        return -3.0 * torch.log1p((x[:, 0] - 1.5) ** 2 / 5.0)
    if case["target"] == "logistic":
        X, y, _ = inputs.logistic_data(case["m"], case["d"], seed)
        X, y = torch.from_numpy(X).cuda().double(), torch.from_numpy(y).cuda().double()
        out = torch.empty(x.shape[0], dtype=torch.float64, device="cuda")
        rows = max(1, (1 << 27) // case["m"])
        for a in range(0, x.shape[0], rows):
            z = x[a:a + rows] @ X.T
            out[a:a + rows] = z @ y - torch.logaddexp(z, torch.zeros_like(z)).sum(1)
        return out - (x * x).sum(1) / (2.0 * _PRIOR)
    mu, sigma = inputs.gaussian_target(case["d"], seed)
    v = x - torch.from_numpy(mu).cuda()
    return -0.5 * (v @ torch.from_numpy(np.linalg.inv(sigma)).cuda() * v).sum(1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "raw":
        state = prepare(case, seed)
        w, m = state["logw"], state["logw"].max()
        e = torch.exp(w - m)
        lse = m + torch.log(e.sum())
        stats = torch.stack([lse, lse, e.sum() ** 2 / (e * e).sum(), m])
        return dict(ncopies=None, x=None, stats=stats, counts=None)
    if kind != "loop":
        return None  # later iterations depend on every rounding before them through the copies
    n, d = case["n"], case["d"]
    x0 = _SCALE * _normals(n, d, seed, 0, 1, case["dtype"])
    x = x0 + _STEP * _normals(n, d, seed, 1, 2, case["dtype"])
    logpi = _logpi(case, seed, x)
    logw = logpi + (x0 * x0).sum(1) / (2.0 * _SCALE**2)
    w = torch.exp(logw - logw.max())
    w = w / w.sum()
    mean = w @ x
    cov = (x - mean).T @ (w[:, None] * (x - mean))
    return dict(x=x, logpi=logpi, logw=logw, mean=mean, cov=cov)
