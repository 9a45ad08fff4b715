"""The work a user of this framework has it do, as cases to be timed and compared.

A case is one pass through the public entry points (``paper_1501_05427_gb300.ulisse``) on inputs
made from a seed on the GPU: covariance products K V (FP32, mixed, FP64; one problem or many),
the gradient's bilinear forms, ULISSE solves, SGLD steps and chains, the posterior predictive.
``work`` counts what a pass cannot do without: every distinct kernel value once (k_ij = k_ji),
the contractions, every input read and every output written once.  ``exact`` is the same
result in 64 bits from plain torch and numpy.

The entry points hand host results (gradients, parameters) back as doubles whatever the
context's precision; FP32 and mixed contexts compute them in 32 bits, so their cases return
them as 32-bit values, as a user's trace tensor keeps them.
"""
import math

import numpy as np
import torch

from paper_1501_05427_gb300 import ulisse as u

PREC = {"fp32": u.PREC_FP32, "mixed": u.PREC_MIXED, "fp64": u.PREC_FP64}


def listed():
    return [
        # one product on a Concrete-sized problem (n = 1,030, d = 8; y and 4 probes): a call
        # whose launches weigh as much as its arithmetic
        {"name": "kmv_fp32_concrete", "op": "kmv", "prec": "fp32", "n": 1030, "d": 8, "R": 5,
         "which": -1},
        # the default precision on the Census data set's own size (n = 22,784, d = 8), y and 16
        # probes: the product every CG round of a gradient repeats
        {"name": "kmv_fp32_census", "op": "kmv", "prec": "fp32", "n": 22784, "d": 8, "R": 17,
         "which": -1},
        # the same product on the tensor cores at the benchmark's size
        {"name": "kmv_mixed_census", "op": "kmv", "prec": "mixed", "n": 50000, "d": 8, "R": 17,
         "which": -1},
        # the largest: 200,000 16-dimensional inputs, 64 right-hand sides
        {"name": "kmv_mixed_200k", "op": "kmv", "prec": "mixed", "n": 200000, "d": 16, "R": 64,
         "which": -1},
        # double precision (the paper's own products) on the small 2-D problem
        {"name": "kmv_fp64_small_2d", "op": "kmv", "prec": "fp64", "n": 1000, "d": 2, "R": 5,
         "which": -1},
        # many uneven problems in one launch, the batched sampler's product (8 probes)
        {"name": "kmv_batch_mixed", "op": "batch_kmv", "prec": "mixed", "problems": 16,
         "n_lo": 2000, "n_hi": 20000, "R": 9},
        # the gradient's pass over the covariance at the benchmark's size, tensor cores
        {"name": "bilinear_mixed_census", "op": "bilinear", "prec": "mixed", "n": 50000, "d": 8,
         "M": 17},
        # the same pass in the default precision, an odd size and a 4-dimensional problem
        {"name": "bilinear_fp32_odd", "op": "bilinear", "prec": "fp32", "n": 9937, "d": 4,
         "M": 9},
        # one ULISSE solve of y and 16 probes from zero, as a gradient without warm starts
        {"name": "solve_fp32", "op": "solve", "prec": "fp32", "n": 9937, "d": 16, "R": 17},
        # one whole SGLD step (solves, gradient, update), mixed precision
        {"name": "step_mixed", "op": "step", "prec": "mixed", "n": 20000, "d": 16, "probes": 16},
        # the double-precision chain on the small 2-D problem, ten steps resident on the device
        {"name": "chain_fp64_small_2d", "op": "chain", "prec": "fp64", "n": 1000, "d": 2,
         "probes": 4, "steps": 10},
        # serving: mean and variance of new labels at one parameter sample, exact solves
        {"name": "predict_fp64", "op": "predict", "prec": "fp64", "n": 1030, "d": 2, "m": 100},
    ]


def _between(rng, lo, hi):
    """A whole number between lo and hi, spread over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["kmv", "kmv", "kmv", "batch_kmv", "bilinear", "bilinear", "solve", "step",
                     "chain", "predict"])
    if op == "kmv":
        prec = rng.choice(["fp32", "mixed", "fp64"])
        hi = {"fp32": 50000, "mixed": 150000, "fp64": 6000}[prec]
        d = rng.randint(1, 16)
        # one product in four is a derivative's, dK/dlog l_k V
        which = rng.randrange(d) if rng.random() < 0.25 and prec != "mixed" else -1
        return {"op": op, "prec": prec, "n": _between(rng, 500, hi), "d": d,
                "R": _between(rng, 1, 32 if prec != "mixed" else 64), "which": which}
    if op == "batch_kmv":
        lo = _between(rng, 500, 4000)
        return {"op": op, "prec": rng.choice(["fp32", "mixed"]), "problems": rng.randint(2, 24),
                "n_lo": lo, "n_hi": lo + _between(rng, 1000, 12000), "R": rng.randint(1, 17)}
    if op == "bilinear":
        prec = rng.choice(["fp32", "mixed", "fp64"])
        return {"op": op, "prec": prec,
                "n": _between(rng, 500, {"fp32": 30000, "mixed": 70000, "fp64": 4000}[prec]),
                "d": rng.randint(1, 16), "M": rng.choice([2, 5, 9, 17, 17, 33])}
    if op == "solve":
        return {"op": op, "prec": rng.choice(["fp32", "fp64"]), "n": _between(rng, 500, 4000),
                "d": rng.randint(12, 16), "R": rng.randint(1, 24)}
    if op == "step":
        return {"op": op, "prec": rng.choice(["fp32", "mixed"]), "n": _between(rng, 1000, 20000),
                "d": 16, "probes": rng.randint(2, 16)}
    if op == "chain":
        return {"op": op, "prec": "fp64", "n": rng.randint(200, 1500), "d": 2,
                "probes": rng.randint(2, 6), "steps": rng.randint(2, 10)}
    return {"op": op, "prec": "fp64", "n": rng.randint(300, 1500), "d": rng.randint(1, 3),
            "m": rng.randint(1, 100)}


# ------------------------------------------------------------------------------------------
# Inputs
# ------------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _labels(X, ls, noise, g):
    """A random-Fourier-feature draw of the covariance's signal part plus noise."""
    F = 512
    om = torch.randn(X.shape[1], F, generator=g, device="cuda") / ls[:, None]
    ph = torch.rand(F, generator=g, device="cuda") * (2 * math.pi)
    w = torch.randn(F, generator=g, device="cuda")
    y = torch.cos(X @ om + ph) @ w * math.sqrt(2.0 / F)
    return y + math.sqrt(noise) * torch.randn(X.shape[0], generator=g, device="cuda")


def _problem(n, d, g):
    """Inputs, labels and parameters (log l_1..log l_d, log sigma^2, log lambda): up to three
    dimensions as the small 2-D workload (uniform inputs), more as the Census-like and the
    16-dimensional ones (normal inputs, lengthscales log-uniform in [0.5, 2] times
    sqrt(d / 8) above eight)."""
    if d <= 3:
        X = torch.rand(n, d, generator=g, device="cuda")
        ls = torch.full((d,), 0.3, device="cuda")
        noise = 0.1
    else:
        X = torch.randn(n, d, generator=g, device="cuda")
        r = torch.rand(d, generator=g, device="cuda")
        ls = torch.exp(math.log(0.5) + r * math.log(4.0)) * math.sqrt(max(1.0, d / 8.0))
        noise = 0.05
    y = _labels(X, ls, noise, g)
    psi = np.concatenate([np.log(ls.double().cpu().numpy()), [0.0, math.log(noise)]])
    return X, y, psi


def _columns(n, R, g, dtype=torch.float32):
    """An (n, R) block of normal columns in the layout the library takes (column-major)."""
    return torch.randn(R, n, generator=g, device="cuda", dtype=dtype).t()


def _signs(n, R, g):
    return (torch.randint(0, 2, (R, n), generator=g, device="cuda") * 2 - 1).float().t()


def _inputs(case, seed):
    """What a case reads, from the seed alone: shared by prepare and exact."""
    g = _gen(seed)
    op = case["op"]
    s = {}
    if op == "batch_kmv":
        # the sizes belong to the case: uneven over [n_lo, n_hi], one problem at the upper end
        gh = np.random.default_rng([case["n_lo"], case["n_hi"], case["problems"]])
        ns = gh.integers(case["n_lo"], case["n_hi"] + 1, case["problems"])
        ns[-1] = case["n_hi"]
        ds = gh.choice([2, 4, 8], case["problems"])
        s["Xs"], s["ys"], psis = [], [], []
        for n, d in zip(ns, ds):
            X, y, psi = _problem(int(n), int(d), g)
            s["Xs"].append(X)
            s["ys"].append(y)
            psis.append(psi)
        s["psis"] = psis
        s["Vs"] = [_columns(X.shape[0], case["R"], g) for X in s["Xs"]]
        return s
    n, d = case["n"], case["d"]
    s["X"], s["y"], s["psi"] = _problem(n, d, g)
    if op == "kmv":
        s["V"] = _columns(n, case["R"], g,
                          torch.float64 if case["prec"] == "fp64" else torch.float32)
    elif op == "bilinear":
        # the factors of Eq. gradient:unbiased: solver estimates on the left, on the right
        # a second estimate of K^{-1} y and the probes the other estimates belong to
        M = case["M"]
        P = _signs(n, M, g)
        s["B"] = P
        s["A"] = (P * (0.5 + torch.rand(M, n, generator=g, device="cuda").t())).t().contiguous().t()
        s["scale"] = np.array([0.5] + [-0.5 / max(1, M - 1)] * (M - 1))
    elif op == "solve":
        B = _signs(n, case["R"], g).t().contiguous()
        B[0] = s["y"]
        s["B"] = B.t()
        s["n_est"] = [2] + [1] * (case["R"] - 1)
    elif op == "predict":
        s["Xs"] = torch.rand(case["m"], d, generator=g, device="cuda")
    return s


def _config(case):
    prec = PREC[case["prec"]]
    if case["op"] in ("step", "chain"):
        kind = u.PROBE_GAUSSIAN if case["op"] == "chain" else u.PROBE_RADEMACHER
        return u.ulisse_config_default(precision=prec, n_probes=case["probes"], probe_kind=kind,
                                       seed=1501)
    if case["op"] == "solve":
        return u.ulisse_config_default(precision=prec, seed=1501)
    if case["op"] == "predict":   # q = 0: every column to its convergence threshold
        return u.ulisse_config_default(precision=prec, q=0.0, eps=1e-7, max_iter=5000)
    return u.ulisse_config_default(precision=prec)


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = dict(case)
    if case["op"] == "batch_kmv":
        s["ctx"] = u.BatchContext(s["Xs"], s["ys"], _config(case))
        s["psi"] = np.concatenate(s["psis"])
        return s
    s["ctx"] = u.Context(s["X"], s["y"], _config(case))
    if case["op"] == "chain":
        p = case["d"] + 2
        s["psi0"] = torch.from_numpy(s["psi"]).cuda()
        s["psi_dev"] = s["psi0"].clone()
        s["eps"] = torch.full((case["steps"],), 1e-4, dtype=torch.float64, device="cuda")
        s["trace"] = torch.empty(case["steps"], p, dtype=torch.float64, device="cuda")
    return s


# ------------------------------------------------------------------------------------------
# One pass
# ------------------------------------------------------------------------------------------
def run(s):
    c, ctx = s["case"], s["ctx"]
    op = c["op"]
    if op == "kmv":
        return ctx.kmv(s["psi"], s["V"], which=c["which"])
    if op == "batch_kmv":
        return ctx.kmv(s["psi"], s["Vs"])
    if op == "bilinear":
        g = ctx.dk_bilinear(s["psi"], s["A"], s["B"], s["scale"])
        return g if c["prec"] == "fp64" else g.astype(np.float32)
    if op == "solve":
        return ctx.solve(s["psi"], s["B"], n_est=s["n_est"], step=3)[0]
    if op == "step":
        psi, g = ctx.sgld_step(s["psi"], 1e-4, 3)
        return psi.astype(np.float32), g.astype(np.float32)
    if op == "chain":
        s["psi_dev"].copy_(s["psi0"])
        ctx.sgld_chain(s["psi_dev"], s["eps"], step0=3, trace_dev=s["trace"])
        return s["trace"].float()
    return ctx.predict(s["psi"], s["Xs"], step=3)


# ------------------------------------------------------------------------------------------
# Work
# ------------------------------------------------------------------------------------------
def _kv_flops(n, d, R):
    return n * (n + 1) / 2 * (3 * d + 2) + 2.0 * R * n * n


def work(case):
    op = case["op"]
    e = 8 if case["prec"] == "fp64" else 4
    if op == "batch_kmv":
        n = (case["n_lo"] + case["n_hi"]) / 2
        n2 = n * n + (case["n_hi"] - case["n_lo"]) ** 2 / 12
        B, R, d = case["problems"], case["R"], 5
        return {"bytes": B * n * 4 * (d + 2 * R), "flops": B * (n2 / 2 * (3 * d + 2) + 2 * R * n2)}
    n, d = case["n"], case["d"]
    if op == "kmv":
        return {"bytes": n * (4 * d + 2 * e * case["R"]), "flops": _kv_flops(n, d, case["R"])}
    if op == "bilinear":
        M = case["M"]
        return {"bytes": 4 * n * (d + 2 * M), "flops": n * (n + 1) / 2 * (5 * d + 4 + 4 * M)}
    if op == "solve":     # a few CG rounds on 16-dimensional inputs
        R = case["R"]
        return {"bytes": 4 * n * (d + 2 * R + 1), "flops": 4 * _kv_flops(n, d, R)}
    if op == "step":
        M = 1 + case["probes"]
        return {"bytes": 4 * n * (d + 1),
                "flops": 4 * _kv_flops(n, d, M) + n * (n + 1) / 2 * (5 * d + 4 + 4 * M)}
    if op == "chain":
        M = 1 + case["probes"]
        per = 20 * _kv_flops(n, d, M) + n * (n + 1) / 2 * (5 * d + 4 + 4 * M)
        return {"bytes": 4 * n * (d + 1), "flops": case["steps"] * per}
    return {"bytes": 4 * (n * (d + 1) + case["m"] * (d + 2)),
            "flops": 50 * _kv_flops(n, d, 1 + case["m"])}


# ------------------------------------------------------------------------------------------
# The same results in 64 bits
# ------------------------------------------------------------------------------------------
def _signal(Xa, Xb, psi, d):
    """sigma^2 exp(-|xa - xb|^2 / 2) on prescaled rows, 64 bits."""
    D = torch.cdist(Xa, Xb, compute_mode="donot_use_mm_for_euclid_dist") if d <= 3 else None
    if D is not None:
        return math.exp(psi[d]) * torch.exp(-0.5 * D * D)
    sq = (Xa * Xa).sum(1)[:, None] + (Xb * Xb).sum(1)[None, :]
    sq.addmm_(Xa, Xb.t(), alpha=-2.0)
    return math.exp(psi[d]) * sq.clamp_(min=0).mul_(-0.5).exp_()


def _scaled(X, psi):
    d = X.shape[1]
    return X.double() / torch.from_numpy(np.exp(psi[:d])).cuda()


def _exact_kv(X, psi, V, which=-1):
    d, n = X.shape[1], X.shape[0]
    Z = _scaled(X, psi)
    V = V.double().contiguous()
    U = torch.empty_like(V)
    step = max(256, int(2e8) // n)
    for i in range(0, n, step):
        K = _signal(Z[i:i + step], Z, psi, d)
        if which >= 0:
            K *= (Z[i:i + step, which, None] - Z[None, :, which]) ** 2
        U[i:i + step] = K @ V
    return U if which >= 0 else U + math.exp(psi[d + 1]) * V


def _exact_bilinear(X, psi, A, B, scale):
    d, n = X.shape[1], X.shape[0]
    Z = _scaled(X, psi)
    A = A.double() * torch.from_numpy(scale).cuda()
    B = B.double().contiguous()
    out = torch.zeros(d + 2, dtype=torch.float64, device="cuda")
    step = max(256, int(1e8) // n)
    for i in range(0, n, step):
        Zi = Z[i:i + step]
        P = _signal(Zi, Z, psi, d) * (A[i:i + step] @ B.t())
        for k in range(d):
            out[k] += (P * (Zi[:, k, None] - Z[None, :, k]) ** 2).sum()
        out[d] += P.sum()
    out[d + 1] = math.exp(psi[d + 1]) * (A * B).sum()
    return out


def _accepted(seed, step, column, estimator, most):
    """J: steps kept after the early stop, j = 1, 2, ... while u_j < exp(-j) (beta = 1)."""
    for j in range(1, most + 1):
        c = j + (column << 64) + (step << 128) + ((2 | estimator << 8) << 192)
        word = int(np.random.Philox(counter=c - 1, key=seed).random_raw())
        if not (word >> 11) * 2.0 ** -53 < math.exp(-j):
            return j - 1
    return most


def _exact_solve(X, psi, B, n_est, step, seed=1501, most=1000):
    """Conjugate gradients from zero on every column, truncated and reweighted (q = beta = 1)."""
    d, n = X.shape[1], X.shape[0]
    Z = _scaled(X, psi)
    K = _signal(Z, Z, psi, d)
    K.diagonal().add_(math.exp(psi[d + 1]))
    out = []
    for c, ne in enumerate(n_est):
        b = B[:, c].double()
        s, e, dv = torch.zeros_like(b), b.clone(), b.clone()
        ee = float(e @ e)
        J = [_accepted(seed, step, c, t, most) for t in range(ne)]
        est, l = None, 0
        for m in range(1, most + 1):
            kd = K @ dv
            al = ee / float(dv @ kd)
            s = s + al * dv
            if est is not None:
                w = math.exp((m - l) * (m - l + 1) / 2)
                for t in range(ne):
                    if J[t] >= m - l:
                        est[t] = est[t] + w * al * dv
            e = e - al * kd
            new = float(e @ e)
            if est is None and math.sqrt(new) < math.sqrt(n):
                l, est = m, [s] * ne
            if est is not None and m - l >= max(J):
                break
            dv = e + (new / ee) * dv
            ee = new
        out += est
    return torch.stack(out, 1)


def exact(case, seed):
    op = case["op"]
    if op in ("step", "chain"):   # whole steps: their parts are cases of their own
        return None
    s = _inputs(case, seed)
    if op == "batch_kmv":
        return [_exact_kv(X, p, V) for X, p, V in zip(s["Xs"], s["psis"], s["Vs"])]
    if op == "kmv":
        return _exact_kv(s["X"], s["psi"], s["V"], case["which"])
    if op == "bilinear":
        return _exact_bilinear(s["X"], s["psi"], s["A"], s["B"], s["scale"])
    if op == "solve":
        return _exact_solve(s["X"], s["psi"], s["B"], s["n_est"], 3)
    d = case["d"]
    psi, Z = s["psi"], _scaled(s["X"], s["psi"])
    K = _signal(Z, Z, psi, d)
    K.diagonal().add_(math.exp(psi[d + 1]))
    ks = _signal(Z, _scaled(s["Xs"], psi), psi, d)
    S = torch.linalg.solve(K, torch.cat([s["y"].double()[:, None], ks], 1))
    mean = ks.t() @ S[:, 0]
    var = math.exp(psi[d]) + math.exp(psi[d + 1]) - (ks * S[:, 1:]).sum(0)
    return mean, var
