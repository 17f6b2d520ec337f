"""Performance cases of the exact sparse GP: the calls a user of the library makes once a point set is assembled.

A case is one pass of a user's inner loop through the Python binding of the C-ABI: settings in
(Factor.update), log-likelihoods out (Factor.loglik), and where the user predicts, means (Factor.predict) or
variances (Factor.predict_var); or a burst of requests through the request server. What a program sets up once
and keeps -- the assembled point set, the factor's memory, the server with its point sets -- is prepared outside the
pass. Inputs are the seeded synthetic workloads of the package (`synth`), drawn anew from the case's seed.
"""
import math

import numpy as np
import torch

from paper_2411_05869_gb300 import gp, synth

PREC = {"fp64": gp.GP_FP64, "mixed": gp.GP_MIXED}
EXACT_MAX_N = 32000        # dense 64-bit references up to this many points
EXACT_MAX_REQUEST_N = 10000


def _case(kind, n, prec, m=0, B=1, **kw):
    c = {"kind": kind, "n": n, "prec": prec, "m": m, "B": B, "nnz_row": 50, "bumps": 8, "var": False,
         "group": 0, "default_stream": False}
    c.update(kw)
    return c


def listed():
    def named(name, c):
        return {"name": name, **c}
    return [
        # the smallest data set of the paper's simulations: 2000 points on the unit square, FP64, fit and predict;
        # launches and dependent steps count
        named("spatial_2k_fp64", _case("spatial", 2000, "fp64", m=500, bumps=4)),
        # the smaller end of a serving catalogue: one client's likelihood and prediction on 9000 space-time points
        named("spacetime_9k_mixed", _case("spacetime", 9000, "mixed", m=1000, nnz_row=60, bumps=16)),
        # the non-compact core of App. B at the size of its parity tests, FP64
        named("noncompact_12k_fp64", _case("noncompact", 12000, "fp64", bumps=4)),
        # 5000 stations x 6 days: the window on which results are checked in FP64
        named("station_30k_fp64", _case("station", 30000, "fp64", nnz_row=100, bumps=16)),
        # the non-compact core at its benchmark size, mixed precision
        named("noncompact_50k_mixed", _case("noncompact", 50000, "mixed", bumps=4)),
        # a burst of requests of uneven sizes through the request server, 70 % likelihoods and 30 % predictions
        named("serving_mix", {"kind": "serving", "n": 5000, "n_max": 50000, "sets": 5, "requests": 20, "slots": 4,
                              "prec": "mixed", "nnz_row": 60, "bumps": 16, "m": 10000}),
        # 100,000 space-time points: likelihood and predictive mean at 10,000 points, in both precisions
        named("spacetime_100k_mixed", _case("spacetime", 100000, "mixed", m=10000)),
        named("spacetime_100k_fp64", _case("spacetime", 100000, "fp64", m=10000)),
        # predictive variance on the same field, settings given once
        named("variance_100k_mixed", _case("spacetime", 100000, "mixed", m=2048, var=True)),
        # eight chains of an MCMC run on 200,000 points, one batched factorization per step
        named("chains_200k_mixed", _case("spacetime", 200000, "mixed", B=8, nnz_row=80, default_stream=True)),
        # the same point set in FP64, one setting: the reference value of a mixed run
        named("spacetime_200k_fp64", _case("spacetime", 200000, "fp64", nnz_row=80)),
        # the full station field, 5000 sites x 240 days, with the posterior mean on a 200 x 200 x 30 grid; groups of
        # 32 blocks is what the autotuner picks at this size
        named("station_1.2M_mixed", _case("station", 1200000, "mixed", m=1200000, nnz_row=100, bumps=16, group=32)),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["spatial", "spacetime", "spacetime", "station", "noncompact", "variance", "serving"])
    if kind == "serving":
        lo = _log_uniform(rng, 2000, 10000)
        return {"kind": "serving", "n": lo, "n_max": lo * rng.randint(3, 10), "sets": rng.randint(3, 6),
                "requests": rng.randint(8, 30), "slots": rng.choice([2, 4]), "prec": rng.choice(["mixed", "mixed", "fp64"]),
                "nnz_row": rng.randint(40, 80), "bumps": rng.choice([4, 8, 16]), "m": _log_uniform(rng, 1000, 50000)}
    prec = rng.choice(["fp64", "mixed"])
    bumps = rng.choice([4, 8, 16])
    stream = rng.random() < 0.25
    if kind == "spatial":
        return _case(kind, _log_uniform(rng, 1500, 30000), prec, m=_log_uniform(rng, 300, 5000), bumps=bumps,
                     B=rng.choice([1, 1, 4, 16]), default_stream=stream)
    if kind == "noncompact":
        return _case(kind, _log_uniform(rng, 3000, 50000), prec, bumps=4, B=rng.choice([1, 1, 3]),
                     m=rng.choice([0, 777]), default_stream=stream)
    if kind == "station":
        sites, days = rng.choice([1000, 3001, 5000]), _log_uniform(rng, 5, 240 if prec == "mixed" else 16)
        return _case(kind, sites * days, prec, sites=sites, nnz_row=rng.randint(60, 100), bumps=16,
                     m=rng.choice([0, _log_uniform(rng, 1000, 300000)]), default_stream=stream)
    if kind == "variance":
        return _case("spacetime", _log_uniform(rng, 5000, 100000), prec, m=_log_uniform(rng, 33, 2048 if prec == "mixed" else 256),
                     bumps=bumps, var=True, default_stream=stream)
    B = rng.choice([1, 1, 2, 5, 8])
    n = _log_uniform(rng, 5000, 200000 // (1 if prec == "mixed" else B))
    return _case(kind, n, prec, B=B, nnz_row=rng.randint(40, 80), bumps=bumps,
                 m=rng.choice([0, _log_uniform(rng, 1000, 50000)]), default_stream=stream)


# ---------------------------------------------------------------------------------------------------------- inputs
def _workload(case, seed):
    """The seeded workload of a case: points, test points, settings and residuals."""
    n, m, B = case["n"], case["m"], case["B"]
    rng = np.random.default_rng([seed, 77])
    if case["kind"] == "spatial":
        w = synth.spatial_2d(n, max(m, 1), seed=seed, nbumps=case["bumps"], rho=0.05 * math.sqrt(2000 / n))
        w.resid = np.sin(9.0 * w.X[:, 0]) * np.cos(7.0 * w.X[:, 1]) + math.sqrt(w.hyper.noise_var) * w.noise
    elif case["kind"] == "spacetime":
        # days in proportion to the points, as a longer record has
        w = synth.uniform_spacetime(n, max(m, 1), float(case["nnz_row"]), case["bumps"], seed,
                                    ndays=365 if n >= 50000 else max(30, round(365 * n / 50000)))
    elif case["kind"] == "station":
        sites = case.get("sites", 5000)
        full = m == 1200000
        w = synth.station_spacetime(sites, n // sites, nnz_row=float(case["nnz_row"]), nbumps=case["bumps"], seed=seed,
                                    with_test=full)
        if not full:
            w.Xtest = rng.uniform(size=(max(m, 1), 3))
            w.mu_test = np.zeros(max(m, 1))
    else:
        w = synth.noncompact_spatial(n, max(m, 1), seed=seed)
    w.thetas = [w.hyper] + [synth.perturb(rng, w.hyper) for _ in range(B - 1)]
    w.residuals = np.stack([w.resid] + [w.resid + 0.1 * rng.standard_normal(n) for _ in range(B - 1)])
    return w


def _serving_workload(case, seed):
    rng = np.random.default_rng([seed, 99])
    ns = np.exp(np.linspace(math.log(case["n"]), math.log(case["n_max"]), case["sets"])).astype(int)
    sets = [synth.uniform_spacetime(int(k), 0, float(case["nnz_row"]), case["bumps"], int(rng.integers(1 << 30)),
                                    ndays=max(30, round(365 * int(k) / 50000))) for k in ns]
    reqs = []
    for q in range(case["requests"]):
        i = q % case["sets"]
        m = case["m"] // (1 + q % 4) if q % 10 in (2, 5, 8) else 0
        xt = rng.uniform(size=(m, 3)) if m else None
        reqs.append((i, synth.perturb(rng, sets[i].hyper), xt))
    return sets, reqs


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


class _State:
    pass


_STREAMS = []


def _stream():
    """The program's one explicit stream: evaluations follow one another, as the steps of a sampler do."""
    if not _STREAMS:
        _STREAMS.append(torch.cuda.Stream())
    return _STREAMS[0]


def prepare(case, seed):
    s = _State()
    s.case = case
    if case["kind"] == "serving":
        sets, reqs = _serving_workload(case, seed)
        s.server = gp.Server(0, slots=case["slots"], mem_budget_bytes=16 << 30)
        s.resid = [_dev(w.resid) for w in sets]
        s.ids = [s.server.add_pointset(_dev(w.X), w.hyper.core_radius) for w in sets]
        s.reqs = [(i, th, None if xt is None else _dev(xt)) for i, th, xt in reqs]
        torch.cuda.synchronize()
        return s
    w = _workload(case, seed)
    s.stream = torch.cuda.default_stream() if case["default_stream"] else _stream()
    s.thetas, s.resid = w.thetas, _dev(w.residuals)
    s.Xt, s.mu = (_dev(w.Xtest), _dev(w.mu_test)) if case["m"] else (None, None)
    X = _dev(w.X)
    torch.cuda.synchronize()
    s.ctx = gp.Context(0, stream=s.stream)
    if case["kind"] == "noncompact":
        s.ps = s.ctx.assemble_sparse_support(X, w.hyper)
    else:
        s.ps = s.ctx.assemble(X, w.hyper.core_radius)
    if case["group"]:
        s.ps.set_blocking(case["group"], 256)
    s.factor = s.ctx.factor(s.ps, s.thetas, PREC[case["prec"]])
    torch.cuda.synchronize()
    return s


def run(s):
    case = s.case
    if case["kind"] == "serving":
        outs = []
        for i, th, xt in s.reqs:
            out = torch.empty(1 if xt is None else xt.shape[0], dtype=torch.float64, device="cuda")
            s.server.submit(s.ids[i], th, s.resid[i], out, PREC[case["prec"]], Xtest=xt)
            outs.append(out)
        s.server.wait()
        done = s.server.poll(len(outs))
        assert all(c["status"] == 0 for c in done)
        return outs
    with torch.cuda.stream(s.stream):
        if case["var"]:
            return {"variance": s.factor.predict_var(s.Xt)}
        s.factor.update(s.thetas)
        out = {"loglik": s.factor.loglik(s.resid)}
        if s.Xt is not None:
            out["mean"] = [s.factor.predict(s.Xt, s.mu, b=b) for b in range(case["B"])]
    return out


# ------------------------------------------------------------------------------------------------------------- work
def _factor_work(info, d, B, prec, m):
    """Bytes: points, residual and test points read, the pattern read, the factor written by the factorization and
    read by the backward solve (the forward solve can follow the factorization). Flops: sum of the squared column
    counts, the two triangular solves, and about 40 per pattern entry for the kernel values."""
    n, size = info["n"], 8 if prec == "fp64" else 4
    by = n * d * 8 + info["nnz"] * 4 + B * (n * 8 + 2 * info["nnzL"] * size + m * 16) + m * d * 8
    fl = B * (info["flops"] + 4 * info["nnzL"] + 40 * info["nnz"])
    if m:
        fl += B * m * 45 * (info["nnz"] / n)
    return by, fl


def _info(w, noncompact):
    ctx = gp.Context(0)
    ps = ctx.assemble_sparse_support(_dev(w.X), w.hyper) if noncompact else ctx.assemble(_dev(w.X), w.hyper.core_radius)
    info = ps.info()
    ps.free()
    ctx.close()
    return info


def work(case):
    if case["kind"] == "serving":
        by = fl = 0
        sets, reqs = _serving_workload(case, 1)
        infos = [_info(w, False) for w in sets]
        for i, _, xt in reqs:
            b, f = _factor_work(infos[i], 3, 1, case["prec"], 0 if xt is None else xt.shape[0])
            by, fl = by + b, fl + f
        return {"bytes": by, "flops": fl}
    w = _workload(case, 1)
    info = _info(w, case["kind"] == "noncompact")
    d = w.X.shape[1]
    if case["var"]:
        # every test point's forward solve passes the fronts on its neighbours' paths to the root; most of those
        # columns are in the top separators: counted as half of the factor's entries, read once for all test points
        size = 8 if case["prec"] == "fp64" else 4
        return {"bytes": info["nnzL"] * size + case["m"] * (d + 1) * 8, "flops": case["m"] * info["nnzL"]}
    by, fl = _factor_work(info, d, case["B"], case["prec"], case["m"])
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------------------------- 64-bit references (dense torch)
def _wendland(q):
    q = q.clamp(max=1.0)
    return (1 - q) ** 8 * (((35 * q + 25) * q + 8) * q + 1)


def _scaled_dist(A, B, rad):
    d2 = torch.zeros(A.shape[0], B.shape[0], dtype=torch.float64, device=A.device)
    for k in range(A.shape[1]):
        d2 += (A[:, k, None] / rad[k] - B[None, :, k] / rad[k]) ** 2
    return d2.sqrt()


def _features(hp, X):
    h, a, b, r = hp.h.reshape(-1, hp.bump_dims), hp.a, hp.b, hp.r
    out = torch.zeros(X.shape[0], hp.n1, dtype=torch.float64, device=X.device)
    for i in range(hp.n1):
        for j in range(hp.n2):
            q = i * hp.n2 + j
            t = sum((X[:, k] - h[q, k]) ** 2 for k in range(hp.bump_dims)) / r[q] ** 2
            inside = t < 1
            t = torch.where(inside, t, torch.zeros_like(t))
            out[:, i] += torch.where(inside, a[q] * torch.exp(b[q] * (1 - 1 / (1 - t))), torch.zeros_like(t))
    return out


def _cov(hp, A, B):
    """C_y(A, B) without the noise term."""
    sparse = hp.s0 * _wendland(_scaled_dist(A, B, hp.r0)) + _features(hp, A) @ _features(hp, B).T
    if hp.core_kind == 0:
        return hp.core_var * _wendland(_scaled_dist(A, B, hp.core_radius)) * sparse
    ph_s = torch.as_tensor(hp.phi_sigma, device=A.device)
    ph_S = torch.as_tensor(hp.phi_Sigma, device=A.device)
    d = A.shape[1]
    sa, sb = hp.sigma0 * torch.exp(A @ ph_s), hp.sigma0 * torch.exp(B @ ph_s)
    Sa, Sb = hp.Sigma0 * torch.exp(A @ ph_S), hp.Sigma0 * torch.exp(B @ ph_S)
    avg = (Sa[:, None] + Sb[None, :]) / 2
    t = _scaled_dist(A, B, [1.0] * d) / avg.sqrt() * math.sqrt(3.0)
    return sa[:, None] * sb[None, :] * (Sa[:, None] * Sb[None, :]) ** (d / 4) / avg ** (d / 2) * (1 + t) * torch.exp(-t) * sparse


def _cov_z(hp, X):
    n = X.shape[0]
    C = torch.empty(n, n, dtype=torch.float64, device=X.device)
    for r in range(0, n, 2048):
        C[r:r + 2048] = _cov(hp, X[r:r + 2048], X)
    C.diagonal().add_(hp.noise_var)
    return C


def _dense(hp, X, resid, Xt, mu, want_var=False):
    """(log-likelihood, predictive mean or None, predictive variance or None) through a dense Cholesky."""
    L = torch.linalg.cholesky(_cov_z(hp, X))
    y = torch.linalg.solve_triangular(L, resid[:, None], upper=False)
    ll = -L.diagonal().log().sum() - 0.5 * (y * y).sum() - 0.5 * X.shape[0] * math.log(2 * math.pi)
    mean = var = None
    if Xt is not None and not want_var:
        alpha = torch.linalg.solve_triangular(L.T, y, upper=True)
        mean = torch.cat([(_cov(hp, Xt[r:r + 2048], X) @ alpha)[:, 0] for r in range(0, Xt.shape[0], 2048)])
        mean = mean if mu is None else mean + mu
    if want_var:
        V = torch.linalg.solve_triangular(L, _cov(hp, X, Xt), upper=False)
        prior = torch.cat([_cov(hp, Xt[k:k + 1], Xt[k:k + 1])[0] for k in range(Xt.shape[0])])
        var = prior - (V * V).sum(0)
    return ll, mean, var


def exact(case, seed):
    if case["kind"] == "serving":
        sets, reqs = _serving_workload(case, seed)
        outs = []
        for i, th, xt in reqs:
            if len(sets[i].X) > EXACT_MAX_REQUEST_N:
                outs.append(None)
                continue
            ll, mean, _ = _dense(th, _dev(sets[i].X), _dev(sets[i].resid), None if xt is None else _dev(xt), None)
            outs.append(ll.reshape(1) if xt is None else mean)
        return outs
    if case["n"] * math.sqrt(case["B"]) > EXACT_MAX_N or case["m"] > 100000:
        return None
    w = _workload(case, seed)
    X, Xt = _dev(w.X), _dev(w.Xtest) if case["m"] else None
    if case["var"]:
        return {"variance": _dense(w.hyper, X, _dev(w.resid), Xt, None, want_var=True)[2]}
    res = [_dense(hp, X, _dev(r), Xt, _dev(w.mu_test) if case["m"] else None) for hp, r in zip(w.thetas, w.residuals)]
    out = {"loglik": torch.stack([r[0] for r in res])}
    if case["m"]:
        out["mean"] = [r[1] for r in res]
    return out
