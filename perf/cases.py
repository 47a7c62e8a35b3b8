"""Performance cases of the matrix-free GP library: what a user's program asks of its entry points, over the range of
sizes, dimensions, kernels, column counts and precisions that they take.

``listed()`` holds twelve fixed cases, ``draw(rng)`` gives further ones of the same ranges. ``prepare`` makes a case's
inputs on the GPU from a seed, ``run`` is one call as a user's program makes it, ``work`` what the call cannot do
without, ``exact`` its outputs in 64 bits by dense linear algebra that shares no code with the library.

The data follow the recipes of ``workloads``: points uniform in a box or standard normal, lengthscales log-spaced over
[0.3, 2] (0.2 or 0.5 in the two-dimensional and the D = 4 recipes), targets that are sums of sinusoids with noise, and
standard normal right-hand sides. Solves draw a noise variance that leaves the system well enough conditioned for its
float32 solution to be determined to a few units in the fifth digit.
"""
import math

import numpy as np
import torch

import paper_2605_17898_gb300 as lgp

RBF, MATERN52, MATERN12, MATERN32 = 0, 1, 2, 3
KINDS = (RBF, MATERN52, MATERN12, MATERN32)
AUTO, FP32, BF16, F16 = lgp.LGP_PREC_AUTO, lgp.LGP_PREC_FP32, lgp.LGP_PREC_SPLIT_BF16, lgp.LGP_PREC_SPLIT_F16


def _product(name, n, d, kind, t, prec=AUTO, box="unit", lo=0.3, hi=2.0):
    c = {"op": "product", "n": n, "d": d, "kind": kind, "t": t, "prec": prec, "box": box, "lo": lo, "hi": hi}
    return {"name": name, **c} if name else c


def _derivatives(name, n, d, kind, t):
    c = {"op": "derivatives", "n": n, "d": d, "kind": kind, "t": t, "box": "pm1", "lo": 0.3, "hi": 2.0}
    return {"name": name, **c} if name else c


def _solve(name, n, d, kind, t, noise, rank=0, box="pm1", lo=0.3, hi=2.0):
    c = {"op": "solve", "n": n, "d": d, "kind": kind, "t": t, "noise": noise, "rank": rank, "box": box, "lo": lo, "hi": hi}
    return {"name": name, **c} if name else c


def _fit(name, n, d, kind, probes, noise):
    c = {"op": "fit", "n": n, "d": d, "kind": kind, "probes": probes, "noise": noise, "box": "pm1", "lo": 0.3, "hi": 2.0}
    return {"name": name, **c} if name else c


def _predict(name, n, m, d, kind, probes, noise):
    c = {"op": "predict", "n": n, "m": m, "d": d, "kind": kind, "probes": probes, "noise": noise, "box": "pm1", "lo": 0.3,
         "hi": 2.0}
    return {"name": name, **c} if name else c


def _batch(name, n_gp, n_lo, n_hi, t, noise):
    c = {"op": "batch", "n_gp": n_gp, "n_lo": n_lo, "n_hi": n_hi, "t": t, "noise": noise, "box": "pm1", "lo": 0.3, "hi": 2.0}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest call: one product of a thousand-point problem, where launches and latency count
        _product("product_1k_rbf_t1", 1024, 2, RBF, 1, lo=0.2, hi=0.2),
        # the headline shape: the float32 product of one column, RBF, D = 4, at the largest tabulated size
        _product("product_50k_rbf_t1", 50000, 4, RBF, 1, lo=0.5, hi=0.5),
        # an odd size and column count on the float32 path, for the kernel that is not smooth at zero distance
        _product("product_4099_m12_t5", 4099, 5, MATERN12, 5),
        # a block product of a mid-size problem on the tensor cores, low dimension
        _product("product_20k_m52_t16", 20000, 3, MATERN52, 16, box="normal"),
        # the largest: the block product of the training workload
        _product("product_100k_m52_t32", 100000, 8, MATERN52, 32, box="pm1"),
        # the bfloat16 split on request, an odd size
        _product("product_30011_rbf_bf16", 30011, 6, RBF, 32, prec=BF16, box="pm1"),
        # the derivative blocks of the covariance, for callers that assemble their own gradients
        _derivatives("derivatives_6k_m52_t4", 6000, 8, MATERN52, 4),
        # one small GP solved for its targets: a CG loop bound by launches
        _solve("solve_1k_rbf_t1", 1024, 2, RBF, 1, 0.25, box="unit", lo=0.2, hi=0.2),
        # one training step (likelihood and gradient, forward and backward) of a small and of a large problem
        _fit("fit_2k_rbf_t16", 2000, 8, RBF, 15, 0.1),
        _fit("fit_20k_m52_t32", 20000, 8, MATERN52, 31, 0.1),
        # predictive mean and variance at test points
        _predict("predict_8k_m52", 8000, 1000, 8, MATERN52, 31, 0.1),
        # many independent GPs of uneven size in one call
        _batch("batch_48_t8", 48, 200, 2000, 8, 0.25),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["product", "product", "product", "derivatives", "solve", "fit", "predict", "batch"])
    kind = rng.choice(KINDS)
    if op == "product":
        t = rng.choice([1, 1, 2, 3, 4, 6, 8, 12, 16, 16, 32, 32])
        prec = rng.choice([AUTO, AUTO, F16, BF16, FP32]) if t in (16, 32) else AUTO
        slow = prec == FP32 and t > 8
        n = _log_int(rng, 500, 20000 if slow else 100000)
        return _product("", n, rng.randint(1, 8), kind, t, prec, box=rng.choice(["unit", "pm1", "normal"]))
    if op == "derivatives":
        return _derivatives("", _log_int(rng, 500, 12000), rng.randint(1, 8), kind, rng.choice([1, 2, 4, 8, 16]))
    noise = rng.choice([0.1, 0.15, 0.25])
    d = rng.randint(6, 8)
    if op == "solve":
        t = rng.choice([1, 1, 2, 4, 8, 16, 32])
        return _solve("", _log_int(rng, 500, 12000), d, kind, t, noise, rank=rng.choice([0, 0, 0, 16]))
    if op == "fit":
        return _fit("", _log_int(rng, 500, 15000), d, kind, rng.choice([7, 15, 15, 31, 31]), noise)
    if op == "predict":
        return _predict("", _log_int(rng, 500, 8000), _log_int(rng, 20, 2000), d, kind, rng.choice([15, 31]), noise)
    lo = _log_int(rng, 150, 500)
    return _batch("", rng.randint(8, 60), lo, lo * rng.randint(2, 5), rng.choice([1, 2, 4, 8]), max(noise, 0.15))


# ---------------------------------------------------------------------------------------------- inputs


def _points(g, n, d, box):
    if box == "normal":
        return torch.randn((n, d), generator=g, device="cuda")
    x = torch.rand((n, d), generator=g, device="cuda")
    return 2.0 * x - 1.0 if box == "pm1" else x


def _lengthscales(d, lo, hi):
    return np.linspace(math.log(lo), math.log(hi), d) if d > 1 else np.array([0.5 * (math.log(lo) + math.log(hi))])


def _hyper(case, d, kind):
    return lgp.Hyper(kind, _lengthscales(d, case["lo"], case["hi"]).astype(np.float32), 0.0,
                     float(np.float32(math.log(case.get("noise", 0.01)))))


def _targets(g, x):
    f = math.pi * (torch.arange(x.shape[1], device="cuda") + 2) / 2.0
    return torch.sin(x * f).sum(1) + 0.05 * torch.randn(x.shape[0], generator=g, device="cuda")


def _batch_shapes(case, seed):
    r = np.random.default_rng(seed)
    n = np.exp(r.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]), case["n_gp"]))
    return [(int(round(v)), 6 + i % 3, RBF if i % 2 == 0 else MATERN52) for i, v in enumerate(n)]


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    op = case["op"]
    s = {"op": op, "case": dict(case), "seed": int(seed) & 0x7FFFFFFF}
    if op == "batch":
        # the shapes belong to the case, the data to the seed: a program solves the same set of models again
        shapes = _batch_shapes(case, 5)
        s["X"] = [_points(g, n, d, case["box"]) for n, d, _ in shapes]
        s["hyp"] = [_hyper(case, d, kind) for _, d, kind in shapes]
        s["B"] = [torch.randn((n, case["t"]), generator=g, device="cuda") for n, _, _ in shapes]
        for x, b in zip(s["X"], s["B"]):
            b[:, 0] = _targets(g, x)
        return s
    s["X"] = _points(g, case["n"], case["d"], case["box"])
    s["hyp"] = _hyper(case, case["d"], case["kind"])
    if op in ("product", "derivatives", "solve"):
        s["V"] = torch.randn((case["n"], case["t"]), generator=g, device="cuda")
    if op == "solve":
        s["V"][:, 0] = _targets(g, s["X"])
    if op in ("fit", "predict"):
        s["y"] = _targets(g, s["X"])
    if op == "fit":
        h = s["hyp"]
        s["params"] = [torch.tensor(h.log_lengthscale), torch.tensor(h.log_outputscale), torch.tensor(h.log_noise)]
        for p in s["params"]:
            p.requires_grad_(True)
    if op == "predict":
        s["Xs"] = _points(g, case["m"], case["d"], case["box"])
    return s


# ---------------------------------------------------------------------------------------------- the calls


def run(s):
    case, op = s["case"], s["op"]
    if op == "product":
        return lgp.lgp_kernel_matvec(s["X"], s["hyp"], s["V"], prec=case["prec"])
    if op == "derivatives":
        return lgp.lgp_kernel_matvec_grad(s["X"], s["hyp"], s["V"])
    if op == "solve":
        return lgp.lgp_cg_solve(s["X"], s["hyp"], s["V"], tol=1e-6, max_iter=2000, precond_rank=case["rank"])[0]
    if op == "fit":
        for p in s["params"]:
            p.grad = None
        lml = lgp.marginal_likelihood(s["X"], s["y"], *s["params"], kind=case["kind"], n_probes=case["probes"],
                                      seed=s["seed"], tol=1e-6, max_iter=2000)
        loss = -lml / case["n"]
        loss.backward()
        return {"loss": float(loss), "grads": [p.grad for p in s["params"]]}
    if op == "predict":
        mean, var, _, _ = lgp.lgp_predict(s["X"], s["y"], s["hyp"], s["Xs"], n_probes=case["probes"], seed=s["seed"], tol=1e-6,
                                          max_iter=2000)
        return {"mean": mean, "var": var}
    return lgp.lgp_batch_cg_solve(s["X"], s["hyp"], s["B"], tol=1e-6, max_iter=2000)[0]


# ---------------------------------------------------------------------------------------------- work

#: Arithmetic of one kernel entry beside its distance, and of its derivative factor.
_ENTRY = {RBF: 2, MATERN52: 7, MATERN12: 3, MATERN32: 5}


def _product_work(n, d, kind, t):
    """Each unordered pair's entry once (the covariance is symmetric), each entry times t columns."""
    return {"bytes": 4.0 * n * (d + 2 * t), "flops": 0.5 * n * (n + 1.0) * (3 * d + _ENTRY[kind]) + 2.0 * n * n * t}


def _iterations(case, n):
    """A floor of the CG iterations to a relative residual of 1e-6 (a mild fraction of what the data need)."""
    return max(1, int(10.0 * math.sqrt(1.0 + 0.002 * n / case["noise"])))


def work(case):
    op = case["op"]
    if op == "product":
        return _product_work(case["n"], case["d"], case["kind"], case["t"])
    if op == "derivatives":
        n, d, t = case["n"], case["d"], case["t"]
        return {"bytes": 4.0 * n * (d + t + (d + 2) * t),
                "flops": 0.5 * n * (n + 1.0) * (3 * d + 2 * _ENTRY[case["kind"]]) + 2.0 * n * n * t * (d + 1)}
    if op == "batch":
        flops = moved = 0.0
        for n, d, kind in _batch_shapes(case, 5):
            flops += _iterations(case, n) * _product_work(n, d, kind, case["t"])["flops"]
            moved += 4.0 * n * (d + 2 * case["t"])
        return {"bytes": moved, "flops": flops}
    n, d, kind = case["n"], case["d"], case["kind"]
    t = case["t"] if op == "solve" else case["probes"] + 1
    flops = _iterations(case, n) * _product_work(n, d, kind, t)["flops"]
    moved = 4.0 * n * (d + (2 * t if op == "solve" else 1))
    if op == "fit":
        flops += 0.5 * n * (n + 1.0) * (3 * d + 2 * _ENTRY[kind] + 2 * d) + 2.0 * n * n * t
    if op == "predict":
        flops += 2.0 * n * case["m"] * (3 * d + _ENTRY[kind] + 2 * t)
        moved += 4.0 * case["m"] * (d + 2)
    return {"bytes": moved, "flops": flops}


# ---------------------------------------------------------------------------------------------- 64-bit reference

_PRESCALE = {RBF: 1.0, MATERN52: math.sqrt(5.0), MATERN12: 1.0, MATERN32: math.sqrt(3.0)}


def _scaled(x, hyp):
    return x.double() * torch.exp(-torch.tensor(hyp.log_lengthscale, dtype=torch.float64, device="cuda")) * _PRESCALE[hyp.kind]


def _sqdist(a, b):
    r2 = torch.zeros((a.shape[0], b.shape[0]), dtype=torch.float64, device="cuda")
    for d in range(a.shape[1]):
        r2.add_((a[:, d, None] - b[None, :, d]).square_())
    return r2


def _entries(r2, hyp):
    """k of the prescaled squared distances."""
    s2 = math.exp(float(hyp.log_outputscale))
    if hyp.kind == RBF:
        return s2 * torch.exp(-0.5 * r2)
    r = torch.sqrt(r2)
    e = s2 * torch.exp(-r)
    if hyp.kind == MATERN12:
        return e
    return e * (1.0 + r) if hyp.kind == MATERN32 else e * (1.0 + r + r2 / 3.0)


def _psi(r2, hyp):
    """dk/dlog l_d = psi * (prescaled difference of coordinate d)^2."""
    s2 = math.exp(float(hyp.log_outputscale))
    if hyp.kind == RBF:
        return s2 * torch.exp(-0.5 * r2)
    r = torch.sqrt(r2)
    e = s2 * torch.exp(-r)
    if hyp.kind == MATERN12:
        return torch.where(r > 0, e / r.clamp_min(1e-300), torch.zeros_like(r))
    return e if hyp.kind == MATERN32 else e * (1.0 + r) / 3.0


def _cov(z, hyp):
    k = _entries(_sqdist(z, z), hyp)
    k.diagonal().add_(math.exp(float(hyp.log_noise)))
    return k


def _chunks(n, cols):
    step = max(1, min(n, int(2.5e8 / max(1, cols))))
    return [(i, min(n, i + step)) for i in range(0, n, step)]


def _exact_product(s):
    z, v, hyp = _scaled(s["X"], s["hyp"]), s["V"].double(), s["hyp"]
    out = math.exp(float(hyp.log_noise)) * v
    for i, j in _chunks(z.shape[0], z.shape[0]):
        out[i:j] += _entries(_sqdist(z[i:j], z), hyp) @ v
    return out


def _exact_derivatives(s):
    z, w, hyp = _scaled(s["X"], s["hyp"]), s["V"].double(), s["hyp"]
    n, d = z.shape
    out = torch.zeros((d + 2, n, w.shape[1]), dtype=torch.float64, device="cuda")
    for i, j in _chunks(n, n):
        r2 = _sqdist(z[i:j], z)
        psi = _psi(r2, hyp)
        for p in range(d):
            out[p, i:j] = (psi * (z[i:j, p, None] - z[None, :, p]).square()) @ w
        out[d, i:j] = _entries(r2, hyp) @ w
    out[d + 1] = math.exp(float(hyp.log_noise)) * w
    return out


def _rademacher(seed, n, m):
    """The documented probe stream: bit 63 of splitmix64(seed XOR (column << 32 | row))."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) ^ ((np.arange(m, dtype=np.uint64)[None, :] << np.uint64(32)) | np.arange(n, dtype=np.uint64)[:, None])
        z = z + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return torch.tensor(np.where(z >> np.uint64(63), -1.0, 1.0), device="cuda")


def _quadratic_logs(k, z, steps):
    """z_c^T log(K) z_c for every column by Lanczos with full reorthogonalisation."""
    n, m = z.shape
    steps = min(steps, n)
    norm = z.norm(dim=0)
    q = torch.zeros((m, steps, n), dtype=torch.float64, device="cuda")
    a = torch.zeros((m, steps), dtype=torch.float64, device="cuda")
    b = torch.zeros((m, steps), dtype=torch.float64, device="cuda")
    cur = (z / norm).T.contiguous()
    for i in range(steps):
        q[:, i] = cur
        w = (k @ cur.T).T
        a[:, i] = (w * cur).sum(1)
        for _ in range(2):
            c = torch.bmm(q[:, : i + 1], w[:, :, None])
            w = w - torch.bmm(c.transpose(1, 2), q[:, : i + 1])[:, 0]
        b[:, i] = w.norm(dim=1)
        cur = w / b[:, i, None].clamp_min(1e-300)
    t = torch.diag_embed(a) + torch.diag_embed(b[:, :-1], 1) + torch.diag_embed(b[:, :-1], -1)
    lam, vec = torch.linalg.eigh(t.cpu())
    g = (vec[:, 0].square() * torch.log(lam)).sum(1)
    return norm.square() * g.cuda()


def _exact_fit(s):
    x, hyp, case = s["X"], s["hyp"], s["case"]
    n, d = x.shape
    m = case["probes"]
    z = _scaled(x, hyp)
    k = _cov(z, hyp)
    rhs = torch.cat([s["y"].double()[:, None], _rademacher(s["seed"], n, m)], 1)
    u = torch.cholesky_solve(rhs, torch.linalg.cholesky(k))
    logdet = _quadratic_logs(k, rhs[:, 1:], 260).mean()
    lml = -0.5 * ((rhs[:, 0] * u[:, 0]).sum() + logdet + n * math.log(2.0 * math.pi))
    noise = math.exp(float(hyp.log_noise))
    # grad_p = sum_ij dK_p[i, j] W[i, j]
    left, right = 0.5 * u, torch.cat([u[:, :1], -rhs[:, 1:] / m], 1)
    g = torch.zeros(d + 2, dtype=torch.float64, device="cuda")
    for i, j in _chunks(n, n):
        w = left[i:j] @ right.T
        r2 = _sqdist(z[i:j], z)
        pw = _psi(r2, hyp) * w
        for p in range(d):
            g[p] += (pw * (z[i:j, p, None] - z[None, :, p]).square()).sum()
        g[d] += (_entries(r2, hyp) * w).sum()
    g[d + 1] = noise * (left * right).sum()
    g = -g.cpu() / n
    return {"loss": np.float64(-float(lml) / n), "grads": [g[:d], g[d], g[d + 1]]}


def _exact_predict(s):
    x, hyp, case = s["X"], s["hyp"], s["case"]
    z, zs = _scaled(x, hyp), _scaled(s["Xs"], hyp)
    ks = _entries(_sqdist(z, zs), hyp)
    probes = _rademacher(s["seed"], zs.shape[0], case["probes"])
    u = torch.cholesky_solve(torch.cat([s["y"].double()[:, None], ks @ probes], 1), torch.linalg.cholesky(_cov(z, hyp)))
    s2 = math.exp(float(hyp.log_outputscale))
    return {"mean": ks.T @ u[:, 0], "var": s2 - (probes * (ks.T @ u[:, 1:])).mean(1)}


def exact(case, seed):
    s = prepare(case, seed)
    op = case["op"]
    if op == "product":
        return _exact_product(s)
    if op == "derivatives":
        return _exact_derivatives(s)
    if op == "fit":
        return _exact_fit(s)
    if op == "predict":
        return _exact_predict(s)
    if op == "solve":
        return torch.cholesky_solve(s["V"].double(), torch.linalg.cholesky(_cov(_scaled(s["X"], s["hyp"]), s["hyp"])))
    return [torch.cholesky_solve(b.double(), torch.linalg.cholesky(_cov(_scaled(x, h), h)))
            for x, h, b in zip(s["X"], s["hyp"], s["B"])]
