"""The workloads the solver is timed on: inputs, one pass through the public entry points, its
unavoidable work, and the same result in 64-bit torch without the library.

Inputs are synthetic spectra of the recipe in spectra/ (unit-mass Gaussian peaks on a 1-D grid,
sparse Gamma weights, shifted and noisy targets), drawn on the device from the seed alone so that
thousands of targets take milliseconds.  Every solve runs a fixed number of iterations (tol = 0, the
mode of the 500-iteration FP64 workload; with a tolerance a problem near it may stop one iteration
sooner or later on any change of rounding).  The n = 4096 batch runs the 20 iterations that take it
to the 1e-5 tolerance.
"""
import math
import random

import numpy as np
import torch

from paper_2504_04609_gb300 import otlm as api

DEV = "cuda"
TINY32 = 1.17549435e-38
# tile shapes otlm_tune_ragged reports for sizes 256..4096 (otlm_config form)
RAGGED_CTA, RAGGED_ROWS = 512, [1, 1, 1, 1, 2, 2, 2, 2, 3, 3, 3, 3, 3, 3, 3, 3]


def _solve(name, entry, B, n, k, eps, datafit, penalty, alpha, iters, **kw):
    c = dict(kind="solve", entry=entry, precision="fp32", B=B, n=n, k=k, nnz=5, eps=eps, lam=1.0, datafit=datafit,
             penalty=penalty, alpha=alpha, beta=0.0, mm_steps=1, iters=iters, single_until=0.0, cost="sq",
             grid="uniform")
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one spectrum in FP64, 500 iterations: a person fitting one measurement to full accuracy
        _solve("fp64_single_n200", "solve", 1, 200, 10, 1e-2, "kl", "l2sq", 1e-3, 500, precision="fp64", nnz=3),
        # the smallest call: a few short spectra from inside a host framework that owns the memory
        _solve("noalloc_b8_n256", "noalloc", 8, 256, 16, 1e-2, "kl", "l1", 1e-2, 10),
        # an ordinary FP32 batch of spectra sharing one dictionary
        _solve("fp32_b1024_n1024", "solve", 1024, 1024, 64, 5e-3, "kl", "l1", 1e-2, 50),
        # the same batch on a tensor-core handle
        _solve("tc_b1024_n1024", "solve", 1024, 1024, 64, 5e-3, "kl", "l1", 1e-2, 50, precision="bf16tc"),
        # the largest batch, to convergence: throughput serving (the benchmark's workload)
        _solve("tc_b4096_n4096", "solve", 4096, 4096, 128, 1e-2, "l2", "l2sq", 1e-3, 20, precision="bf16tc",
               single_until=3e-5),
        # one target on a fine grid
        _solve("tc_single_n16384", "solve", 1, 16384, 128, 1e-2, "l2", "l2sq", 1e-3, 20, precision="bf16tc"),
        # a dense, non-symmetric, truncated cost shared by a batch (muonic X-ray form: TV + l1)
        _solve("dense_b256_n1024", "cost", 256, 1024, 64, 2e-2, "tv", "l1", 1e-2, 20, precision="bf16tc", cost="dense"),
        # uneven batch: every problem its own grid, dictionary and eps
        dict(name="ragged_b800", kind="ragged", B=800, n_lo=256, n_hi=4096, k_lo=8, k_hi=128, nnz=5, eps_lo=2e-3,
             eps_hi=5e-2, lam=1.0, datafit="tv", penalty="l1", alpha=1e-2, iters=20, sizes=4),
        # banded cost and sparse dictionary at the scalability test's largest size (OT ridge)
        dict(name="banded_b32_n100000", kind="banded", B=32, n=100000, k=10000, hw=9, eps=1e-3, lam=1.0, datafit="l2",
             penalty="l2sq", alpha=1e-3, iters=40),
        # one optimiser step of the warm-start network (forward, backward, update)
        dict(name="ws_train_b512", kind="train", B=512, n=2048, k=64, width=512, lr=2e-5),
        # the network's prediction for a serving batch
        dict(name="ws_predict_b4096", kind="predict", B=4096, n=2048, k=64, width=512, eps=5e-3),
        # objective and duality gap of solved states in FP64: the judge of a result's quality
        dict(name="objective_fp64_b16_n512", kind="objective", B=16, n=512, k=32, nnz=5, eps=1e-2, lam=1.0,
             datafit="l2", penalty="l2sq", alpha=1e-3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: any entry point, sizes log-uniform (odd ones included)."""
    kind = rng.choice(["solve", "solve", "solve", "tc", "tc", "tc", "fp64", "noalloc", "host", "cost", "ragged",
                       "banded", "train", "gradients", "predict", "objective"])
    eps = round(math.exp(rng.uniform(math.log(5e-3), math.log(5e-2))), 6)
    datafit = rng.choice(["kl", "l2", "tv", "poisson", "l2"])
    penalty = rng.choice(["l1", "l2sq", "l2sq", "elastic", "none"])
    alpha = 0.0 if penalty == "none" else (1e-3 if penalty == "l2sq" else 1e-2)
    kw = dict(beta=1e-3 if penalty == "elastic" else 0.0, mm_steps=rng.choice([1, 1, 1, 2]),
              grid=rng.choice(["uniform", "uniform", "warped"]), cost=rng.choice(["sq", "sq", "sq", "abs"]))
    if kind == "solve":
        n = _log(rng, 200, 3000)
        return _solve(None, "solve", _log(rng, 1, min(1500, 1.2e9 / n ** 2)), n, _log(rng, 8, 128), eps, datafit, penalty,
                      alpha, 20, **kw)
    if kind == "tc":
        n = _log(rng, 250, 8000)
        return _solve(None, "solve", _log(rng, 1, min(4000, 8e9 / n ** 2)), n, _log(rng, 8, 128), max(eps, 1e-2), datafit,
                      penalty, alpha, 20, precision="bf16tc", **kw)
    if kind == "fp64":
        return _solve(None, "solve", _log(rng, 1, 12), _log(rng, 100, 500), _log(rng, 5, 40), eps, datafit, penalty, alpha,
                      20, precision="fp64", **kw)
    if kind in ("noalloc", "host"):
        n = _log(rng, 100, 1500)
        if kind == "noalloc":
            kw.update(mm_steps=1, cost="sq", beta=0.0)
            if penalty == "elastic":
                penalty = "l1"
        return _solve(None, kind, _log(rng, 1, 64), n, _log(rng, 5, 64), eps, datafit, penalty, alpha, 15, **kw)
    if kind == "cost":
        n = _log(rng, 200, 1500)
        kw.update(cost="dense", mm_steps=1)
        return _solve(None, "cost", _log(rng, 1, 300), n, _log(rng, 8, 100), max(eps, 2e-2), "tv", "l1", 1e-2, 15,
                      precision=rng.choice(["fp32", "bf16tc"]), **dict(kw, beta=0.0))
    if kind == "ragged":
        lo = _log(rng, 64, 600)
        return dict(kind="ragged", B=_log(rng, 20, 400), n_lo=lo, n_hi=min(4096, lo * rng.randint(2, 16)), k_lo=5,
                    k_hi=_log(rng, 16, 128), nnz=5, eps_lo=2e-3, eps_hi=5e-2, lam=1.0, datafit=rng.choice(["tv", "l2", "kl"]),
                    penalty="l1", alpha=1e-2, iters=15, sizes=rng.randrange(1000))
    if kind == "banded":
        n = _log(rng, 2000, 100000)
        return dict(kind="banded", B=_log(rng, 1, 32), n=n, k=n // 10, hw=rng.choice([4, 9, 9, 15, 20]), eps=1e-3,
                    lam=1.0, datafit=rng.choice(["l2", "tv"]), penalty="l2sq", alpha=1e-3, iters=20)
    if kind in ("train", "gradients"):
        return dict(kind=kind, B=_log(rng, 16, 512), n=_log(rng, 200, 2048), k=_log(rng, 8, 100),
                    width=rng.choice([128, 200, 256, 512]), lr=2e-5)
    if kind == "predict":
        return dict(kind="predict", B=_log(rng, 1, 4096), n=_log(rng, 200, 2048), k=_log(rng, 8, 100),
                    width=rng.choice([128, 200, 256, 512]), eps=5e-3)
    return dict(kind="objective", B=_log(rng, 1, 16), n=_log(rng, 100, 512), k=_log(rng, 5, 40), nnz=5, eps=1e-2, lam=1.0,
                datafit="l2", penalty="l2sq", alpha=1e-3)


# ---- inputs --------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _round(a, dtype):
    """Round to the solver's type; float32 subnormals become 0 (the kernels flush them)."""
    a = a.to(dtype)
    return a * (a.abs() >= TINY32) if dtype == torch.float32 else a


def _grid(n, kind):
    u = torch.arange(n, dtype=torch.float64, device=DEV) / (n - 1)
    return u + 0.1 / (2 * math.pi) * torch.sin(2 * math.pi * u) if kind == "warped" else u


def _peaks(x, mu, sig):
    """Unit-mass peaks: x [n], mu and sig [...] -> [..., n]."""
    p = torch.exp(-0.5 * ((x - mu[..., None]) / sig[..., None]) ** 2)
    return p / p.sum(-1, keepdim=True)


def _spectra(g, x, B, k, nnz):
    """Dictionary [n][k] and targets [B][n] in float64."""
    nnz = min(nnz, k)
    rand = lambda *s: torch.rand(*s, generator=g, device=DEV, dtype=torch.float64)  # noqa: E731
    randn = lambda *s: torch.randn(*s, generator=g, device=DEV, dtype=torch.float64)  # noqa: E731
    mu, sig = 0.1 + 0.8 * rand(k), torch.exp(math.log(0.02) + 0.3 * randn(k))
    D = _peaks(x, mu, sig).T.contiguous()
    y = torch.zeros(B, x.shape[0], dtype=torch.float64, device=DEV)
    idx = rand(B, k).argsort(dim=1)[:, :nnz]
    for q in range(nnz):
        wq = -torch.log(rand(B).clamp_min(1e-12)) - torch.log(rand(B).clamp_min(1e-12))  # Gamma(2, 1)
        y += wq[:, None] * _peaks(x, mu[idx[:, q]] + 0.01 * randn(B), sig[idx[:, q]])
    y *= (1.0 + 0.01 * randn(B, x.shape[0])).clamp_min(0.0)
    return D, y


def _dense_cost(x):
    """Non-stationary, truncated cost: 0.5 (g_i - g_j)^2 / g_i^2, +inf beyond 0.3."""
    gx = x + 0.25
    C = 0.5 * (gx[:, None] - gx[None, :]) ** 2 / gx[:, None] ** 2
    return torch.where((x[:, None] - x[None, :]).abs() > 0.3, torch.full_like(C, math.inf), C)


def _cold(D, y):
    return y.double().sum(-1, keepdim=True) / (D.shape[1] * D.double().sum(0))


def _solve_inputs(c, seed):
    dt = torch.float64 if c["precision"] == "fp64" else torch.float32
    g = _gen(seed)
    x = _grid(c["n"], c["grid"])
    D, y = _spectra(g, x, c["B"], c["k"], c["nnz"])
    D, y = _round(D, dt), _round(y, dt)
    if c["cost"] == "dense":
        cost = _round(_dense_cost(x), dt)
    else:
        cost = _round(x * (0.1 if c["cost"] == "abs" else 1.0), dt)
    return cost, D, y, _cold(D, y).to(dt)


def _banded_inputs(c, seed):
    n, k, hw, B = c["n"], c["k"], c["hw"], c["B"]
    g = _gen(seed)
    i = np.arange(n)
    Cd = np.full((2 * hw + 1, n), np.inf, np.float32)
    for d in range(2 * hw + 1):
        ok = (i + d - hw >= 0) & (i + d - hw < n)
        Cd[d, ok] = 0.01 * abs(d - hw)
    mu = np.arange(k) * (n / k)
    rows = np.floor(mu).astype(np.int64)[:, None] + np.arange(-10, 12)[None, :]
    z = (rows - mu[:, None]) / 2.0
    ok = (rows >= 0) & (rows < n) & (np.abs(z) <= 5.0)
    col_ptr = np.concatenate([[0], np.cumsum(ok.sum(1))]).astype(np.int32)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)  # noqa: E731
    # skew-normal components on the sample grid, each within +-24 bins of its mean
    rand = lambda *s: torch.rand(*s, generator=g, device=DEV, dtype=torch.float64)  # noqa: E731
    randn = lambda *s: torch.randn(*s, generator=g, device=DEV, dtype=torch.float64)  # noqa: E731
    m, s, a, gam = n * rand(B, k), (2.0 + 0.2 * randn(B, k)).abs(), (1.0 + 0.2 * randn(B, k)).abs() + 0.01, 2 * randn(B, k)
    one = 2.0 ** 36  # fixed point: the order of the atomic additions leaves no trace
    y = ((0.002 * randn(B, n)).abs() * one).long()
    for o in range(-24, 25):
        r = m.floor() + o
        zz = (r - m) / s
        v = a * 2.0 / s * torch.exp(-0.5 * zz * zz) / math.sqrt(2 * math.pi) * 0.5 * torch.erfc(-gam * zz / math.sqrt(2.0))
        inside = (r >= 0) & (r < n)
        y.scatter_add_(1, r.clamp(0, n - 1).long(), (v * inside * one).long())
    y = y.double() / one
    return dict(Cd=t(Cd), col_ptr=t(col_ptr), row_idx=t(rows[ok].astype(np.int32)), val=t(np.exp(-0.5 * z[ok] ** 2).astype(np.float32)),
                y=_round(y, torch.float32), rows=t(np.where(ok, rows, 0)), vals=t(np.where(ok, np.exp(-0.5 * z ** 2), 0.0).astype(np.float32)))


def _banded_w0(c, d):
    return (d["y"].double().sum(1, keepdim=True) / (c["k"] * d["vals"].double().sum(1))).float()


def _net_inputs(c, seed):
    n, k, H, B = c["n"], c["k"], c["width"], c["B"]
    g = _gen(seed)
    _, y = _spectra(g, _grid(n, "uniform"), B, k, 5)
    y = _round(y, torch.float32)
    dims = [n + 1, H, H, H, n + k]
    parts = []
    for a, b in zip(dims[:-1], dims[1:]):
        lim = math.sqrt(6.0 / (a + b))
        parts.append(lim * (2 * torch.rand(a * b, generator=g, device=DEV) - 1))
        parts.append(0.01 * torch.randn(b, generator=g, device=DEV))
    mean = torch.cat([-5.0 * torch.rand(n, generator=g, device=DEV), -1.0 - torch.rand(k, generator=g, device=DEV)])
    std = 0.5 + torch.rand(n + k, generator=g, device=DEV)
    tgt = mean + std * torch.randn(B, n + k, generator=g, device=DEV)
    tgt[:, :n] = torch.where(y > 0, tgt[:, :n], torch.full_like(y, -math.inf))  # bins without mass are masked
    return y, torch.cat(parts), mean, std, tgt, dims


def _stream():
    return torch.cuda.current_stream().cuda_stream


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "solve":
        cost, D, y, w0 = _solve_inputs(c, seed)
        s = dict(c=c, cost=cost, D=D, y=y, w0=w0)
        if c["entry"] == "host":
            pin = lambda t: t.cpu().pin_memory()  # noqa: E731
            s = dict(c=c, cost=pin(cost), D=pin(D), y=pin(y), w0=pin(w0))
            new = lambda t: torch.empty_like(t, pin_memory=True)  # noqa: E731
            s["iters"], s["status"] = (torch.empty(c["B"], dtype=torch.int32, pin_memory=True) for _ in range(2))
        else:
            new = torch.empty_like
            s["iters"], s["status"] = (torch.empty(c["B"], dtype=torch.int32, device=DEV) for _ in range(2))
        s["w"], s["g"], s["t"] = new(s["w0"]), new(s["y"]), new(s["y"])
        if c["entry"] != "noalloc":
            s["h"] = api.Handle(c["n"], c["k"], c["B"], c["precision"], c["datafit"], c["penalty"], c["iters"], 0.0,
                                poll_every=8, stream=_stream(), beta=c["beta"], mm_steps=c["mm_steps"],
                                bf16_single_until=c["single_until"], cost="sq" if c["cost"] == "dense" else c["cost"])
        return s
    if kind == "ragged":
        r, g, probs = random.Random(c["sizes"]), _gen(seed), []  # sizes and eps belong to the case
        for _ in range(c["B"]):
            n, k = r.randint(c["n_lo"], c["n_hi"]), r.randint(c["k_lo"], c["k_hi"])
            x = _grid(n, "uniform")
            D, y = _spectra(g, x, 1, k, c["nnz"])
            probs.append(dict(n=n, k=k, eps=math.exp(r.uniform(math.log(c["eps_lo"]), math.log(c["eps_hi"]))),
                              x=_round(x, torch.float32), D=_round(D, torch.float32), y=_round(y[0], torch.float32)))
        n, k = np.array([p["n"] for p in probs], np.int32), np.array([p["k"] for p in probs], np.int32)
        off = lambda a: torch.from_numpy(np.concatenate([[0], np.cumsum(a.astype(np.int64))[:-1]])).to(DEV)  # noqa: E731
        cat = lambda key: torch.cat([p[key].reshape(-1) for p in probs])  # noqa: E731
        eps = torch.tensor([p["eps"] for p in probs], dtype=torch.float32, device=DEV)
        rb = api.RaggedBatch(len(probs), torch.from_numpy(n).to(DEV), torch.from_numpy(k).to(DEV), eps, off(n),
                             off(n.astype(np.int64) * k), off(k), cat("x"), cat("D"), cat("y"))
        w0 = torch.cat([_cold(p["D"], p["y"]).float().reshape(-1) for p in probs])
        h = api.Handle(int(n.max()), int(k.max()), len(probs), "fp32", c["datafit"], c["penalty"], c["iters"], 0.0, 8,
                       stream=_stream(), ragged_cta=RAGGED_CTA, ragged_rows_log2=RAGGED_ROWS)
        i32 = lambda: torch.empty(len(probs), dtype=torch.int32, device=DEV)  # noqa: E731
        return dict(c=c, h=h, rb=rb, sizes=(n, k), w0=w0, w=torch.empty_like(w0), g=torch.empty_like(rb.y),
                    t=torch.empty_like(rb.y), iters=i32(), err=torch.empty(len(probs), device=DEV), status=i32())
    if kind == "banded":
        d = _banded_inputs(c, seed)
        h = api.Handle(64, 8, c["B"], "fp32", c["datafit"], c["penalty"], c["iters"], 0.0, 8, stream=_stream())
        i32 = lambda: torch.empty(c["B"], dtype=torch.int32, device=DEV)  # noqa: E731
        w0 = _banded_w0(c, d)
        return dict(c=c, h=h, d=d, w0=w0, w=torch.empty_like(w0), g=torch.empty_like(d["y"]), t=torch.empty_like(d["y"]),
                    iters=i32(), status=i32())
    if kind in ("train", "gradients", "predict"):
        y, p, mean, std, tgt, _ = _net_inputs(c, seed)
        net = api.WarmStart(c["n"], c["k"], c["width"], c["B"], stream=_stream())
        net.set_params(p)
        net.set_normalization(mean, std)
        s = dict(c=c, net=net, y=y, tgt=tgt, keep=(p, mean, std))
        if kind == "predict":
            s.update(cold=y.sum(1, keepdim=True) / c["k"] * torch.ones(1, c["k"], device=DEV), g0=torch.empty_like(y),
                     w0=torch.empty(c["B"], c["k"], device=DEV))
        else:
            s.update(out=torch.empty_like(p), loss=torch.empty(1, device=DEV))
        torch.cuda.synchronize()
        return s
    # objective: a state some iterations into the solve
    c = _solve(None, "solve", c["B"], c["n"], c["k"], c["eps"], c["datafit"], c["penalty"], c["alpha"], 15, precision="fp64")
    cost, D, y, w0 = _solve_inputs(c, seed)
    w, g, _ = _iterate(c, cost, D, y, w0, 15)
    h = api.Handle(c["n"], c["k"], c["B"], "fp64", c["datafit"], c["penalty"], 1, 0.0, 8, stream=_stream())
    out = [torch.empty(c["B"], dtype=torch.float64, device=DEV) for _ in range(2)]
    return dict(c=dict(c, kind="objective"), h=h, cost=cost, D=D, y=y, w=w.contiguous(), g=g.contiguous(), out=out)


def run(s):
    c = s["c"]
    kind = c["kind"]
    if kind == "solve":
        s["w"].copy_(s["w0"])
        s["g"].zero_()
        args = (s["cost"], s["D"], s["y"], c["eps"], c["lam"], c["alpha"])
        if c["entry"] == "noalloc":
            rc = api.solve_noalloc(*args, c["datafit"], c["penalty"], c["iters"], 0.0, s["w"], s["g"], s["t"], s["iters"],
                                   None, s["status"], _stream())
            if rc != api.OTLM_OK:
                raise RuntimeError("otlm_solve_noalloc: %d" % rc)
        else:
            call = {"solve": s["h"].solve, "cost": s["h"].solve_cost, "host": s["h"].solve_host}[c["entry"]]
            call(*args, s["w"], s["g"], s["t"], s["iters"], None, s["status"])
        return dict(w=s["w"], g=s["g"], t=s["t"], iters=s["iters"], status=s["status"])
    if kind == "ragged":
        s["w"].copy_(s["w0"])
        s["g"].zero_()
        s["h"].solve_ragged(s["rb"], c["lam"], c["alpha"], s["w"], s["g"], s["t"], s["iters"], s["err"], s["status"])
        return dict(w=s["w"], g=s["g"], t=s["t"], iters=s["iters"], status=s["status"])
    if kind == "banded":
        d = s["d"]
        s["w"].copy_(s["w0"])
        s["g"].zero_()
        s["h"].solve_banded(d["Cd"], c["hw"], d["col_ptr"], d["row_idx"], d["val"], d["y"], c["eps"], c["lam"], c["alpha"],
                            s["w"], s["g"], s["t"], s["iters"], None, s["status"])
        return dict(w=s["w"], g=s["g"], t=s["t"], iters=s["iters"], status=s["status"])
    if kind == "train":
        s["net"].train_step(s["y"], s["tgt"], c["lr"], 1e-4, s["loss"])
        s["net"].get_params(s["out"])
        return dict(params=s["out"], loss=s["loss"])
    if kind == "gradients":
        s["net"].gradients(s["y"], s["tgt"], s["out"], s["loss"])
        return dict(grad=s["out"], loss=s["loss"])
    if kind == "predict":
        s["net"].predict(s["y"], c["eps"], s["cold"], s["g0"], s["w0"])
        return dict(g0=s["g0"], w0=s["w0"])
    s["h"].objective(s["cost"], s["D"], s["y"], c["eps"], c["lam"], c["alpha"], s["w"], s["g"], *s["out"])
    return dict(primal=s["out"][0], dual=s["out"][1])


def work(case):
    """Inputs read once, outputs written once; operations: the dictionary contractions of every
    iteration and about 40 per bin and iteration for the two applies and the datafit step (a grid
    cost has no matrix entries of its own); a dense cost adds its two products."""
    c, kind = case, case["kind"]
    if kind == "solve":
        B, n, k, E = c["B"], c["n"], c["k"], 8 if c["precision"] == "fp64" else 4
        flops = c["iters"] * B * (4.0 * n * k * c["mm_steps"] + 40.0 * n + (4.0 * n * n if c["cost"] == "dense" else 0))
        return dict(bytes=E * (n * k + 3.0 * B * n + 2.0 * B * k + (n * n if c["cost"] == "dense" else n)), flops=flops)
    if kind == "ragged":
        n, k = (c["n_lo"] + c["n_hi"]) / 2, (c["k_lo"] + c["k_hi"]) / 2
        return dict(bytes=4 * c["B"] * (n * k + 4 * n + 2 * k), flops=c["iters"] * c["B"] * (4 * n * k + 40 * n))
    if kind == "banded":
        B, n, W = c["B"], c["n"], 2 * c["hw"] + 1
        return dict(bytes=4.0 * (W * n + 2 * 21 * c["k"] + 3 * B * n + 2 * B * c["k"]),
                    flops=c["iters"] * B * (n * (4.0 * W + 40) + 4 * 21.0 * c["k"]))
    if kind == "objective":
        B, n, k = c["B"], c["n"], c["k"]
        return dict(bytes=8.0 * (n * k + 2 * B * n + B * k), flops=B * (4.0 * n * n + 4.0 * n * k + 80.0 * n) + 2.0 * n * n)
    d = [c["n"] + 1, c["width"], c["width"], c["width"], c["n"] + c["k"]]
    macs = sum(a * b for a, b in zip(d[:-1], d[1:]))
    if kind == "predict":
        return dict(bytes=2.0 * macs + 4.0 * c["B"] * (d[0] + d[-1]), flops=2.0 * c["B"] * macs)
    first = d[0] * d[1]
    return dict(bytes=4.0 * macs * (6 if kind == "train" else 2) + 4.0 * c["B"] * (d[0] + d[-1]),
                flops=2.0 * c["B"] * (3 * macs - first))


# ---- the same in 64-bit torch --------------------------------------------------------------------
def _omega(z):
    """The solution of w + log w = z."""
    zc = z.clamp_min(-600.0)
    w = torch.where(zc < -1, torch.exp(zc.clamp_max(0)), torch.where(zc > 3, zc - torch.log(zc.clamp_min(1)), 1 + (zc - 1) / 2 + (zc - 1) ** 2 / 16))
    w = torch.where(zc < -1, w * torch.exp(-w), w)
    for _ in range(8):
        w = w * (1 + zc - torch.log(w)) / (1 + w)
    return torch.where(z < -600, torch.zeros_like(w), w)


def _lse(C, v):
    """log sum_j exp(v_bj - C_ij): C [n][n], v [B][n]."""
    B, n = v.shape
    out = torch.empty(B, n, dtype=torch.float64, device=v.device)
    step = max(1, int(3e8) // (n * min(n, 4096)))
    for b in range(0, B, step):
        for i in range(0, n, 4096):
            out[b:b + step, i:i + 4096] = torch.logsumexp(v[b:b + step, None, :] - C[None, i:i + 4096], -1)
    return out


def _datafit(c, lb, y):
    """log u1 from log K^T u2 and the target."""
    eps, lam = c["eps"], c["lam"]
    ly = torch.log(y)
    if c["datafit"] == "kl":
        return lam / (eps + lam) * (ly - lb)
    if c["datafit"] == "tv":
        return (ly - lb).clamp(-lam / eps, lam / eps)
    if c["datafit"] == "l2":
        return lam * y / eps - _omega(math.log(lam / eps) + lb + lam * y / eps)
    lc = math.log(lam / eps) + ly
    return torch.where(y > 0, lc - torch.log(_omega(torch.where(y > 0, lc - lb + lam / eps, torch.ones_like(lb)))) - lb,
                       torch.full_like(lb, -lam / eps))


def _mm(c, w, nu, xcol):
    """Table 2's weight update from nu = log w + D^T log(a / s) / x."""
    eps, al, be = c["eps"], c["alpha"], c.get("beta", 0.0)
    if c["penalty"] in ("l1", "elastic"):
        nu = nu - al / (eps * xcol)
    if c["penalty"] in ("l2sq", "elastic"):
        cc = (be if c["penalty"] == "elastic" else al) / (eps * xcol)
        return _omega(torch.log(cc) + nu) / cc
    return torch.exp(nu)


def _iterate(c, cost, D, y, w0, iters):
    """Algorithm 1 in float64 on the inputs as given; returns (w, g, t)."""
    eps, cost, D, y = c["eps"], cost.double(), D.double(), y.double()
    tiny = TINY32 if c["precision"] != "fp64" else 0.0
    n, xcol, w = y.shape[1], D.sum(0), w0.double().clone()
    if c["cost"] == "dense":
        C = cost / eps
    else:
        dx = cost[:, None] - cost[None, :]
        C = (dx.abs() if c["cost"] == "abs" else dx * dx) / eps
    big = float(y.shape[0]) * n * n * 2 * iters > 4e11
    if big:  # the squared distance at eps = 1e-2 spans e^100: sums around the largest term are safe
        K = torch.exp(-C)

        def apply(v, transpose):
            m = v.amax(1, keepdim=True)
            return m + torch.log(torch.exp(v - m) @ K)
    else:
        Ct = C.T.contiguous()

        def apply(v, transpose):
            return _lse(Ct if transpose else C, v)
    src = lambda w: (lambda s: torch.where(s < tiny, torch.zeros_like(s), s))(w @ D.T)  # noqa: E731
    s, g = src(w), torch.zeros_like(y)
    for _ in range(iters):
        la = apply(g, False)
        for _ in range(c["mm_steps"]):
            r = torch.where(s > 0, la - torch.log(s), torch.zeros_like(s))
            w = _mm(c, w, torch.log(w) + r @ D / xcol, xcol)
            s = src(w)
        lb = apply(torch.log(s) - la, True)
        g = _datafit(c, lb, y)
    return w, g * eps, torch.exp(g + lb)


def _exact_banded(c, seed):
    d = _banded_inputs(c, seed)
    n, hw, eps, B = c["n"], c["hw"], c["eps"], c["B"]
    y, vals, rows = d["y"].double(), d["vals"].double(), d["rows"]
    w, Cd = _banded_w0(c, d).double(), d["Cd"].double() / eps
    xcol = vals.sum(1)

    def src(w):
        s = torch.zeros(B, n, dtype=torch.float64, device=DEV)
        for o in range(rows.shape[1]):
            s.index_add_(1, rows[:, o], w * vals[:, o])
        return torch.where(s < TINY32, torch.zeros_like(s), s)

    def band(v, transpose):
        terms = torch.full((2 * hw + 1, B, n), -math.inf, dtype=torch.float64, device=DEV)
        for q in range(2 * hw + 1):
            o = q - hw  # neighbour offset
            lo, hi = max(0, -o), min(n, n - o)
            cost = Cd[2 * hw - q, lo + o:hi + o] if transpose else Cd[q, lo:hi]
            terms[q, :, lo:hi] = v[:, lo + o:hi + o] - cost
        return torch.logsumexp(terms, 0)

    s, g = src(w), torch.zeros_like(y)
    for _ in range(c["iters"]):
        la = band(g, False)
        r = torch.where(s > 0, la - torch.log(s), torch.zeros_like(s))
        acc = torch.zeros_like(w)
        for o in range(rows.shape[1]):
            acc += r[:, rows[:, o]] * vals[:, o]
        w = _mm(c, w, torch.log(w) + acc / xcol, xcol)
        s = src(w)
        lb = band(torch.log(s) - la, True)
        g = _datafit(c, lb, y)
    it = torch.full((B,), c["iters"], dtype=torch.int32)
    return dict(w=w, g=g * eps, t=torch.exp(g + lb), iters=it, status=torch.full_like(it, api.MAX_ITER))


def _exact_net(c, seed):
    y, p, mean, std, tgt, dims = _net_inputs(c, seed)
    y, p64 = y.double(), p.double()
    W, b, off = [], [], 0
    for a, o in zip(dims[:-1], dims[1:]):
        W.append(p[off:off + a * o].reshape(o, a).to(torch.bfloat16).double().requires_grad_(True))
        off += a * o
        b.append(p64[off:off + o].clone().requires_grad_(True))
        off += o
    tot = y.sum(1, keepdim=True)
    h = torch.cat([y * (c["n"] / tot), torch.log(tot)], 1)
    for q in range(4):
        h = h @ W[q].T + b[q]
        if q < 3:
            h = torch.nn.functional.gelu(h)
    if c["kind"] == "predict":
        v = h.detach() * std.double() + mean.double()
        return dict(g0=c["eps"] * v[:, :c["n"]], w0=torch.exp(v[:, c["n"]:]))
    ok = torch.isfinite(tgt)
    r = torch.where(ok, h - (torch.where(ok, tgt, torch.zeros_like(tgt)).double() - mean.double()) / std.double(),
                    torch.zeros_like(h))
    loss = (r * r).sum() / ok.sum()
    loss.backward()
    grad = torch.cat([t.grad.reshape(-1) for q in range(4) for t in (W[q], b[q])])
    if c["kind"] == "gradients":
        return dict(grad=grad, loss=loss.detach().reshape(1))
    upd = grad / (grad.abs() + 1e-8)  # the first AdamW step: both moments equal the gradient's
    return dict(params=p64 - c["lr"] * (upd + 1e-4 * p64), loss=loss.detach().reshape(1))


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "solve":
        cost, D, y, w0 = _solve_inputs(c, seed)
        w, g, t = _iterate(c, cost, D, y, w0, c["iters"])
        it = torch.full((c["B"],), c["iters"], dtype=torch.int32)
        return dict(w=w, g=g, t=t, iters=it, status=torch.full_like(it, api.MAX_ITER))
    if kind == "ragged":
        s = prepare(case, seed)
        n, k = s["sizes"]
        rb, on, oD, ok, out = s["rb"], 0, 0, 0, []
        for p in range(c["B"]):
            a, b = int(n[p]), int(k[p])
            one = dict(c, eps=float(rb.eps[p]), precision="fp32", cost="sq", mm_steps=1)
            out.append(_iterate(one, rb.x[on:on + a], rb.D[oD:oD + a * b].reshape(a, b), rb.y[on:on + a][None],
                                s["w0"][ok:ok + b][None], c["iters"]))
            on, oD, ok = on + a, oD + a * b, ok + b
        w, g, t = (torch.cat([o[q][0] for o in out]) for q in range(3))
        it = torch.full((c["B"],), c["iters"], dtype=torch.int32)
        return dict(w=w, g=g, t=t, iters=it, status=torch.full_like(it, api.MAX_ITER))
    if kind == "banded":
        return _exact_banded(c, seed)
    if kind in ("train", "gradients", "predict"):
        return _exact_net(c, seed)
    # objective: primal and Fenchel dual of the state (L2 datafit, squared-l2 penalty)
    s = prepare(case, seed)
    c = s["c"]
    eps, lam, al, x, D, y, w, g = c["eps"], c["lam"], c["alpha"], s["cost"], s["D"], s["y"], s["w"], s["g"]
    C = (x[:, None] - x[None, :]) ** 2 / eps
    sm = w @ D.T
    f = torch.log(sm) - _lse(C, g / eps)
    lb = _lse(C.T.contiguous(), f)
    t = torch.exp(g / eps + lb)
    kmass = torch.exp(-C).sum()
    f, gn = eps * f, eps * _datafit(c, lb, y)
    zero = torch.zeros_like(f)
    sf = torch.where(sm > 0, sm * f, zero).sum(1)
    primal = sf + (t * g).sum(1) - eps * sm.sum(1) + eps * kmass + lam * 0.5 * ((t - y) ** 2).sum(1) + 0.5 * al * (w * w).sum(1)
    flo = torch.where(torch.isfinite(f), f, torch.full_like(f, math.inf)).amin(1, keepdim=True)
    xtf = torch.where(torch.isfinite(f), f, flo.expand_as(f)) @ D
    f1 = ((-xtf).clamp_min(0) ** 2).sum(1) / (2 * al)
    f2 = torch.where(y - gn / lam >= 0, -gn * y + gn * gn / (2 * lam), -lam * y * y / 2).sum(1)
    dual = -f1 - f2 - eps * (torch.exp(gn / eps + lb).sum(1) - kmass)
    return dict(primal=primal, dual=dual)
