"""Kernel applies by block expansions (grids whose blocks are short in kernel widths) against the
FP64 oracle, at the edges of the block plan: the smallest grid that qualifies and one bin less,
ragged last blocks, one block, the narrowest blocks, non-uniform, decreasing, shifted and unsorted
grids (the last summed term by term), and potentials that reach -inf or the TV bound.

Bar: the FP32 path's relative L1 error of 1e-5 in w and t.  The expansion's polynomial is within
1.9e-8 of each term and pairs of blocks left out are below 2^-28 of a sum, both under FP32's 6e-8
rounding, so the bar of the path holds unchanged.
"""
import numpy as np
import pytest

import oracle
import spectra

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2504_04609_gb300 import otlm as api  # noqa: E402

TOL32 = 1e-5


def rel_l1(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return float(np.abs(a - b).sum() / max(np.abs(b).sum(), 1e-300))


def _grid(kind, n):
    u = np.arange(n) / (n - 1)
    if kind == "warped":
        return u + 0.12 / (2 * np.pi) * np.sin(2 * np.pi * u)
    if kind == "descending":
        return u[::-1].copy()
    if kind == "shifted":
        return u - 0.5
    if kind == "unsorted":
        return np.concatenate([u[::2], u[1::2]])
    return u


def _problems(kind, n, k, eps, seed, B):
    out = []
    for p in range(B):
        rng = np.random.default_rng([seed, n, p])
        x = _grid(kind, n)
        z = x if kind != "shifted" else x + 0.5
        mu, sig = rng.uniform(0.1, 0.9, k), np.exp(rng.normal(np.log(0.02), 0.3, k))
        D = np.exp(-0.5 * ((z[:, None] - mu) / sig) ** 2)
        D /= D.sum(0)
        y = np.maximum(D[:, :4] @ rng.gamma(2.0, 1.0, min(4, k)) * (1 + 0.01 * rng.normal(size=n)), 0)
        out.append(dict(n=n, k=k, eps=eps, **{q: spectra.to_dtype(v, np.float32) for q, v in (("x", x), ("D", D), ("y", y))}))
    return out


def _oracle(p, eps, datafit, penalty, alpha, T):
    x, D, y = (p[q].astype(np.float64) for q in ("x", "D", "y"))
    return oracle.solve_log(spectra.squared_cost(x), D, y, eps, 1.0, alpha, datafit, penalty,
                            spectra.initial_weights(y, D), T)


CASES = [  # (grid, n, eps, datafit, penalty, alpha)
    ("uniform", 128, 1e-1, "tv", "l1", 1e-2),
    ("uniform", 127, 1e-1, "tv", "l1", 1e-2),
    ("uniform", 130, 3.0, "kl", "l2sq", 1e-3),
    ("uniform", 777, 5e-2, "l2", "l2sq", 1e-3),
    ("uniform", 1025, 1e-2, "kl", "l1", 1e-2),
    ("uniform", 1500, 2e-3, "tv", "l1", 1e-2),
    ("uniform", 2048, 8e-4, "l2", "l2sq", 1e-3),
    ("warped", 900, 1e-2, "tv", "l1", 1e-2),
    ("descending", 640, 2e-2, "kl", "l2sq", 1e-3),
    ("shifted", 513, 2e-2, "l2", "l1", 1e-2),
    ("unsorted", 300, 2e-2, "tv", "l1", 1e-2),
]


@pytest.mark.parametrize("grid,n,eps,datafit,penalty,alpha", CASES)
@pytest.mark.parametrize("cta", [128, 512])
def test_expansion_in_the_uneven_batch(grid, n, eps, datafit, penalty, alpha, cta):
    T, k = 8, 20
    probs = _problems(grid, n, k, eps, 91, 2)
    rb = api.ragged_batch(probs)
    w = torch.tensor(np.concatenate([spectra.initial_weights(p["y"], p["D"]) for p in probs]).astype(np.float32), device="cuda")
    t = torch.empty_like(rb.y)
    it, st = (torch.empty(2, dtype=torch.int32, device="cuda") for _ in range(2))
    err = torch.empty(2, device="cuda")
    h = api.Handle(n, k, 2, "fp32", datafit, penalty, T, 0.0, stream=torch.cuda.current_stream().cuda_stream, ragged_cta=cta)
    h.solve_ragged(rb, 1.0, alpha, w, None, t, it, err, st)
    torch.cuda.synchronize()
    h.close()
    assert np.all(st.cpu().numpy() == api.MAX_ITER)
    for i, p in enumerate(probs):
        o = _oracle(p, float(np.float32(eps)), datafit, penalty, alpha, T)
        assert rel_l1(w.cpu().numpy()[i * k:(i + 1) * k], o["w"]) <= TOL32
        assert rel_l1(t.cpu().numpy()[i * n:(i + 1) * n], o["t"]) <= TOL32


@pytest.mark.parametrize("grid,n,eps,datafit,penalty,alpha", CASES)
@pytest.mark.parametrize("B", [1, 3, 620])
def test_expansion_in_the_shared_grid_batch(grid, n, eps, datafit, penalty, alpha, B):
    """B = 1 and 3 split a problem's row blocks over CTAs, 620 gives one CTA of four warps to a
    problem (620 problems are copies of three)."""
    T, k = 8, 20
    probs = _problems(grid, n, k, eps, 92, min(B, 3))
    x, D = probs[0]["x"], probs[0]["D"]  # the batch shares the first problem's grid and dictionary
    y = np.stack([probs[p % 3]["y"] for p in range(B)])
    w0 = spectra.initial_weights(y, D).astype(np.float32)
    dev = lambda a: torch.tensor(a, device="cuda")  # noqa: E731
    r = api.solve(dev(x), dev(D), dev(y), eps, 1.0, alpha, datafit, penalty, dev(w0), max_iter=T)
    assert np.all(r.iters.cpu().numpy() == T)
    for p in range(min(B, 3)):
        o = _oracle(dict(probs[p], D=D), eps, datafit, penalty, alpha, T)
        for q in range(p, B, 3):
            if q in (p, B - 3 + p):
                assert rel_l1(r.w[q].cpu().numpy(), o["w"]) <= TOL32
                assert rel_l1(r.t[q].cpu().numpy(), o["t"]) <= TOL32


@pytest.mark.parametrize("k", [1, 33, 64, 129, 256])
@pytest.mark.parametrize("B", [2, 200, 700])
def test_batched_mm_step_sizes(k, B):
    """Every dictionary bucket with one, four and eight problems per CTA (a ragged last CTA), two MM
    steps, against the oracle at the FP32 bar."""
    d = spectra.batch(93, min(B, 3), 261, k, 1)
    y = d["y"][np.arange(B) % min(B, 3)]
    w0 = spectra.initial_weights(y, d["D"]).astype(np.float32)
    dev = lambda a: torch.tensor(a, device="cuda")  # noqa: E731
    r = api.solve(dev(d["x"]), dev(d["D"]), dev(y), 5e-2, 1.0, 1e-3, "l2", "l2sq", dev(w0), max_iter=6, mm_steps=2)
    C = spectra.squared_cost(d["x"].astype(np.float64))
    D64 = d["D"].astype(np.float64)
    for p in range(min(B, 3)):
        y64 = y[p].astype(np.float64)
        o = oracle.solve_log(C, D64, y64, 5e-2, 1.0, 1e-3, "l2", "l2sq", spectra.initial_weights(y64, D64), 6, mm_steps=2)
        for q in (p, (B - 1) // 3 * 3 + p if (B - 1) // 3 * 3 + p < B else p):
            assert rel_l1(r.w[q].cpu().numpy(), o["w"]) <= TOL32
            assert rel_l1(r.t[q].cpu().numpy(), o["t"]) <= TOL32
