"""FP64 solves and objective with the stored kernel (linear-domain applies) against the FP64 oracle:
row counts off the CTA's rows, one and several problems per warp, several MM steps, a tolerance stop,
potentials beyond the linear range (sums of 2^-900 and less are redone from the logarithms), and a
handle whose n_max is past the stored kernel's limit (log-sum-exp applies).  Bar: the FP64 path's 1e-9.
"""
import numpy as np
import pytest

import oracle
import spectra

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2504_04609_gb300 import otlm as api  # noqa: E402

TOL64 = 1e-9


def rel_l1(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return float(np.abs(a - b).sum() / max(np.abs(b).sum(), 1e-300))


@pytest.mark.parametrize("n,B,k,datafit,penalty,eps,alpha,cost,mm", [
    (2, 1, 1, "l2", "l2sq", 0.5, 0.1, "sq", 1),
    (33, 3, 5, "kl", "l2sq", 3e-2, 1e-3, "sq", 1),
    (201, 1, 10, "kl", "l2sq", 1e-2, 1e-3, "sq", 2),
    (205, 5, 12, "tv", "l1", 1e-2, 1e-2, "sq", 1),
    (1300, 2, 7, "poisson", "l2sq", 1e-2, 1e-3, "sq", 1),
    (300, 4, 9, "l2", "none", 2e-2, 0.0, "abs", 1),
    (160, 2, 6, "tv", "l1", 8e-4, 1e-2, "sq", 2),   # |potentials| up to 1800: outside the linear range
    (160, 9, 6, "kl", "l1", 4e-4, 1e-2, "sq", 1),
])
@pytest.mark.parametrize("n_max", [0, 4097])
def test_fp64_stored_kernel_parity(n, B, k, datafit, penalty, eps, alpha, cost, mm, n_max):
    T = 12
    if n == 2:
        d = dict(x=np.array([0.0, 1.0]), D=np.array([[0.6], [0.4]]), y=np.array([[0.3, 0.5]]))
    else:
        d = spectra.batch(94, B, n, k, 3, dtype=np.float64)
    x = d["x"] * (0.1 if cost == "abs" else 1.0)
    w0 = spectra.initial_weights(d["y"], d["D"])
    dev = lambda a: torch.tensor(a, dtype=torch.float64, device="cuda")  # noqa: E731
    w, g, t, y = dev(w0), torch.zeros(B, n, dtype=torch.float64, device="cuda"), dev(np.zeros((B, n))), dev(d["y"])
    h = api.Handle(max(n, n_max), k, B, "fp64", datafit, penalty, T, 0.0, 5, stream=torch.cuda.current_stream().cuda_stream,
                   mm_steps=mm, cost=cost)
    h.solve(dev(x), dev(d["D"]), y, eps, 1.0, alpha, w, g, t)
    torch.cuda.synchronize()
    h.close()
    C = spectra.abs_cost(x) if cost == "abs" else spectra.squared_cost(x)
    for p in range(B):
        o = oracle.solve_log(C, d["D"], d["y"][p], eps, 1.0, alpha, datafit, penalty, w0[p], T, mm_steps=mm)
        assert rel_l1(w[p].cpu().numpy(), o["w"]) <= TOL64
        assert rel_l1(t[p].cpu().numpy(), o["t"]) <= TOL64


def test_fp64_tolerance_stop_matches_the_oracle():
    d = spectra.batch(95, 5, 210, 12, 3, dtype=np.float64)
    dev = lambda a: torch.tensor(a, dtype=torch.float64, device="cuda")  # noqa: E731
    w0 = spectra.initial_weights(d["y"], d["D"])
    r = api.solve(dev(d["x"]), dev(d["D"]), dev(d["y"]), 1e-2, 1.0, 1e-3, "kl", "l2sq", dev(w0), max_iter=400, tol=1e-7,
                  precision="fp64", poll_every=6)
    C = spectra.squared_cost(d["x"])
    for p in range(5):
        o = oracle.solve_log(C, d["D"], d["y"][p], 1e-2, 1.0, 1e-3, "kl", "l2sq", w0[p], 400, tol=1e-7)
        want = api.CONVERGED if o["err"] <= 1e-7 else api.MAX_ITER  # one of the five is still at 7e-7 after 400
        assert int(r.status[p]) == want and int(r.iters[p]) == o["iters"]
        assert abs(float(r.err[p]) - o["err"]) <= 1e-6 * o["err"]
        assert rel_l1(r.w[p].cpu().numpy(), o["w"]) <= TOL64


@pytest.mark.parametrize("eps", [1e-2, 6e-4])
def test_fp64_objective_stored_kernel(eps):
    d = spectra.batch(96, 5, 190, 10, 3, dtype=np.float64)
    dev = lambda a: torch.tensor(a, dtype=torch.float64, device="cuda")  # noqa: E731
    w0 = spectra.initial_weights(d["y"], d["D"])
    r = api.solve(dev(d["x"]), dev(d["D"]), dev(d["y"]), eps, 1.0, 1e-3, "l2", "l2sq", dev(w0), max_iter=15, precision="fp64")
    P, D = dev(np.zeros(5)), dev(np.zeros(5))
    h = api.Handle(190, 10, 5, "fp64", "l2", "l2sq", 1, 0.0, 4, stream=torch.cuda.current_stream().cuda_stream)
    h.objective(dev(d["x"]), dev(d["D"]), dev(d["y"]), eps, 1.0, 1e-3, r.w, r.g, P, D)
    torch.cuda.synchronize()
    h.close()
    C = spectra.squared_cost(d["x"])
    for p in range(5):
        Po, Do, _ = oracle.objective_and_dual(r.w[p].cpu().numpy(), r.g[p].cpu().numpy(), C, d["D"], d["y"][p], eps, 1.0,
                                              1e-3, "l2", "l2sq")
        assert P[p].item() == pytest.approx(Po, rel=TOL64) and D[p].item() == pytest.approx(Do, rel=TOL64)
