"""FP64 solves and objective where products or kernel entries leave FP64's range, against the FP64
oracle at the path's 1e-9: source marginals down to the subnormals, weights whose product with the
penalty's coefficient is subnormal, and transport so far that exp(-C / eps) underflows where mass
still moves.  The oracle works on logarithms throughout."""
import numpy as np
import pytest
from scipy.special import logsumexp

import oracle
import spectra

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2504_04609_gb300 import otlm as api  # noqa: E402

TOL64 = 1e-9


def rel_l1(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return float(np.abs(a - b).sum() / max(np.abs(b).sum(), 1e-300))


def _peaks(x, mu, sig):
    D = np.exp(-0.5 * ((x[:, None] - np.asarray(mu)) / sig) ** 2)
    return D / D.sum(0)


def _solve_and_compare(x, D, y, w0, eps, alpha, datafit, penalty, T, n_max=0, mm_steps=1):
    dev = lambda a: torch.tensor(a, dtype=torch.float64, device="cuda")  # noqa: E731
    B, n = y.shape
    w, t = dev(w0), torch.empty(B, n, dtype=torch.float64, device="cuda")
    st = torch.empty(B, dtype=torch.int32, device="cuda")
    h = api.Handle(max(n, n_max), D.shape[1], B, "fp64", datafit, penalty, T, 0.0, 5,
                   stream=torch.cuda.current_stream().cuda_stream, mm_steps=mm_steps)
    h.solve(dev(x), dev(D), dev(y), eps, 1.0, alpha, w, None, t, None, None, st)
    torch.cuda.synchronize()
    h.close()
    assert np.all(st.cpu().numpy() == api.MAX_ITER)
    for p in range(B):
        o = oracle.solve_log(spectra.squared_cost(x), D, y[p], eps, 1.0, alpha, datafit, penalty, w0[p], T,
                             mm_steps=mm_steps)
        assert rel_l1(w[p].cpu().numpy(), o["w"]) <= TOL64, p
        assert rel_l1(t[p].cpu().numpy(), o["t"]) <= TOL64, p


@pytest.mark.parametrize("mm_steps", [1, 2])
@pytest.mark.parametrize("n,k,sig", [(500, 1, 0.01), (500, 3, 0.008), (1000, 10, 0.005)])
@pytest.mark.parametrize("seed", range(4))
def test_source_marginals_down_to_the_subnormals(n, k, sig, mm_steps, seed):
    """Bins far from every atom have a source marginal s near 2^-1074; s / a is then below any double."""
    rng = np.random.default_rng([71, n, k, seed])
    x = np.arange(n) / (n - 1)
    D = _peaks(x, rng.uniform(0.1, 0.9, k), sig)
    y = np.abs(D @ rng.gamma(2.0, 1.0, (k, 5)) + 1e-3 * rng.random((n, 5))).T.copy()
    _solve_and_compare(x, D, y, spectra.initial_weights(y, D), 1e-2, 1e-3, "l2", "l2sq", 15, mm_steps=mm_steps)


def _far_transport(n=400):
    """Atoms at 0.2 and 0.35, the target's peak at 0.7 over a floor of 1e-6."""
    x = np.arange(n) / (n - 1)
    D = _peaks(x, [0.2, 0.35], 0.02)
    y = _peaks(x, [0.7], 0.02).T + 1e-6
    return x, D, y, spectra.initial_weights(y, D)


@pytest.mark.parametrize("eps", [1e-4, 2e-4])
@pytest.mark.parametrize("datafit", ["kl", "tv"])
def test_transport_beyond_the_stored_kernel(eps, datafit):
    """K_ij = exp(-C_ij / eps) is 0 beyond |x_i - x_j| = 0.27 to 0.39, where u_j = 2^1000 makes the
    term matter: no sum of the rows it reaches may be taken from the stored kernel."""
    x, D, y, w0 = _far_transport()
    _solve_and_compare(x, D, y, w0, eps, 1e-2, datafit, "l1", 100)


@pytest.mark.parametrize("B", [1, 5])
@pytest.mark.parametrize("datafit", ["kl", "tv"])
def test_objective_of_transport_beyond_the_stored_kernel(datafit, B):
    """Against a handle past the stored kernel's size (log-sum-exp applies), and the primal against its
    formula with log Q - log K = (f + g) / eps (the oracle's own divides by K)."""
    x, D, y, w0 = _far_transport()
    eps, C = 1e-4, spectra.squared_cost(x)
    o = oracle.solve_log(C, D, y[0], eps, 1.0, 1e-2, datafit, "l1", w0[0], 40)
    dev = lambda a: torch.tensor(np.tile(a, (B, 1)), dtype=torch.float64, device="cuda")  # noqa: E731
    out = {}
    for n_max in (400, 4097):
        P, Dv = (torch.zeros(B, dtype=torch.float64, device="cuda") for _ in range(2))
        h = api.Handle(n_max, 2, B, "fp64", datafit, "l1", 1, 0.0, 4, stream=torch.cuda.current_stream().cuda_stream)
        h.objective(torch.tensor(x, device="cuda"), torch.tensor(D, device="cuda"), dev(y[0]), eps, 1.0, 1e-2, dev(o["w"]),
                    dev(o["g"]), P, Dv)
        torch.cuda.synchronize()
        h.close()
        out[n_max] = P.cpu().numpy(), Dv.cpu().numpy()
    np.testing.assert_allclose(out[400], out[4097], rtol=TOL64)
    s = D @ o["w"]
    log_a = logsumexp((o["g"][None, :] - C) / eps, axis=1)
    with np.errstate(divide="ignore"):
        fg = np.log(s)[:, None] - log_a[:, None] + o["g"][None, :] / eps
    Q = np.exp(fg - C / eps)
    kl = np.sum(Q[s > 0] * fg[s > 0]) - Q.sum() + np.exp(-C / eps).sum()
    t = Q.sum(axis=0)
    fit = np.sum(t * np.log(t / y[0]) - t + y[0]) if datafit == "kl" else np.abs(t - y[0]).sum()
    np.testing.assert_allclose(out[400][0], eps * kl + fit + 1e-2 * o["w"].sum(), rtol=TOL64)


@pytest.mark.parametrize("n_max", [0, 4097])
@pytest.mark.parametrize("penalty", ["l2sq", "elastic"])
@pytest.mark.parametrize("w_start,coef", [(1e-300, 1e-20), (0.5, 1e-312)])
def test_weights_whose_product_with_the_coefficient_is_subnormal(n_max, penalty, w_start, coef):
    """w = 1e-300 with alpha / (eps x_j) = 1e-18, and a coefficient whose reciprocal overflows (stored
    kernel and log-sum-exp applies)."""
    rng = np.random.default_rng(73)
    n, k = 200, 3
    x = np.arange(n) / (n - 1)
    D = _peaks(x, [0.25, 0.5, 0.7], 0.03)
    y = (D @ rng.gamma(2.0, 1.0, (k, 2)) + 1e-3).T.copy()
    w0 = np.full((2, k), w_start)
    dev = lambda a: torch.tensor(a, dtype=torch.float64, device="cuda")  # noqa: E731
    w = dev(w0)
    alpha, beta = (coef, 0.0) if penalty == "l2sq" else (1e-3, coef)
    h = api.Handle(max(n, n_max), k, 2, "fp64", "kl", penalty, 2, 0.0, 5, stream=torch.cuda.current_stream().cuda_stream,
                   beta=beta)
    h.solve(dev(x), dev(D), dev(y), 1e-2, 1.0, alpha, w)
    torch.cuda.synchronize()
    h.close()
    for p in range(2):
        o = oracle.solve_log(spectra.squared_cost(x), D, y[p], 1e-2, 1.0, alpha, "kl", penalty, w0[p], 2, beta=beta)
        assert rel_l1(w[p].cpu().numpy(), o["w"]) <= TOL64
