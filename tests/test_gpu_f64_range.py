"""FP64 solves and objective where products leave FP64's range, against the FP64 oracle at the path's
1e-9.  The oracle works on logarithms throughout."""
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
