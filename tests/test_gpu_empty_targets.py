"""Targets without mass beside others on a tensor-core handle: the empty problem collapses (its violation is
0 / 0), its transported marginal is 0 on every route, and the others are solved as without it."""
import numpy as np
import pytest

import oracle
import spectra

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2504_04609_gb300 import otlm as api  # noqa: E402


@pytest.mark.parametrize("datafit", ["kl", "balanced"])
@pytest.mark.parametrize("n,grid,route", [(600, "uniform", "one launch"), (4200, "uniform", "expansion"), (600, "unsorted", "tensor")])
def test_transported_marginal_of_an_empty_target(datafit, n, grid, route):
    B, k, T = 4, 8, 6
    d = spectra.batch(79, B, n, k, 3)
    order = np.random.default_rng(3).permutation(n) if grid == "unsorted" else np.arange(n)
    x, D, y = d["x"][order], np.ascontiguousarray(d["D"][order]), np.ascontiguousarray(d["y"][:, order])
    y = y + np.float32(1e-3)
    y[1] = 0.0
    w0 = spectra.initial_weights(y, D).astype(np.float32)
    w0[1] = w0[0]
    dev = lambda a: torch.tensor(a, device="cuda")  # noqa: E731
    w, t, st = dev(w0), torch.ones(B, n, device="cuda"), torch.empty(B, dtype=torch.int32, device="cuda")
    h = api.Handle(n, k, B, "bf16tc", datafit, "l2sq", T, 0.0, 4, stream=torch.cuda.current_stream().cuda_stream)
    h.solve(dev(x), dev(D), dev(y), 2e-2, 1.0, 1e-3, w, None, t, None, None, st)
    torch.cuda.synchronize()
    assert h.route == route
    h.close()
    assert st.cpu().numpy().tolist() == [api.MAX_ITER, api.NONFINITE, api.MAX_ITER, api.MAX_ITER]
    assert bool((t[1] == 0).all())
    C, D64 = spectra.squared_cost(x.astype(np.float64)), D.astype(np.float64)
    for p in (0, 3):
        o = oracle.solve_log(C, D64, y[p].astype(np.float64), 2e-2, 1.0, 1e-3, datafit, "l2sq", w0[p].astype(np.float64), T)
        assert np.abs(w[p].cpu().numpy() - o["w"]).sum() <= 1e-5 * np.abs(o["w"]).sum()
        assert np.abs(t[p].cpu().numpy() - o["t"]).sum() <= 1e-5 * np.abs(o["t"]).sum()
