"""otlm_solve_route: the kernels a solve ran, at the lines between the routes; bench.py labels its results
by it and knows every route its workloads may take."""
import numpy as np
import pytest

import bench
import spectra

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2504_04609_gb300 import otlm as api  # noqa: E402

SMS = 152
CASES = [  # precision, problems, bins, eps, grid, handle options, route
    ("fp32", 4 * SMS, 512, 1e-2, "uniform", {}, "one launch"),
    ("fp32", 4 * SMS + 1, 512, 1e-2, "uniform", {}, "expansion"),
    ("fp32", 4 * SMS + 1, 512, 1e-2, "unsorted", {}, "log"),
    ("fp32", 2 * SMS + 1, 513, 1e-2, "uniform", {}, "expansion"),
    ("fp32", 2, 2048, 1e-2, "unsorted", {}, "one launch"),
    ("fp32", 2, 2049, 1e-2, "unsorted", {}, "log"),
    ("fp32", 2, 2049, 1e-2, "uniform", {}, "one launch"),
    ("fp32", 2, 2049, 1e-2, "uniform", dict(poll_every=9), "device"),
    ("fp32", 2, 4097, 1e-2, "uniform", {}, "expansion"),
    ("fp32", 2, 300, 1e-2, "uniform", dict(dw_tol=1e-9), "expansion"),
    ("fp32", 2, 300, 1e-2, "uniform", dict(cost="abs"), "log"),
    ("bf16tc", SMS, 2048, 1e-2, "uniform", {}, "one launch"),
    ("bf16tc", 64, 4097, 1e-2, "uniform", {}, "expansion"),
    ("bf16tc", 1280, 1024, 1e-2, "uniform", {}, "expansion"),
    ("bf16tc", 1281, 1024, 1e-2, "uniform", {}, "tensor"),
    ("bf16tc", 1280, 1024, 1e-3, "uniform", {}, "tensor"),   # more than 18 blocks
    ("bf16tc", 2, 300, 1e-2, "unsorted", {}, "tensor"),
    ("bf16tc", 2, 300, 1e-2, "uniform", dict(bf16_single_until=1e-5), "tensor"),
    ("fp64", 2, 300, 1e-2, "uniform", {}, "stored"),
    ("fp64", 2, 300, 1e-2, "uniform", dict(check_every=2), "log"),
]


@pytest.mark.parametrize("precision,B,n,eps,grid,options,route", CASES)
def test_route_of_a_solve(precision, B, n, eps, grid, options, route):
    d = spectra.batch(76, 2, n, 8, 3, dtype=np.float64 if precision == "fp64" else np.float32)
    x, D, y = d["x"], d["D"], d["y"][np.arange(B) % 2]
    if grid == "unsorted":
        perm = np.random.default_rng(9).permutation(n)
        x, D, y = x[perm], np.ascontiguousarray(D[perm]), np.ascontiguousarray(y[:, perm])
    dt = torch.float64 if precision == "fp64" else torch.float32
    dev = lambda a: torch.tensor(a, dtype=dt, device="cuda")  # noqa: E731
    h = api.Handle(n, 8, B, precision, "l2", "l2sq", 8, 0.0, stream=torch.cuda.current_stream().cuda_stream, **options)
    assert h.route == "none"
    w = dev(spectra.initial_weights(y, D))
    h.solve(dev(x), dev(D), dev(y), eps, 1.0, 1e-3, w)
    torch.cuda.synchronize()
    assert h.route == route and bool(torch.isfinite(w).all())
    if precision != "fp64" and route != "device":
        assert route in bench.ROUTE_LABELS
    h.close()


def test_route_of_a_dense_cost():
    d = spectra.batch(76, 2, 200, 8, 3)
    C = torch.tensor(spectra.squared_cost(d["x"].astype(np.float64)).astype(np.float32), device="cuda")
    for precision, route in (("fp32", "log"), ("bf16tc", "tensor")):
        h = api.Handle(200, 8, 2, precision, "l2", "l2sq", 4, 0.0, stream=torch.cuda.current_stream().cuda_stream)
        w = torch.tensor(spectra.initial_weights(d["y"], d["D"]).astype(np.float32), device="cuda")
        h.solve_cost(C, torch.tensor(d["D"], device="cuda"), torch.tensor(d["y"], device="cuda"), 1e-2, 1.0, 1e-3, w)
        torch.cuda.synchronize()
        assert h.route == route
        h.close()
