"""The routes of a tensor-core handle by batch size against the FP64 oracle: one launch (small batches),
expansion applies (batches whose GEMMs do not fill the SM pairs, long grids included), GEMMs with split
reductions (dense costs, mid-size batches) and GEMMs with their fix-up, whose rows go to CTAs or, above
the number of CTAs, to warps.

Bar: the paths' relative L1 error of 1e-5 in w and t; every route's arithmetic is that of a path that
has this bar already (FP32 expansions, BF16 hi/lo products, log-domain rows)."""
import numpy as np
import pytest

import oracle
import spectra

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2504_04609_gb300 import otlm as api  # noqa: E402

TOL = 1e-5


def rel_l1(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return float(np.abs(a - b).sum() / max(np.abs(b).sum(), 1e-300))


def _dev(a):
    return torch.tensor(a, device="cuda")


def _compare(r, d, B, ref, C, eps, alpha, datafit, penalty, T, mm_steps=1):
    """The first and the last copy of each of the problems d holds."""
    P = d["y"].shape[0]
    D64 = d["D"].astype(np.float64)
    for p in range(P):
        y64 = d["y"][p].astype(np.float64)
        o = ref(C, D64, y64, eps, 1.0, alpha, datafit, penalty, spectra.initial_weights(y64, D64), T, mm_steps=mm_steps)
        for q in {q for q in (p, (B - 1 - p) // P * P + p) if q < B}:
            assert rel_l1(r["w"][q].cpu().numpy(), o["w"]) <= TOL, (p, q)
            assert rel_l1(r["t"][q].cpu().numpy(), o["t"]) <= TOL, (p, q)


@pytest.mark.parametrize("B,n,k", [(70, 300, 12), (620, 300, 12), (1, 4200, 20), (3, 4200, 20), (80, 4200, 20)])
@pytest.mark.parametrize("mm_steps", [1, 2])
def test_grid_solves_of_every_batch_size(B, n, k, mm_steps):
    d = spectra.batch(97, min(B, 3), n, k, 3)
    y = d["y"][np.arange(B) % min(B, 3)]
    w0 = spectra.initial_weights(y, d["D"]).astype(np.float32)
    r = api.solve(_dev(d["x"]), _dev(d["D"]), _dev(y), 2e-2, 1.0, 1e-3, "l2", "l2sq", _dev(w0), max_iter=8,
                  precision="bf16tc", mm_steps=mm_steps)
    assert np.all(r.iters.cpu().numpy() == 8)
    _compare(dict(w=r.w, t=r.t), d, B, oracle.solve_log, spectra.squared_cost(d["x"].astype(np.float64)), 2e-2, 1e-3, "l2",
             "l2sq", 8, mm_steps)


@pytest.mark.parametrize("precision", ["fp32", "bf16tc"])
@pytest.mark.parametrize("B,n", [(2, 300), (2, 2100), (620, 300)])
def test_grids_without_a_plan(precision, B, n):
    """An unsorted grid keeps the log-domain or GEMM applies (or one launch) at every batch size."""
    d = spectra.batch(96, 2, n, 12, 3)
    perm = np.random.default_rng(5).permutation(n)
    d = dict(d, x=d["x"][perm], D=np.ascontiguousarray(d["D"][perm]), y=np.ascontiguousarray(d["y"][:, perm]))
    y = d["y"][np.arange(B) % 2]
    w0 = spectra.initial_weights(y, d["D"]).astype(np.float32)
    r = api.solve(_dev(d["x"]), _dev(d["D"]), _dev(y), 2e-2, 1.0, 1e-3, "l2", "l2sq", _dev(w0), max_iter=8,
                  precision=precision)
    _compare(dict(w=r.w, t=r.t), d, B, oracle.solve_log, spectra.squared_cost(d["x"].astype(np.float64)), 2e-2, 1e-3, "l2",
             "l2sq", 8)


@pytest.mark.parametrize("B", [65, 150, 256])
@pytest.mark.parametrize("n", [300, 1000])
def test_dense_cost_split_reductions_of_mid_size_batches(B, n):
    """A non-symmetric truncated cost: source and target sums through the split, underflowed rows listed
    by the sum of the splits."""
    d = spectra.batch(98, 3, n, 10, 3)
    x = 0.25 + d["x"].astype(np.float64)
    C = 0.5 * (x[:, None] - x[None, :]) ** 2 / x[:, None] ** 2
    C[np.abs(x[:, None] - x[None, :]) > 0.3] = np.inf
    C = C.astype(np.float32)
    y = d["y"][np.arange(B) % 3]
    w = _dev(spectra.initial_weights(y, d["D"]).astype(np.float32))
    t = torch.empty(B, n, device="cuda")
    h = api.Handle(n, 10, B, "bf16tc", "tv", "l1", 10, 0.0)
    h.solve_cost(_dev(C), _dev(d["D"]), _dev(y), 2e-2, 1.0, 1e-2, w, None, t)
    torch.cuda.synchronize()
    h.close()
    _compare(dict(w=w, t=t), d, B, oracle.solve_log, C.astype(np.float64), 2e-2, 1e-2, "tv", "l1", 10)


@pytest.mark.parametrize("holes", [0, 1, 2600])
def test_listed_rows_by_cta_and_by_warp(holes):
    """KL at eps = 1e-3: a problem whose bins 60..459 are zero has 100 to 300 underflowed rows per apply.
    One such problem: a CTA per row, potentials formed again; all 2600: a warp per row, stored."""
    B, n = 2600, 512
    d = spectra.batch(33, 6, n, 16, 3)
    y = np.tile(d["y"], (B // 6 + 1, 1))[:B].copy()
    y[:holes, 60:460] = 0.0
    w0 = spectra.initial_weights(y, d["D"]).astype(np.float32)
    r = api.solve(_dev(d["x"]), _dev(d["D"]), _dev(y), 1e-3, 1.0, 1e-3, "kl", "l2sq", _dev(w0), max_iter=20,
                  precision="bf16tc")
    C = spectra.squared_cost(d["x"].astype(np.float64))
    D64 = d["D"].astype(np.float64)
    for p in (0, 1, 5, B - 1):
        y64 = y[p].astype(np.float64)
        o = oracle.solve_log(C, D64, y64, 1e-3, 1.0, 1e-3, "kl", "l2sq", spectra.initial_weights(y64, D64), 20)
        assert rel_l1(r.w[p].cpu().numpy(), o["w"]) <= TOL, p
        assert rel_l1(r.t[p].cpu().numpy(), o["t"]) <= TOL, p


@pytest.mark.parametrize("long_column", [False, True])
def test_banded_dictionary_interleaved_and_by_columns(long_column):
    """A column much longer than the mean keeps the dictionary's columns apart in the MM step."""
    from scipy.sparse import csc_matrix
    n, k, B = 700, 70, 3
    Cd, half = spectra.truncated_cost_band(n, rho=0.01, delta=10.0)
    Cd = spectra.to_dtype(Cd, np.float32)
    cp, ri, vv = spectra.scaling_dictionary(n, k)
    if long_column:
        ri, vv = np.concatenate([np.arange(n, dtype=ri.dtype), ri[cp[1]:]]), np.concatenate([np.full(n, 1.0 / n), vv[cp[1]:]])
        cp = np.concatenate([cp[:1], cp[1:] - cp[1] + n]).astype(cp.dtype)
        assert n * k > 2 * cp[-1]
    vv = spectra.to_dtype(vv, np.float32)
    x_col = np.add.reduceat(vv.astype(np.float64), cp[:-1])
    y = spectra.to_dtype(np.stack([spectra.scaling_target(n, k, np.random.default_rng(650 + p)) for p in range(B)]), np.float32)
    w0 = y.astype(np.float64).sum(1, keepdims=True) / (k * x_col)
    w, t = _dev(w0.astype(np.float32)), torch.empty(B, n, device="cuda")
    g, it, err, st = torch.zeros(B, n, device="cuda"), *(torch.empty(B, dtype=q, device="cuda")
                                                         for q in (torch.int32, torch.float32, torch.int32))
    h = api.Handle(64, 8, B, "fp32", "kl", "l1", 25, 0.0, 8, stream=torch.cuda.current_stream().cuda_stream)
    h.solve_banded(_dev(Cd), half, _dev(cp.astype(np.int32)), _dev(ri.astype(np.int32)), _dev(vv), _dev(y), 5e-2, 1.0, 1e-3,
                   w, g, t, it, err, st)
    torch.cuda.synchronize()
    h.close()
    X = csc_matrix((vv.astype(np.float64), ri, cp), shape=(n, k))
    for p in range(B):
        o = oracle.solve_log_banded(Cd.astype(np.float64), half, X, y[p].astype(np.float64), 5e-2, 1.0, 1e-3, "kl", "l1",
                                    w0[p], 25)
        assert rel_l1(w[p].cpu().numpy(), o["w"]) <= TOL and rel_l1(t[p].cpu().numpy(), o["t"]) <= TOL
