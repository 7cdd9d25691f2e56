"""The tensor-core applies at the sizes that batches on sorted grids solve by block expansions or in one
launch: the same problems with their bins in another order (no block plan, so the GEMMs run), against the
FP64 oracle at the path's relative L1 error of 1e-5; and the FP32 expansion applies that split a problem
over CTAs, for small batches that the one-launch route would take (a weight-change criterion keeps them
off it)."""
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


def _reordered(d):
    perm = np.random.default_rng(11).permutation(len(d["x"]))
    return dict(d, x=d["x"][perm], D=np.ascontiguousarray(d["D"][perm]), y=np.ascontiguousarray(d["y"][:, perm]))


def _solve(d, eps, alpha, datafit, penalty, T, tol=0.0, precision="bf16tc", route="tensor", **options):
    x, D, y = (torch.tensor(d[q], device="cuda") for q in ("x", "D", "y"))
    B, n = y.shape
    w = torch.tensor(spectra.initial_weights(d["y"], d["D"]).astype(np.float32), device="cuda")
    t, err = torch.empty_like(y), torch.empty(B, device="cuda")
    it, st = (torch.empty(B, dtype=torch.int32, device="cuda") for _ in range(2))
    h = api.Handle(n, D.shape[1], B, precision, datafit, penalty, T, tol, 4, stream=torch.cuda.current_stream().cuda_stream,
                   **options)
    h.solve(x, D, y, eps, 1.0, alpha, w, None, t, it, err, st)
    torch.cuda.synchronize()
    assert h.route == route
    h.close()
    return {q: v.cpu().numpy() for q, v in dict(w=w, t=t, it=it, err=err, st=st).items()}


def _oracle(d, p, eps, alpha, datafit, penalty, T, **kw):
    D, y = d["D"].astype(np.float64), d["y"][p].astype(np.float64)
    return oracle.solve_log(spectra.squared_cost(d["x"].astype(np.float64)), D, y, eps, 1.0, alpha, datafit, penalty,
                            spectra.initial_weights(y, D), T, **kw)


def _same(r, p, o):
    assert rel_l1(r["w"][p], o["w"]) <= TOL and rel_l1(r["t"][p], o["t"]) <= TOL, p


@pytest.mark.parametrize("datafit,penalty,eps,alpha", [("l2", "l2sq", 1e-2, 1e-3), ("l2", "l1", 2e-2, 1e-2),
                                                       ("kl", "l2sq", 5e-2, 1e-3), ("tv", "l1", 5e-2, 1e-2),
                                                       ("poisson", "l2sq", 2e-2, 1e-3)])
def test_trajectory_with_split_reductions(datafit, penalty, eps, alpha):
    """Nine problems (the reduction split over five 64-wide blocks), n = 300 (a ragged third row tile)."""
    d = _reordered(spectra.batch(31, 9, 300, 12, 3))
    r = _solve(d, eps, alpha, datafit, penalty, 30)
    assert np.all(r["st"] == api.MAX_ITER) and np.all(r["it"] == 30)
    for p in range(9):
        _same(r, p, _oracle(d, p, eps, alpha, datafit, penalty, 30))


@pytest.mark.parametrize("n,k,B", [(200, 10, 4), (256, 9, 20), (300, 5, 3)])
def test_dictionary_sizes_off_the_tf32_row_pitch(n, k, B):
    """k not a multiple of 4: TF32 rows at a pitch of k rounded up to 4, partial sums of D^T r apart."""
    d = _reordered(spectra.batch(84, B, n, k, 3))
    r = _solve(d, 2e-2, 1e-2, "tv", "l1", 12)
    for p in range(B):
        _same(r, p, _oracle(d, p, 2e-2, 1e-2, "tv", "l1", 12))


def test_two_sm_apply_with_a_partial_row_tile_and_compaction():
    """130 problems of 300 bins to 1e-5 on the two-SM kernel: a partial row tile on the even CTA, none on
    the odd one, and a compacted column list.  The violation is a sum of differences of nearly equal
    ratios: 2.5e-6 absolute, as for the same batch on the sorted grid."""
    d = _reordered(spectra.batch(37, 130, 300, 12, 3))
    args = (1e-2, 1e-3, "l2", "l2sq")
    r = _solve(d, *args, 400, tol=1e-5)
    assert np.all(r["st"] == api.CONVERGED) and np.all(r["err"] <= 1e-5) and len(np.unique(r["it"])) > 1
    for p in (0, 1, 63, 127, 128, 129):
        o = _oracle(d, p, *args, int(r["it"][p]))
        assert abs(float(r["err"][p]) - o["err"]) <= 2.5e-6
        _same(r, p, o)


def test_single_target_streams_the_stored_kernel():
    """n = 8192: 256 MiB of BF16 hi/lo kernel per apply, one column, the reduction over 16 ranges."""
    d = _reordered(spectra.batch(34, 1, 8192, 64, 5))
    r = _solve(d, 1e-2, 1e-3, "l2", "l2sq", 6)
    _same(r, 0, _oracle(d, 0, 1e-2, 1e-3, "l2", "l2sq", 6))


@pytest.mark.parametrize("mm_steps", [2, 3])
def test_inner_steps_over_two_column_tiles(mm_steps):
    """130 problems: two 128-wide column tiles of every GEMM, no split reduction, elastic net."""
    d = _reordered(spectra.batch(53, 130, 256, 16, 3))
    r = _solve(d, 1e-2, 1e-3, "l2", "elastic", 15, beta=5e-3, mm_steps=mm_steps)
    for p in range(0, 130, 7):
        _same(r, p, _oracle(d, p, 1e-2, 1e-3, "l2", "elastic", 15, beta=5e-3, mm_steps=mm_steps))


def test_weight_change_criterion():
    d = _reordered(spectra.batch(38, 5, 300, 12, 3))
    r = _solve(d, 2e-2, 1e-3, "l2", "l2sq", 400, tol=1e-4, dw_tol=1e-3)
    assert np.all(r["st"] == api.CONVERGED)
    for p in range(5):
        o = _oracle(d, p, 2e-2, 1e-3, "l2", "l2sq", int(r["it"][p]), tol=0.0)
        assert o["dw_hist"][-1] <= 1.01e-3 and o["err"] <= 1e-4 + 2.5e-6
        _same(r, p, o)


@pytest.mark.parametrize("n,eps,datafit,penalty,alpha", [(128, 1e-1, "tv", "l1", 1e-2), (130, 3.0, "kl", "l2sq", 1e-3),
                                                         (1025, 1e-2, "kl", "l1", 1e-2), (2048, 8e-4, "l2", "l2sq", 1e-3)])
@pytest.mark.parametrize("B", [1, 3, 40])
def test_fp32_expansions_split_over_ctas(n, eps, datafit, penalty, alpha, B):
    """Up to 32 CTAs per problem, more than row blocks; the last to finish decides."""
    d = spectra.batch(77, min(B, 3), n, 20, 3)
    d["y"] = d["y"][np.arange(B) % min(B, 3)]
    r = _solve(d, eps, alpha, datafit, penalty, 8, precision="fp32", route="expansion", dw_tol=1e-30)
    assert np.all(r["it"] == 8) and np.all(r["st"] == api.MAX_ITER)
    for p in range(min(B, 3)):
        o = _oracle(d, p, eps, alpha, datafit, penalty, 8)
        for q in {p, (B - 1 - p) // 3 * 3 + p}:
            assert abs(float(r["err"][q]) - o["err"]) <= 2.5e-6 + 1e-5 * o["err"]
            _same(r, q, o)
