"""Solves beside other work: two host threads on two handles and streams, calls that do not poll and so
must not wait for the stream, and solves captured into a graph, on grids with and without a block plan.  Bar of the results:
the FP32 path's relative L1 error of 1e-5."""
import threading

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


def _problem(B, n, k, grid="uniform"):
    d = spectra.batch(74, min(B, 3), n, k, 3)
    x, D, y = d["x"], d["D"], d["y"][np.arange(B) % min(B, 3)]
    if grid == "unsorted":
        perm = np.random.default_rng(7).permutation(n)
        x, D, y = x[perm], D[perm], y[:, perm]
    c = np.ascontiguousarray
    x, D, y = c(x), c(D), c(y)
    return x, D, y, spectra.initial_weights(y, D).astype(np.float32)


def _dev(*arrays):
    return [torch.tensor(a, device="cuda") for a in arrays]


def _compare(w, t, x, D, y, eps, T, penalty="l2sq", alpha=1e-3):
    C, D64 = spectra.squared_cost(x.astype(np.float64)), D.astype(np.float64)
    for p in {0, min(len(y), 3) - 1}:
        y64 = y[p].astype(np.float64)
        o = oracle.solve_log(C, D64, y64, eps, 1.0, alpha, "l2", penalty, spectra.initial_weights(y64, D64), T)
        for q in (p, (len(y) - 1 - p) // 3 * 3 + p):  # the first and the last copy
            assert rel_l1(w[q].cpu().numpy(), o["w"]) <= TOL32 and rel_l1(t[q].cpu().numpy(), o["t"]) <= TOL32


@pytest.mark.parametrize("kind,sizes", [("shared", (16000, 5000)), ("shared", (2000, 600)), ("ragged", (4000, 600))])
def test_two_threads_with_different_sizes(kind, sizes):
    """Each thread repeats one solve on its own handle and stream; every call succeeds with one result."""
    failures, barrier = [], threading.Barrier(2)

    def work(n, reps):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                x, D, y, w0 = _problem(1, n, 16)
                w0_d, t = torch.tensor(w0, device="cuda"), torch.empty(1, n, device="cuda")
                w, first = w0_d.clone(), None
                h = api.Handle(n, 16, 1, "fp32", "l2", "l2sq", 12, 0.0, 6, stream=torch.cuda.current_stream().cuda_stream)
                if kind == "shared":
                    xd, Dd, yd = _dev(x, D, y)
                    call = lambda: h.solve(xd, Dd, yd, 1e-2, 1.0, 1e-3, w, None, t)  # noqa: E731
                else:
                    rb = api.ragged_batch([dict(n=n, k=16, eps=1e-2, x=x, D=D, y=y[0])])
                    it, st = (torch.empty(1, dtype=torch.int32, device="cuda") for _ in range(2))
                    err = torch.empty(1, device="cuda")
                    call = lambda: h.solve_ragged(rb, 1.0, 1e-3, w, None, t, it, err, st)  # noqa: E731
                barrier.wait(60)
                for _ in range(reps):
                    w.copy_(w0_d)
                    call()
                    torch.cuda.current_stream().synchronize()
                    first = w.clone() if first is None else first
                    assert torch.equal(w, first)
                h.close()
        except Exception as e:  # noqa: BLE001
            failures.append((n, repr(e)))
            barrier.abort()

    threads = [threading.Thread(target=work, args=(n, 150)) for n in sizes]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not failures, failures


def _busy_stream():
    """About 0.2 s of work on the current stream and an event behind it."""
    torch.cuda._sleep(400_000_000)
    ev = torch.cuda.Event()
    ev.record()
    return ev


@pytest.mark.parametrize("grid", ["uniform", "unsorted"])
@pytest.mark.parametrize("B,n", [(2, 300), (700, 300), (4, 3000), (1, 8192)])
def test_solve_that_never_polls_does_not_wait(B, n, grid):
    T = 6
    x, D, y, w0 = _problem(B, n, 12, grid)
    xd, Dd, yd, wd = _dev(x, D, y, w0)
    w, t = wd.clone(), torch.empty(B, n, device="cuda")
    h = api.Handle(n, 12, B, "fp32", "l2", "l2sq", T, 0.0, T + 1, stream=torch.cuda.current_stream().cuda_stream)
    h.solve(xd, Dd, yd, 2e-2, 1.0, 1e-3, w, None, t)  # loads the kernels
    torch.cuda.synchronize()
    w.copy_(wd)
    ev = _busy_stream()
    h.solve(xd, Dd, yd, 2e-2, 1.0, 1e-3, w, None, t)
    returned_early = not ev.query()
    torch.cuda.synchronize()
    h.close()
    assert returned_early
    _compare(w, t, x, D, y, 2e-2, T)


@pytest.mark.parametrize("n", [300, 3000])
def test_noalloc_that_never_polls_does_not_wait(n):
    """otlm_solve_noalloc polls every eight iterations."""
    x, D, y, w0 = _problem(3, n, 12)
    xd, Dd, yd, wd = _dev(x, D, y, w0)
    w, t, g = wd.clone(), torch.empty(3, n, device="cuda"), torch.zeros(3, n, device="cuda")
    args = (xd, Dd, yd, 2e-2, 1.0, 1e-3, "l2", "l2sq", 7, 0.0, w, g, t, None, None, None,
            torch.cuda.current_stream().cuda_stream)
    assert api.solve_noalloc(*args) == api.OTLM_OK
    torch.cuda.synchronize()
    w.copy_(wd)
    g.zero_()
    ev = _busy_stream()
    assert api.solve_noalloc(*args) == api.OTLM_OK
    returned_early = not ev.query()
    torch.cuda.synchronize()
    assert returned_early
    _compare(w, t, x, D, y, 2e-2, 7)


@pytest.mark.parametrize("grid", ["uniform", "unsorted"])
@pytest.mark.parametrize("B,n", [(2, 300), (700, 300), (4, 3000), (1, 8192)])
def test_captured_solve(B, n, grid):
    """A solve without polls captured into a graph and replayed on other targets than it was captured
    with: the host cannot read the grid's plan, and the kernels follow it on the device."""
    T = 6
    x, D, y, w0 = _problem(B, n, 12, grid)
    xd, Dd, yd, wd = _dev(x, D, y, w0)
    w, t, y_in = wd.clone(), torch.empty(B, n, device="cuda"), torch.ones_like(yd)
    s = torch.cuda.Stream()
    h = api.Handle(n, 12, B, "fp32", "l2", "l2sq", T, 0.0, T + 1, stream=s.cuda_stream)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=s):
        h.solve(xd, Dd, y_in, 2e-2, 1.0, 1e-3, w, None, t)
    y_in.copy_(yd)
    for _ in range(2):
        w.copy_(wd)
        t.zero_()
        graph.replay()
    torch.cuda.synchronize()
    h.close()
    _compare(w, t, x, D, y, 2e-2, T)
