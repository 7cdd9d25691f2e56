"""Solves beside other work: two host threads on two handles and streams."""
import threading

import numpy as np
import pytest

import spectra

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2504_04609_gb300 import otlm as api  # noqa: E402


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
