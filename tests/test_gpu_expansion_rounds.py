"""Expansion applies of the uneven batch in one round of row blocks and in several: a handle for large
problems keeps the scratch small where a larger one would cost a CTA its place on the SM.  The rounds
change no sum, so the results are equal to the bit; one of them is held to the oracle at the FP32 path's
relative L1 error of 1e-5."""
import numpy as np
import pytest

import oracle
import spectra

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2504_04609_gb300 import otlm as api  # noqa: E402


def _solve(d, n, k, eps, cta, n_max, k_max, T):
    rb = api.ragged_batch([dict(n=n, k=k, eps=eps, x=d["x"], D=d["D"], y=y) for y in d["y"]])
    B = len(d["y"])
    w = torch.tensor(spectra.initial_weights(d["y"], d["D"]).astype(np.float32).ravel(), device="cuda")
    t, err = torch.empty_like(rb.y), torch.empty(B, device="cuda")
    it, st = (torch.empty(B, dtype=torch.int32, device="cuda") for _ in range(2))
    h = api.Handle(n_max, k_max, B, "fp32", "l2", "l2sq", T, 0.0, stream=torch.cuda.current_stream().cuda_stream, ragged_cta=cta)
    h.solve_ragged(rb, 1.0, 1e-3, w, None, t, it, err, st)
    torch.cuda.synchronize()
    h.close()
    assert np.all(st.cpu().numpy() == api.MAX_ITER)
    return w.cpu().numpy().reshape(B, k), t.cpu().numpy().reshape(B, n)


@pytest.mark.parametrize("cta", [128, 256])
@pytest.mark.parametrize("n,eps", [(128, 1e-1), (1025, 1e-2), (1500, 2e-3), (2048, 8e-4)])  # 3, 9, 18 and 28 blocks
@pytest.mark.parametrize("k_max", [20, 256])
def test_rounds_of_row_blocks(cta, n, eps, k_max):
    T, k = 6, 20
    d = spectra.batch(75, 2, n, k, 3)
    w1, t1 = _solve(d, n, k, eps, cta, n, k, T)          # all row blocks in one round
    w, t = _solve(d, n, k, eps, cta, 4096, k_max, T)
    assert np.array_equal(w, w1) and np.array_equal(t, t1)
    D, y = d["D"].astype(np.float64), d["y"][0].astype(np.float64)
    o = oracle.solve_log(spectra.squared_cost(d["x"].astype(np.float64)), D, y, float(np.float32(eps)), 1.0, 1e-3, "l2", "l2sq",
                         spectra.initial_weights(y, D), T)
    assert np.abs(w[0] - o["w"]).sum() <= 1e-5 * np.abs(o["w"]).sum()
    assert np.abs(t[0] - o["t"]).sum() <= 1e-5 * np.abs(o["t"]).sum()
