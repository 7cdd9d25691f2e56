"""Training contractions at sizes off the GEMM's tiles: one row, batches around the 128-row tile,
reductions shorter than one k block, widths and outputs that are not multiples of four, and two sizes
in turn on one network (the smaller must not see the larger one's operands).  Bar, layer by layer: the
2-norm of the error at most 1e-5 of the 2-norm of the entries' sums of absolute term values through
the chain rule (oracle.mlp.grad_magnitudes): FP32 accumulation errs by about sqrt(K) 2^-24 of it
(K <= 400: 1.2e-6), and a unit whose GELU' happens to be near 0, known to 2^-24 absolutely only, weighs
little in a norm."""
import numpy as np
import pytest

from oracle import mlp as ref

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2504_04609_gb300 import otlm as api  # noqa: E402


def _check(net, n, k, H, B, seed):
    rng = np.random.default_rng(seed)
    y = rng.uniform(0.0, 1.0, (B, n)).astype(np.float32)
    y[:, :2] = 0.0
    t = rng.normal(-5, 2, (B, n + k)).astype(np.float32)
    t[:, 1] = -np.inf
    mean, std = rng.normal(-5, 1, n + k).astype(np.float32), rng.uniform(1, 3, n + k).astype(np.float32)
    dev = lambda a: torch.tensor(a, device="cuda")  # noqa: E731
    net.set_normalization(dev(mean), dev(std))
    params, grads = (torch.empty(net.num_params, device="cuda") for _ in range(2))
    loss = torch.empty(1, device="cuda")
    net.get_params(params)
    net.gradients(dev(y), dev(t), grads, loss)
    torch.cuda.synchronize()
    p = params.cpu().numpy().astype(np.float64)
    args = (p, ref.layer_dims(n, k, H), y, t, mean.astype(np.float64), std.astype(np.float64))
    lo, go = ref.loss_and_grad(*args, round_weights=True)
    mag = ref.grad_magnitudes(*args, round_weights=True)
    assert loss.item() == pytest.approx(lo, rel=1e-5)
    got, off = grads.cpu().numpy().astype(np.float64), 0
    dims = ref.layer_dims(n, k, H)
    for a, b in zip(dims[:-1], dims[1:]):
        for size in (a * b, b):
            q = slice(off, off + size)
            assert np.linalg.norm(got[q] - go[q]) <= 1e-5 * np.linalg.norm(mag[q]), (a, b, size)
            off += size


@pytest.mark.parametrize("n,k,H,batches", [(33, 3, 20, (1, 5)), (130, 7, 45, (129, 31)), (399, 18, 64, (200, 33, 128))])
def test_gradients_at_odd_sizes(n, k, H, batches):
    net = api.WarmStart(n, k, H, max(batches), seed=5)
    for i, B in enumerate(batches):
        _check(net, n, k, H, B, 7 + i)
    net.close()


def test_training_step_follows_the_gradient():
    """One AdamW step from the gradients the same network reports: p - lr (g / (|g| + 1e-8) + wd p)."""
    n, k, H, B = 60, 6, 24, 40
    net = api.WarmStart(n, k, H, B, seed=9)
    rng = np.random.default_rng(3)
    y = torch.tensor(rng.uniform(0.1, 1.0, (B, n)).astype(np.float32), device="cuda")
    t = torch.tensor(rng.normal(0, 1, (B, n + k)).astype(np.float32), device="cuda")
    p0, p1, g = (torch.empty(net.num_params, device="cuda") for _ in range(3))
    net.get_params(p0)
    net.gradients(y, t, g)
    net.train_step(y, t, 1e-3, 1e-2)
    net.get_params(p1)
    torch.cuda.synchronize()
    p0, p1, g = (a.cpu().numpy().astype(np.float64) for a in (p0, p1, g))
    want = p0 - 1e-3 * (g / (np.abs(g) + 1e-8) + 1e-2 * p0)
    # FP32 evaluation of the update: m / bc1 and sqrt(v / bc2) each carry a few 2^-24 relative errors
    assert np.max(np.abs(p1 - want)) <= 1e-3 * 2e-5 + 2.0 ** -23 * np.abs(p0).max()
    net.close()
