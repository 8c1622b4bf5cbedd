"""Screener gradient at the edges of its tiles and of the split over the batch, against the float64
back-propagation: the bounds of test_gradient_matches_oracle (FP32 accumulation, blockwise relative 1e-4), and
for hidden units whose pre-activation vanishes to FP32 rounding, where ReLU's derivative may come out as 0 or 1,
what such a unit adds to each gradient."""
import numpy as np
import pytest
import torch

from oracle import mlp
from paper_2410_04204_gb300 import inputs, tgba

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _kinks(theta, H, x, t, eps=1e-5):
    """What the units with |pre-activation| < eps (FP32 sums of 256 terms) may change in the gradient."""
    W1, b1, W2, b2, w3, b3 = mlp.unflatten(theta, H)
    z1 = x @ W1.T + b1
    h1 = np.maximum(z1, 0.0)
    z2 = h1 @ W2.T + b2
    dy = np.abs(2.0 * (np.maximum(z2, 0.0) @ w3 + b3[0] - t) / len(t))[:, None]
    n1, n2 = np.abs(z1) < eps, np.abs(z2) < eps
    p2 = dy * np.abs(w3) * n2
    p1 = (p2 @ np.abs(W2)) * ((z1 > 0) | n1) + n1 * ((dy * np.abs(w3) * ((z2 > 0) | n2)) @ np.abs(W2))
    return np.concatenate([(p1.T @ np.abs(x)).ravel(), p1.sum(0), (p2.T @ h1).ravel(), p2.sum(0), np.zeros(H + 1)])


@pytest.mark.parametrize("H,B", [(256, 1), (256, 63), (256, 64), (256, 65), (256, 129), (256, 4097), (128, 1000)])
def test_gradient_of_ragged_batches(H, B):
    theta = mlp.init(H, inputs.SEED).astype(np.float32)
    try:
        s = tgba.tgba_screen_create(H, theta)
    except tgba.TgbaError as e:
        assert e.code == tgba.TGBA_EINVAL and H != 256
        pytest.skip("width not taken")
    try:
        g = inputs.rng(B)
        x = g.uniform(-1, 1, (B, mlp.D_IN)).astype(np.float32)
        t = g.normal(-4, 2, B).astype(np.float32)
        grad = torch.full((len(theta),), float("nan"), dtype=torch.float32, device="cuda")
        loss = tgba.tgba_screen_grad(s, torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda(), grad)
        lo, go = mlp.loss_and_grad(theta.astype(np.float64), H, x.astype(np.float64), t.astype(np.float64))
        gg = grad.cpu().numpy()
        kink = _kinks(theta.astype(np.float64), H, x.astype(np.float64), t.astype(np.float64))
        assert abs(loss - lo) <= 1e-5 * lo
        o = 0
        for shape in mlp.shapes(H):
            n = int(np.prod(shape))
            ref = go[o:o + n]
            assert (np.abs(gg[o:o + n] - ref) <= 1e-4 * np.abs(ref).max() + 1e-7 + kink[o:o + n]).all(), shape
            o += n
    finally:
        tgba.tgba_screen_free(s)
