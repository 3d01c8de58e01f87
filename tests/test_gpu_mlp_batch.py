"""The training products at the edges of their tiles and split: batches of one
tile and of more tiles than SMs, widths that leave quarters of the columns
empty or uneven, class counts on both sides of 256 and of the multiples of
16; and a training step recorded in a graph against the same step's gradient.
Tolerances as in test_gpu_mlp."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp  # noqa: E402
from test_gpu_mlp import GRAD_RTOL, NAMES, at_compute_precision, bf, dev, kp, random_params  # noqa: E402,F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,H,C,B", [(17, 65, 16, 256), (65, 200, 17, 384), (256, 256, 512, 512),
                                     (8, 130, 257, 640), (12, 32, 33, 153 * 128)])
def test_gradient_edges(kp, D, H, C, B):  # noqa: F811
    rng = np.random.default_rng(D + H + C + B)
    params = random_params(D, H, C, seed=D + C)
    X = rng.normal(0, 1.5, (B, D)).astype(np.float32)
    y = rng.integers(0, C, B).astype(np.int32)
    loss_ref, g_ref = mlp.loss_and_grad(at_compute_precision(params), bf(X), y)
    net = kp.MLP(D, H, C)
    net.set_params({k: dev(v) for k, v in params.items()})
    grad = torch.full((net.n_params(),), float("nan"), dtype=torch.float32, device="cuda")
    for _ in range(2):  # the second pass finds the plan made
        loss = net.gradient(dev(X), dev(y, np.int32), grad)
        g = net.split(grad.cpu().numpy().astype(np.float64))
        assert abs(loss - loss_ref) <= GRAD_RTOL * loss_ref, (loss, loss_ref)
        for k in NAMES:
            err = float(np.abs(g[k] - g_ref[k]).max())
            assert err <= GRAD_RTOL * float(np.abs(g_ref[k]).max()), k
    net.close()


def test_batch_size_changes(kp):  # noqa: F811
    """Gradients of batches of different sizes, in turn, on one network."""
    D, H, C = 16, 64, 20
    rng = np.random.default_rng(2)
    params = random_params(D, H, C, seed=4)
    net = kp.MLP(D, H, C)
    net.set_params({k: dev(v) for k, v in params.items()})
    for B in (256, 1024, 128, 256):
        X = rng.normal(0, 1.5, (B, D)).astype(np.float32)
        y = rng.integers(0, C, B).astype(np.int32)
        _, g_ref = mlp.loss_and_grad(at_compute_precision(params), bf(X), y)
        grad = torch.empty(net.n_params(), dtype=torch.float32, device="cuda")
        net.gradient(dev(X), dev(y, np.int32), grad)
        g = net.split(grad.cpu().numpy().astype(np.float64))
        for k in NAMES:
            assert float(np.abs(g[k] - g_ref[k]).max()) <= GRAD_RTOL * float(np.abs(g_ref[k]).max()), (B, k)
    net.close()
