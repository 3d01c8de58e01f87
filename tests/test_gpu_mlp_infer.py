"""The fused inference kernel at the edges of its tiles: one row, ragged and
odd numbers of tiles (a group without work, more than one tile per group),
widths and class counts around the multiples of 16, 64 and 256, rows that do
not allow 16-byte loads.  Against O3 at the bfloat16 values of weights and
inputs: the predicted class's logit is within 1e-2 of the logit scale of the
largest (the bfloat16 activations move a logit by less, see test_gpu_mlp), and
is the argmax where the two largest are further apart than that."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp  # noqa: E402
from test_gpu_mlp import at_compute_precision, bf, dev, kp, random_params  # noqa: E402,F401

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 16, 1), (127, 8, 64, 2), (128, 17, 65, 16), (129, 64, 1, 17), (257, 65, 128, 255),
          (4000, 256, 256, 256), (1001, 33, 200, 257), (300, 128, 256, 512), (2 * 152 * 128 + 77, 12, 32, 40)]


@pytest.mark.parametrize("N,D,H,C", SHAPES, ids=[f"N{s[0]}_D{s[1]}_H{s[2]}_C{s[3]}" for s in SHAPES])
def test_predict_edges(kp, N, D, H, C):  # noqa: F811
    rng = np.random.default_rng(N + D + H + C)
    params = random_params(D, H, C, seed=C)
    X = rng.normal(0, 2.0, (N, D)).astype(np.float32)
    logits, _ = mlp.forward(at_compute_precision(params), bf(X))
    net = kp.MLP(D, H, C)
    net.set_params({k: dev(v) for k, v in params.items()})
    pred = torch.full((N + 1,), -7, dtype=torch.int32, device="cuda")
    net.predict(dev(X), pred[:N])
    net.close()
    got = pred.cpu().numpy()
    assert got[N] == -7  # nothing past the rows
    got = got[:N]
    assert got.min() >= 0 and got.max() < C
    scale = np.abs(logits).max(axis=1) + 1.0
    assert np.all(logits[np.arange(N), got] >= logits.max(axis=1) - 1e-2 * scale)
    if C > 1:
        srt = np.sort(logits, axis=1)
        clear = (srt[:, -1] - srt[:, -2]) > 1e-2 * scale
        assert np.array_equal(got[clear], np.argmax(logits, axis=1)[clear])
