"""The drift of the centroids (it ages the filters' bounds) at the ends of FP32's
range: squares that FP32 cannot hold.  max_drift is the FP64 norm of the move
rounded up to FP32: no smaller, and larger by a rounding or two of FP32 and the
inflation for the FP64 sum (4e-16) only, 2^-22 together."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from test_gpu_parity import kp  # noqa: E402,F401


@pytest.mark.gpu
@pytest.mark.parametrize("scale", [1e-37, 1e-26, 1e-21, 1e-19, 1e-18, 1.0, 1e18, 3e19, 1e25, 1e36])
@pytest.mark.parametrize("algo", [0, 1])
def test_max_drift(kp, scale, algo):  # noqa: F811
    rng = np.random.default_rng(2)
    X = (rng.normal(size=(96, 5)) * scale).astype(np.float32)
    C0 = X[:1].copy()
    km = kp.KMeans(torch.from_numpy(X).cuda(), torch.from_numpy(C0).cuda(), 1, algo=algo)
    st = km.iterate()
    C = np.empty((1, 5), np.float32)
    km.centroids(C)
    km.close()
    d = np.sqrt(((C.astype(np.float64) - C0) ** 2).sum())
    assert d > 0.1 * scale
    assert d <= st["max_drift"] <= d * (1 + 2.0 ** -22), (d, st["max_drift"])
