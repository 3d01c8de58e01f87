"""Near-ties behind the tensor-core pass: points halfway between two centroids
(within a few FP32 roundings), exactly halfway, and between three, so that
FP32 cannot order the nearest ones; every width of the settle kernel, group
masks, bounds windows over more than 32 and 64 groups, centroids in shared and
in global memory, groups of one centroid.  Labels, update, objective and
bounds against the FP64 oracle as in test_gpu_parity (same tolerances)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from test_gpu_parity import kp, lockstep  # noqa: E402,F401

pytestmark = pytest.mark.gpu

SHAPES = [(32, 40, 4), (64, 64, 6), (64, 256, 100), (64, 130, 130), (128, 256, 25), (32, 300, 30), (64, 700, 70),
          (128, 400, 129)]


@pytest.mark.parametrize("D,K,G", SHAPES, ids=[f"D{s[0]}_K{s[1]}_G{s[2]}" for s in SHAPES])
@pytest.mark.parametrize("kind", ["rounded", "exact", "three"])
def test_settle_near_ties(kp, D, K, G, kind):  # noqa: F811
    rng = np.random.default_rng(D * 7 + K + len(kind))
    if kind == "rounded":
        C0 = rng.normal(size=(K, D)).astype(np.float32)
    else:  # eighths: sums and halves are exact
        C0 = (rng.integers(-16, 17, size=(K, D)) / 8).astype(np.float32)
    N = 1200
    a, b, c = (rng.integers(0, K, size=N) for _ in range(3))
    if kind == "three":  # equal distances along an axis where three centroids were put in a row
        C0[1], C0[2] = C0[0], C0[0]
        C0[1, 0] += 2.0
        C0[2, 1] += 2.0
        X = np.repeat(C0[:1], N, 0)
        X[:, :2] += 1.0
        X[:, 2:] += (rng.integers(-1, 2, size=(N, D - 2)) / 64).astype(np.float32)
    else:
        X = ((C0[a].astype(np.float64) + C0[b]) / 2).astype(np.float32)
        if kind == "rounded":
            X = np.nextafter(X, C0[c]).astype(np.float32)
    X[:K] = C0
    for algo in (kp.KM_ALGO_FILTERED, kp.KM_ALGO_LLOYD):
        lockstep(kp, X, C0, G, 2, algo=algo, check_bounds=algo == kp.KM_ALGO_FILTERED)
