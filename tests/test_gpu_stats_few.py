"""Cluster sums when few labels change: none, one, as many as are still moved
one by one and one more (by number, per cluster and by coordinates), with D on
both sides of a warp's width.  Labels, update, counts (through the objective)
against the FP64 oracle as in test_gpu_parity (same tolerances)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from test_gpu_parity import kp, lockstep  # noqa: E402,F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,K,moved", [(3, 2, 0), (3, 2, 1), (5, 2, 16), (5, 2, 17), (17, 8, 64), (17, 8, 65),
                                       (64, 200, 1024), (64, 200, 1025), (200, 100, 655), (200, 100, 656),
                                       (256, 80, 512), (256, 80, 513)])
def test_few_moves(kp, D, K, moved):  # noqa: F811
    """Clusters along the first axis, every pile a little to the left of its
    centroid; `moved` points sit just on its side of the border to the next
    cluster, which the first update pulls to the left."""
    rng = np.random.default_rng(D + moved)
    N = max(16 * moved + 16, 8 * K)
    C0 = np.zeros((K, D), np.float32)
    C0[:, 0] = 8.0 * np.arange(K)
    k = np.arange(N) % K
    X = C0[k] + 0.25 * rng.integers(-2, 3, size=(N, D)).astype(np.float32)
    X[:, 0] = C0[k, 0] - 1.0
    j = np.flatnonzero(k % 2 == 0)[:moved]
    X[j, 0] = C0[k[j], 0] + 3.875  # nearer to their own now, to the neighbour after the update
    for algo in (kp.KM_ALGO_FILTERED, kp.KM_ALGO_LLOYD):
        lockstep(kp, X, C0, max(1, K // 10), 4, algo=algo)
