"""The FP32 dense pass where its tiling can go wrong: every padded width (a
row on one, two or four lanes), dimensions that are no multiple of the width
or of a 16-byte load, one or several points per lane, ragged last tiles, an
odd number of centroids, centroids that do not fit the shared-memory tile,
group bounds that do not fit theirs, groups of one centroid, and exact ties.
Labels, update, objective and bounds against the FP64 oracle as in
test_gpu_parity (same tolerances)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1905_09345_gb300 import synth  # noqa: E402
from test_gpu_parity import kp, lockstep  # noqa: E402,F401

pytestmark = pytest.mark.gpu

# fewer than 77824 points: one per lane; from there on four lane-slots
SHAPES = [(n, d, 9, 3) for n in (513, 77824 + 129) for d in (1, 4, 7, 12, 16, 17, 24, 27, 32, 33, 48, 50, 64, 65, 100, 128)]
SHAPES += [(1, 5, 1, 1), (700, 6, 301, 301), (1030, 129, 21, 4), (3001, 20, 1001, 100), (78337, 50, 300, 7)]


@pytest.mark.parametrize("N,D,K,G", SHAPES, ids=[f"N{s[0]}_D{s[1]}_K{s[2]}_G{s[3]}" for s in SHAPES])
def test_dense_fp32_lockstep(kp, N, D, K, G):  # noqa: F811
    rng = np.random.default_rng(N + 1000 * D + K)
    X, _ = synth.gaussian_mixture(rng, N, D, min(K, 32), centre_range=4.0, scale="blob_uniform",
                                  scale_args=(0.5, 2.0))
    C0 = synth.sample_init(rng, X, K)
    for algo in (kp.KM_ALGO_FILTERED, kp.KM_ALGO_LLOYD):
        lockstep(kp, X, C0, G, 2, algo=algo, dense=kp.KM_DENSE_FP32, check_bounds=N * K < 800_000)


@pytest.mark.parametrize("D", [3, 17, 40, 96])
def test_dense_fp32_ties(kp, D):  # noqa: F811
    """Small integers: points at equal distances from several centroids."""
    rng = np.random.default_rng(D)
    X = rng.integers(0, 2, size=(1500, D)).astype(np.float32)
    C0 = np.concatenate([X[:20], X[:12]]).astype(np.float32)
    for grouping in (kp.KM_GROUP_CONTIGUOUS, kp.KM_GROUP_CLUSTERED):
        lockstep(kp, X, C0, 5, 2, dense=kp.KM_DENSE_FP32, check_bounds=True, grouping=grouping)


@pytest.mark.parametrize("N,D,K,G", [(2000, 130, 33, 4), (1537, 200, 64, 6), (900, 401, 21, 21), (5000, 256, 130, 13),
                                     (700, 1000, 9, 2)])
def test_dense_fp32_wide(kp, N, D, K, G):  # noqa: F811
    """Rows of more than 128 coordinates, and exact ties among them."""
    rng = np.random.default_rng(N + D)
    X, _ = synth.gaussian_mixture(rng, N, D, min(K, 32), centre_range=4.0, scale="blob_uniform",
                                  scale_args=(0.5, 2.0))
    Y = rng.integers(0, 2, size=(400, D)).astype(np.float32)
    Y[:, 20:] = 0.0
    for algo in (kp.KM_ALGO_FILTERED, kp.KM_ALGO_LLOYD):
        lockstep(kp, X, synth.sample_init(rng, X, K), G, 3, algo=algo, check_bounds=N * K < 150_000)
        lockstep(kp, Y, Y[:K].copy(), G, 2, algo=algo, check_bounds=True)
