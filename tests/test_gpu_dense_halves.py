"""The one-accumulator tensor-core pass (K <= 256) where its two column halves
meet: no column or group of the second half, the border inside and between
groups, four groups that share a 16-byte store, more than 64 groups, groups of
one centroid, the most groups that fit shared memory, ragged last tiles and
several tiles per scanning warp.  Labels, update, objective and bounds against
the FP64 oracle as in test_gpu_parity (same tolerances)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1905_09345_gb300 import synth  # noqa: E402
from test_gpu_parity import kp, lockstep  # noqa: E402,F401

pytestmark = pytest.mark.gpu

MOST = 88  # of 256 centroids in 64 dimensions: one stage of points is left
SHAPES = [(130, 64, 1, 1), (257, 32, 16, 5), (300, 64, 17, 17), (1000, 32, 33, 6), (640, 128, 96, 7), (2001, 64, 112, 13),
          (777, 64, 200, 64), (777, 64, 200, 65), (900, 64, 256, MOST), (97357, 32, 50, 9), (5000, 128, 224, 22)]


@pytest.mark.parametrize("N,D,K,G", SHAPES, ids=[f"N{s[0]}_D{s[1]}_K{s[2]}_G{s[3]}" for s in SHAPES])
def test_halves_lockstep(kp, N, D, K, G):  # noqa: F811
    rng = np.random.default_rng(N + K)
    X, _ = synth.gaussian_mixture(rng, N, D, min(K, 32), centre_range=5.0, scale="blob_uniform",
                                  scale_args=(0.5, 2.0))
    C0 = synth.sample_init(rng, X, K)
    for algo in (kp.KM_ALGO_FILTERED, kp.KM_ALGO_LLOYD):
        lockstep(kp, X, C0, G, 3, algo=algo, check_bounds=algo == kp.KM_ALGO_FILTERED and N * K < 800_000)


@pytest.mark.parametrize("big_first", [True, False])
def test_halves_clustered(kp, big_first):  # noqa: F811
    """Groups of very different sizes: one that spans the border, the others
    single centroids on one side of it."""
    rng = np.random.default_rng(11 + big_first)
    D, K, G, N = 64, 220, 40, 4000
    far = rng.uniform(-1000.0, 1000.0, size=(G - 1, D)).astype(np.float32)
    near = rng.normal(size=(K - G + 1, D)).astype(np.float32)
    C0 = np.concatenate([near[:1], far, near[1:]] if big_first else [far, near])
    X = (C0[rng.integers(0, K, size=N)] + 0.3 * rng.normal(size=(N, D))).astype(np.float32)
    X[:K] = C0
    for algo in (kp.KM_ALGO_FILTERED, kp.KM_ALGO_LLOYD):
        lockstep(kp, X, C0, G, 3, algo=algo, check_bounds=algo == kp.KM_ALGO_FILTERED,
                 grouping=kp.KM_GROUP_CLUSTERED)
