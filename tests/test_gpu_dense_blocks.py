"""The streamed-centroid tensor-core pass (K > 256) where its tiling can go
wrong: the border between the two halves of the centroids, odd numbers of
64- and 128-column blocks, groups of one to three centroids (several closing
among four columns), a ragged last tile, a last tile without a partner, and
clustered groups of one centroid each in a row.  Labels, update, objective and
bounds against the FP64 oracle as in test_gpu_parity (same tolerances)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1905_09345_gb300 import synth  # noqa: E402
from test_gpu_parity import kp, lockstep  # noqa: E402,F401

pytestmark = pytest.mark.gpu

SHAPES = [(300, 64, 257, 128), (129, 32, 128 + 129, 86), (4000, 128, 385, 33), (6001, 64, 577, 192),
          (3000, 32, 1025, 410), (2 * 128 * 152 + 300, 32, 300, 30)]


@pytest.mark.parametrize("N,D,K,G", SHAPES, ids=[f"N{s[0]}_D{s[1]}_K{s[2]}_G{s[3]}" for s in SHAPES])
@pytest.mark.parametrize("algo", [0, 1])
def test_blocks_lockstep(kp, N, D, K, G, algo):  # noqa: F811
    rng = np.random.default_rng(N + K)
    N = max(N, K)
    X, _ = synth.gaussian_mixture(rng, N, D, min(K, 64), centre_range=10.0, scale="blob_uniform",
                                  scale_args=(0.5, 2.0))
    C0 = synth.sample_init(rng, X, K)
    lockstep(kp, X, C0, G, 3, algo=algo, check_bounds=N * K < 4_000_000)


def test_clustered_singletons(kp):  # noqa: F811
    """Over a hundred groups of one centroid in adjacent columns, then one of
    several hundred: more groups close among 64 columns than the contiguous
    grouping could."""
    rng = np.random.default_rng(7)
    D, K, G, N = 64, 500, 130, 4000
    far = rng.uniform(-1000.0, 1000.0, size=(G - 1, D)).astype(np.float32)
    near = rng.normal(size=(K - G + 1, D)).astype(np.float32)
    C0 = np.concatenate([far, near])
    X = (C0[rng.integers(0, K, size=N)] + 0.3 * rng.normal(size=(N, D))).astype(np.float32)
    X[:K] = C0
    for algo in (kp.KM_ALGO_FILTERED, kp.KM_ALGO_LLOYD):
        st = lockstep(kp, X, C0, G, 3, algo=algo, check_bounds=algo == kp.KM_ALGO_FILTERED,
                      grouping=kp.KM_GROUP_CLUSTERED)
        assert st[0]["path"] == kp.KM_PATH_DENSE_TC


@pytest.mark.parametrize("D,K", [(32, 900), (32, 1025), (128, 900)])
def test_last_pair_lacks_second_tile(kp, D, K):  # noqa: F811
    """Three tiles per CTA and four or more centroid blocks per half: the last
    pair has one tile, and the norms' slots are filled again while nobody waits
    for the second tile's warps block by block."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    N = 3 * 128 * sms - 77
    rng = np.random.default_rng(K + D)
    X, _ = synth.gaussian_mixture(rng, N, D, 64, centre_range=10.0, scale="blob_uniform", scale_args=(0.5, 2.0))
    C0 = synth.sample_init(rng, X, K)
    st = lockstep(kp, X, C0, K // 10, 2, algo=kp.KM_ALGO_LLOYD, check_bounds=False)
    assert all(s["path"] == kp.KM_PATH_DENSE_TC for s in st)
