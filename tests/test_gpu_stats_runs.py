"""The cluster sums where their runs and batches can go wrong: fewer points than
a batch, runs that end with a cluster, clusters of one point, every number of
coordinates per lane, D at and beside multiples of 32.
Update, objective and labels against the FP64 oracle as in test_gpu_parity
(same tolerances)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1905_09345_gb300 import synth  # noqa: E402
from test_gpu_parity import kp, lockstep  # noqa: E402,F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [1, 31, 32, 33, 64, 65, 100, 129, 200, 256])
@pytest.mark.parametrize("N,K", [(1, 1), (7, 3), (8, 8), (65, 2), (3000, 700)])
def test_stats_runs(kp, N, K, D):  # noqa: F811
    rng = np.random.default_rng(N * 1000 + D)
    X, _ = synth.gaussian_mixture(rng, N, D, min(K, 16), centre_range=3.0, scale="blob_uniform",
                                  scale_args=(0.5, 2.0))
    C0 = synth.sample_init(rng, X, K)
    for algo in (kp.KM_ALGO_FILTERED, kp.KM_ALGO_LLOYD):
        lockstep(kp, X, C0, max(1, K // 10), 4, algo=algo)
