"""k-means++ seeding where device memory is short: 8 bytes of scratch per point
have to do.  In a process of its own, whose memory pool is empty, with all but
12 bytes per point of the device's memory taken."""
import os
import subprocess
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import sys
import numpy as np
import torch
from paper_1905_09345_gb300 import kpynq as kp
N, D, K = (int(a) for a in sys.argv[1:4])
X = torch.from_numpy(np.load(sys.argv[4] + "/X.npy")).cuda()
u = np.load(sys.argv[4] + "/u.npy")
C = torch.empty(K, D, device="cuda")
idx = torch.empty(K, dtype=torch.int64, device="cuda")
kp.kmeans_init_kmeanspp(X, 1000, D, K, u, C, idx)  # everything loaded
free, _ = torch.cuda.mem_get_info()
filler = torch.empty(free - 12 * N, dtype=torch.uint8, device="cuda")
kp.kmeans_init_kmeanspp(X, N, D, K, u, C, idx)
np.save(sys.argv[4] + "/idx.npy", idx.cpu().numpy())
"""


@pytest.mark.gpu
@pytest.mark.parametrize("N,D,K", [(1 << 24, 1, 12), ((1 << 23) + 1, 4, 12)])
def test_eight_bytes_a_point(N, D, K, tmp_path):
    oracle.build()
    rng = np.random.default_rng(N)
    X = (rng.normal(size=(N, D)) * 5.0 + rng.integers(0, 30, size=(N, 1)) * 40.0).astype(np.float32)
    u = rng.uniform(size=K)
    np.save(tmp_path / "X.npy", X)
    np.save(tmp_path / "u.npy", u)
    r = subprocess.run([sys.executable, "-c", CHILD, str(N), str(D), str(K), str(tmp_path)], cwd=ROOT,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-1500:]
    ref, _ = oracle.kmeanspp(X.astype(np.float64), K, u)
    assert np.array_equal(np.load(tmp_path / "idx.npy"), ref)


@pytest.mark.gpu
def test_more_points_than_32_bits_count(kp_lib):
    """2^32 points at the largest distance: with a 32-bit count of them, zero, the
    weights would be scaled by the one point that is nearer."""
    N, K = 2 ** 32 + 2, 2
    if torch.cuda.mem_get_info()[0] < 16 * N:
        pytest.skip("needs 64 GB of device memory")
    X = torch.ones(N, 1, device="cuda")
    X[0], X[1] = 0.0, 0.5
    C = torch.empty(K, 1, device="cuda")
    idx = torch.empty(K, dtype=torch.int64, device="cuda")
    kp_lib.kmeans_init_kmeanspp(X, N, 1, K, np.array([0.0, 0.25]), C, idx)
    assert idx.tolist() == [0, 1 + 2 ** 30]
    assert C.flatten().tolist() == [0.0, 1.0]


@pytest.fixture
def kp_lib():
    from paper_1905_09345_gb300 import build, kpynq
    build.build()
    yield kpynq
    torch.cuda.empty_cache()
