"""k-means++ seeding at the edges of its filter, lists and weights: chunk and
warp remainders, odd and long rows, misaligned points, distances over many
binary orders of magnitude (the weights' scale then falls by more than one
step at a time, and past the stored bits), subnormal coordinates, points far
from the origin.  The indices must equal O4's bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kp():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1905_09345_gb300 import build, kpynq
    build.build()
    oracle.build()
    return kpynq


def check(kp, X, K, seed, shift=0):
    """shift: floats by which the device copy of X is misaligned."""
    N, D = X.shape
    u = np.random.default_rng(seed).uniform(size=K)
    buf = torch.empty(N * D + shift, dtype=torch.float32, device="cuda")
    buf[shift:] = torch.from_numpy(np.ascontiguousarray(X, np.float32)).cuda().reshape(-1)
    C = torch.empty(K, D, dtype=torch.float32, device="cuda")
    idx = torch.empty(K, dtype=torch.int64, device="cuda")
    kp.kmeans_init_kmeanspp(buf[shift:].reshape(N, D), N, D, K, u, C, idx)
    ref, _ = oracle.kmeanspp(X.astype(np.float64), K, u)
    got = idx.cpu().numpy()
    assert np.array_equal(got, ref), np.flatnonzero(got != ref)[:5]
    assert np.array_equal(C.cpu().numpy(), X[ref])


SHAPES = [(1, 1, 1), (2, 5, 2), (31, 4, 31), (33, 8, 20), (1000, 1, 30), (4097, 12, 40), (131073, 3, 20),
          (131072, 8, 25), (20000, 129, 30), (9000, 260, 25), (300, 4096, 12), (600000, 4, 12)]


@pytest.mark.parametrize("N,D,K", SHAPES, ids=[f"N{s[0]}_D{s[1]}_K{s[2]}" for s in SHAPES])
def test_shapes(kp, N, D, K):
    rng = np.random.default_rng(N + D)
    X = (rng.normal(size=(N, D)) * rng.uniform(0.1, 10.0, size=(1, D))).astype(np.float32)
    check(kp, X, K, seed=D)
    if N < 50000:
        check(kp, X, K, seed=D + 1, shift=1)


@pytest.mark.parametrize("span", [6, 40, 120])
def test_scales(kp, span):
    """Points at distances 2^0 .. 2^-span: each centre removes the largest."""
    rng = np.random.default_rng(span)
    N, D = 3000, 6
    X = rng.normal(size=(N, D)) * np.exp2(-rng.uniform(0, span, size=(N, 1)))
    check(kp, X.astype(np.float32), 120, seed=1)


def test_far_from_origin_and_subnormal(kp):
    rng = np.random.default_rng(5)
    X = (rng.normal(size=(5000, 16)) * 1e-2 + 1e4).astype(np.float32)
    X[rng.integers(0, 5000, size=1500)] = X[7]  # many duplicates
    check(kp, X, 60, seed=2)
    Y = rng.normal(size=(2000, 5)).astype(np.float32)
    Y[:, 2] = (rng.integers(0, 50, size=2000) * 2.0 ** -149).astype(np.float32)  # subnormal coordinates
    Y[::3, 0] = 0.0
    check(kp, Y, 50, seed=3)
    check(kp, np.zeros((500, 3), np.float32), 20, seed=4)  # every weight zero


@pytest.mark.parametrize("N,D,K", [(6000, 3, 1100), (5000, 20, 400), (70000, 32, 64)])
@pytest.mark.parametrize("kind", ["blobs", "line", "copies"])
def test_bound_alone(kp, N, D, K, kind):
    """The filter by the bound alone where it skips nearly everything, more
    centres than its table holds, points and centres on a line (the triangle
    inequality holds with equality there) and many copies of few points."""
    rng = np.random.default_rng(N + D)
    if kind == "blobs":
        X = rng.normal(size=(50, D))[rng.integers(0, 50, size=N)] * 100.0 + rng.normal(size=(N, D))
    elif kind == "line":
        X = rng.integers(0, 4096, size=(N, 1)) * np.ones((1, D))
    else:
        X = rng.integers(-2, 3, size=(max(K // 2, 2), D))[rng.integers(0, max(K // 2, 2), size=N)]
    check(kp, X.astype(np.float32), K, seed=K)


def weights_reference(X, K, u):
    """The draw of the header with Python integers.  A NaN distance never becomes
    the smallest and weighs nothing; an infinite one weighs 2^64 - 1, sums modulo
    2^64."""
    N = len(X)
    X = X.astype(np.float64)
    d = np.full(N, np.nan)
    idx = []
    for j in range(K):
        pick = min(int(np.floor(u[j] * N)), N - 1)
        w = d[~np.isnan(d)].max(initial=0.0)
        if w > 0:
            e = 1025 if np.isinf(w) else np.frexp(w)[1]
            q = [0 if np.isnan(v) else (2 ** 64 - 1 if np.isinf(v) else int(np.floor(np.ldexp(v, 32 - e)))) for v in d]
            W = sum(q) % 2 ** 64
            if W:
                T = min(int(np.floor(u[j] * float(W))), W - 1)
                run = 0
                for pick in range(N):
                    run = (run + q[pick]) % 2 ** 64
                    if run > T:
                        break
        idx.append(pick)
        s = np.zeros(N)
        with np.errstate(invalid="ignore", over="ignore"):
            for i in range(X.shape[1]):
                t = X[:, i] - X[pick, i]
                s = s + t * t
        d = np.fmin(d, s)
    return np.array(idx)


def check_weights(kp, X, K, seed, u0):
    N, D = X.shape
    u = np.random.default_rng(seed).uniform(size=K) * 0.99
    u[0] = u0
    C = torch.empty(K, D, dtype=torch.float32, device="cuda")
    idx = torch.empty(K, dtype=torch.int64, device="cuda")
    kp.kmeans_init_kmeanspp(torch.from_numpy(X).cuda(), N, D, K, u, C, idx)
    got, ref = idx.cpu().numpy(), weights_reference(X, K, u)
    assert np.array_equal(got, ref), (got, ref)


@pytest.mark.parametrize("where", ["first", "later"])
@pytest.mark.parametrize("scale", [1e-6, 1.0, 1e6])
def test_nan_rows(kp, where, scale):
    """Rows with a NaN: as the first centre one leaves no distance to scale by,
    and the next draw is uniform."""
    rng = np.random.default_rng(3)
    X = (rng.normal(size=(700, 6)) * np.exp2(rng.uniform(-6, 6, size=(700, 1))) * scale).astype(np.float32)
    X[10:700:97, 2] = np.nan
    check_weights(kp, X, 12, 6, (10 if where == "first" else 11) / 700 + 1e-9)
    X[10:20] = np.nan  # (two such centres in a row)
    u = np.concatenate([[10.5 / 700, 12.5 / 700], np.random.default_rng(5).uniform(size=8)])
    C = torch.empty(10, 6, device="cuda")
    idx = torch.empty(10, dtype=torch.int64, device="cuda")
    kp.kmeans_init_kmeanspp(torch.from_numpy(X).cuda(), 700, 6, 10, u, C, idx)
    assert np.array_equal(idx.cpu().numpy(), weights_reference(X, 10, u))


@pytest.mark.parametrize("first", [0, 300])
def test_infinite_coordinates(kp, first):
    """Infinite distances outweigh all others together, the first of them every
    time; as the first centre such a row leaves the rest infinitely far."""
    rng = np.random.default_rng(first)
    X = rng.normal(size=(900, 5)).astype(np.float32)
    X[300, 1] = np.inf
    X[450, 3] = -np.inf
    X[700, 1] = np.inf
    check_weights(kp, X, 9, 2, (first + 0.5) / 900)


@pytest.mark.parametrize("N,D,K", [(120000, 3, 400), (60000, 8, 90), (940000, 2, 1060)])
def test_more_centres_than_the_table(kp, N, D, K):
    """The table of the bound's filter holds half as many centres as a block has
    points (none below 128 points), and 1024 at most."""
    rng = np.random.default_rng(N)
    X = rng.normal(size=(K, D))[rng.integers(0, K, size=N)] * 50.0 + rng.normal(size=(N, D)) * 0.1
    check(kp, X.astype(np.float32), K, seed=K)
