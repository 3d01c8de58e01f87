"""Calls from several host threads at a time: contexts, networks and seedings are
independent of one another, whatever sizes the others have (a kernel's
shared-memory limit is one value per process)."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from test_gpu_parity import kp  # noqa: E402,F401

pytestmark = pytest.mark.gpu


def together(*loops):
    """Every loop in a thread of its own; their first error is raised."""
    errors = []

    def guard(f):
        try:
            f()
        except BaseException as e:  # noqa: BLE001
            errors.append(e)
    ts = [threading.Thread(target=guard, args=(f,)) for f in loops]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    if errors:
        raise errors[0]


def test_networks_of_two_sizes(kp):  # noqa: F811
    def loop(D, H, C, N):
        net = kp.MLP(D, H, C, seed=3)
        X = torch.randn(N, D, device="cuda")
        want = torch.empty(N, dtype=torch.int32, device="cuda")
        got = torch.empty_like(want)

        def run():
            with torch.cuda.device(0):
                net.predict(X, want)
                for _ in range(2000):
                    net.predict(X, got)
                assert torch.equal(got, want)
        return run
    together(loop(256, 256, 512, 300), loop(8, 16, 2, 300), loop(64, 64, 40, 300))


def test_seedings_of_two_widths(kp):  # noqa: F811
    def loop(N, D, K, reps):
        rng = np.random.default_rng(D)
        X = torch.from_numpy(rng.normal(size=(N, D)).astype(np.float32)).cuda()
        u = rng.uniform(size=K)
        C = torch.empty(K, D, device="cuda")
        want = torch.empty(K, dtype=torch.int64, device="cuda")
        got = torch.empty_like(want)

        def run():
            with torch.cuda.device(0):
                kp.kmeans_init_kmeanspp(X, N, D, K, u, C, want)
                for _ in range(reps):
                    kp.kmeans_init_kmeanspp(X, N, D, K, u, C, got)
                    assert torch.equal(got, want)
        return run
    together(loop(200, 4096, 4, 1500), loop(200, 4, 4, 1500), loop(200, 900, 4, 1500))


def test_contexts_of_many_sizes(kp):  # noqa: F811
    """Contexts made, fitted and closed side by side: every dense engine, the
    settle, both survivor kernels, clustered groups."""
    def loop(N, D, K, G, grouping, reps):
        rng = np.random.default_rng(D + K)
        centres = rng.normal(size=(K, D)) * 4.0
        X = (centres[rng.integers(0, K, size=N)] + rng.normal(size=(N, D))).astype(np.float32)
        X, C0 = torch.from_numpy(X).cuda(), torch.from_numpy(X[:K].copy()).cuda()
        got = torch.empty(N, dtype=torch.int32, device="cuda")

        def run():
            with torch.cuda.device(0):
                want = None
                for _ in range(reps):
                    km = kp.KMeans(X, C0, G, grouping=grouping)
                    r = km.fit(4, 0.0, got)
                    km.close()
                    want = got.clone() if want is None else want
                    assert torch.equal(got, want) and r.n_iter <= 4
        return run
    sizes = [(1500, 32, 256, 25, 0), (1500, 32, 1500, 150, 1), (1500, 64, 200, 20, 0), (1500, 128, 32, 3, 0),
             (1500, 128, 900, 90, 0), (1500, 17, 100, 10, 1), (1500, 17, 1400, 10, 0), (700, 400, 64, 6, 1),
             (700, 300, 500, 50, 0)]
    together(*[loop(*s, 60) for s in sizes])
