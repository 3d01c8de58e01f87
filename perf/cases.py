"""Performance cases: what a program does with this library, through its public
Python entry points (``paper_1905_09345_gb300.kpynq``), at the sizes of the
repository's own workloads, tests and benchmark.

Kinds of case
  fit        a context that a program keeps (``KMeans``), restarted from its
             initial centroids and fitted: labels, centroids, objective and
             iterations.  The filtered method or plain Lloyd, either grouping,
             FP32 or bfloat16 points.
  oneshot    a data set handled once: context from host arrays, fit, results
             back in host arrays, context closed.
  batch      many uneven problems fitted by one graph launch (``KMeansBatch``).
  step       one allocation-free Lloyd iteration on caller-owned memory.
  seeding    k-means++ initial centroids.
  gradient   forward and backward pass of the proposal network on a batch
             (what a training step does before its update).
  predict    inference of the proposal network.

Inputs are seeded Gaussian mixtures in the shapes of ``synth.py``, drawn on
the GPU.  ``exact`` restates each computation in plain FP64 torch.
"""
import math
import random

import torch

from paper_1905_09345_gb300 import kpynq

DEV = "cuda"


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest job: the latency of a 20-iteration fit (16 blobs)
        dict(name="fit_small_16k", kind="fit", N=16384, D=16, K=16, G=2, iters=20, tol=0.0, data="blobs",
             algo="filtered", grouping="contiguous", dtype="f32"),
        # the benchmark's job: anisotropic mixture, tensor-core dense passes and
        # filtered iterations, stopped by the tolerance
        dict(name="fit_aniso_1m", kind="fit", N=1 << 20, D=64, K=256, G=26, iters=50, tol=1e-4, data="aniso",
             algo="filtered", grouping="clustered", dtype="f32"),
        # plain Lloyd (every distance, every iteration) on a ragged size
        dict(name="lloyd_aniso_300k", kind="fit", N=300007, D=64, K=200, G=20, iters=10, tol=0.0, data="aniso",
             algo="lloyd", grouping="contiguous", dtype="f32"),
        # the largest job: high-dimensional bfloat16 points, 1024 centroids
        dict(name="fit_highdim_4m", kind="fit", N=1 << 22, D=128, K=1024, G=103, iters=30, tol=0.0,
             data="lognormal", algo="filtered", grouping="contiguous", dtype="bf16"),
        # many centroids in few dimensions (the learned proposal's data family)
        dict(name="fit_k4096_1m", kind="fit", N=1 << 20, D=32, K=4096, G=410, iters=20, tol=0.0,
             data="blob_uniform", algo="filtered", grouping="contiguous", dtype="f32"),
        # an odd dimension and ragged sizes: no tensor-core pass, FP32 dense engine
        dict(name="fit_ragged_d17", kind="fit", N=200003, D=17, K=100, G=10, iters=20, tol=0.0, data="blobs",
             algo="filtered", grouping="contiguous", dtype="f32"),
        # a new data set in page-locked host memory, end to end
        dict(name="oneshot_aniso_1m", kind="oneshot", N=1 << 20, D=64, K=256, G=26, iters=50, tol=1e-4,
             data="aniso", grouping="clustered", pinned=True),
        # many small uneven problems at once
        dict(name="batch_48", kind="batch", P=48, n_lo=1000, n_hi=200000, k_lo=8, k_hi=512, iters=25),
        # the iteration for callers that own all device memory
        dict(name="step_262k", kind="step", N=262144, D=64, K=256, data="aniso"),
        # seeding of the skewed, real-data-like job
        dict(name="seeding_1m", kind="seeding", N=1 << 20, D=32, K=128, data="aniso"),
        # the proposal network: one training batch, and inference over a data set
        dict(name="gradient_8192", kind="gradient", B=8192, D=32, H=256, C=410),
        dict(name="predict_1m", kind="predict", N=1 << 20, D=32, H=256, C=410),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fit"] * 5 + ["oneshot", "batch", "step", "seeding", "gradient", "predict"])
    if kind == "fit":
        D = rng.choice([3, 8, 16, 17, 32, 32, 50, 64, 64, 100, 128, 128])
        tensor = D in (32, 64, 128)
        K = _logint(rng, 8, 2048 if tensor else 512)
        most = min(1 << 22, (1 << 38 if tensor else 1 << 32) // (K * D))
        N = _logint(rng, max(1024, 8 * K), max(most, 16 * K, 2048))
        algo = rng.choice(["filtered"] * 4 + ["lloyd"])
        return dict(kind="fit", N=N, D=D, K=K, G=max(1, K // 10), iters=rng.choice([10, 20, 30]),
                    tol=rng.choice([0.0, 1e-4]), data=rng.choice(["blobs", "aniso", "lognormal", "blob_uniform"]),
                    algo=algo, grouping=rng.choice(["contiguous", "clustered"]),
                    dtype=rng.choice(["f32", "f32", "f32", "bf16"]))
    if kind == "oneshot":
        D = rng.choice([16, 17, 32, 64, 128])
        K = _logint(rng, 8, 512)
        return dict(kind="oneshot", N=_logint(rng, 8192, (1 << 26) // D), D=D, K=K, G=max(1, K // 10), iters=20,
                    tol=1e-4, data=rng.choice(["blobs", "aniso"]), grouping=rng.choice(["contiguous", "clustered"]),
                    pinned=rng.choice([True, False]))
    if kind == "batch":
        return dict(kind="batch", P=rng.randint(6, 48), n_lo=1000, n_hi=_logint(rng, 20000, 200000), k_lo=8,
                    k_hi=_logint(rng, 32, 512), iters=rng.choice([10, 25]))
    if kind == "step":
        D = rng.choice([2, 7, 16, 32, 50, 64, 100, 128])
        K = _logint(rng, 4, 1024)
        return dict(kind="step", N=_logint(rng, max(1000, 4 * K), max((1 << 33) // (K * D), 8 * K, 2000)) % (1 << 21) + K,
                    D=D, K=K, data=rng.choice(["blobs", "aniso"]))
    if kind == "seeding":
        D = rng.choice([2, 8, 16, 17, 32, 64, 100])
        return dict(kind="seeding", N=_logint(rng, 2000, (1 << 25) // D), D=D, K=_logint(rng, 4, 300),
                    data=rng.choice(["blobs", "aniso"]))
    if kind == "gradient":
        return dict(kind="gradient", B=128 * _logint(rng, 1, 256), D=rng.choice([8, 17, 32, 64, 128]),
                    H=rng.choice([32, 64, 100, 128, 256]), C=_logint(rng, 8, 512))
    return dict(kind="predict", N=_logint(rng, 1000, 1 << 21), D=rng.choice([8, 17, 32, 64, 128]),
                H=rng.choice([32, 64, 100, 128, 256]), C=_logint(rng, 8, 512))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _mixture(g, N, D, blobs, data):
    """N x D float32 points of a Gaussian mixture, rows in random order."""
    def uniform(lo, hi, *shape):
        return torch.rand(*shape, generator=g, device=DEV) * (hi - lo) + lo

    reach = 10.0 if data == "blobs" else 20.0
    centres = uniform(-reach, reach, blobs, D)
    if data == "blobs":            # isotropic, standard deviation 1
        sig = torch.ones(blobs, 1, device=DEV)
    elif data == "aniso":          # a standard deviation per axis
        sig = uniform(0.5, 2.0, blobs, D)
    elif data == "lognormal":      # blobs of very different widths
        sig = torch.exp(0.5 * torch.randn(blobs, 1, generator=g, device=DEV))
    else:                          # "blob_uniform"
        sig = uniform(0.3, 1.5, blobs, 1)
    if data == "aniso":            # Dirichlet(1) weights: exponentials, normalised
        cum = torch.cumsum(-torch.log1p(-torch.rand(blobs, generator=g, device=DEV, dtype=torch.float64)), 0)
        blob = torch.searchsorted(cum, torch.rand(N, generator=g, device=DEV, dtype=torch.float64) * cum[-1])
        blob.clamp_(max=blobs - 1)
    else:
        blob = torch.randint(blobs, (N,), generator=g, device=DEV)
    X = torch.empty(N, D, device=DEV)
    for a in range(0, N, 1 << 19):
        b = blob[a:a + (1 << 19)]
        X[a:a + (1 << 19)] = centres[b] + torch.randn(len(b), D, generator=g, device=DEV) * sig[b]
    return X


def _points(case, seed):
    g = _gen(seed)
    X = _mixture(g, case["N"], case["D"], case["K"], case["data"])
    C0 = X[torch.randperm(case["N"], generator=g, device=DEV)[:case["K"]]].contiguous()
    if case.get("dtype") == "bf16":
        X = X.to(torch.bfloat16)
        C0 = C0.to(torch.bfloat16).float()
    return X, C0


def _sizes(case):
    """(N, D, K) of a batch's problems: the case's own, whatever the seed."""
    r = random.Random(case["P"] * 1000003 + case["n_hi"] * 1009 + case["k_hi"])
    return [(_logint(r, case["n_lo"], case["n_hi"]), r.choice((8, 32, 64, 128)),
             _logint(r, case["k_lo"], case["k_hi"])) for _ in range(case["P"])]


def _problems(case, seed):
    out = []
    for p, (N, D, K) in enumerate(_sizes(case)):
        X = _mixture(_gen(seed * 1000 + p), N, D, K, "blobs")
        out.append((X, X[:K].contiguous(), max(1, K // 10)))
    return out


def _network(case, seed):
    """Xavier-uniform weights, small biases."""
    g = _gen(seed)
    D, H, C = case["D"], case["H"], case["C"]

    def uniform(a, *shape):
        return (torch.rand(*shape, generator=g, device=DEV) * 2 - 1) * a

    params = dict(W1=uniform(math.sqrt(6 / (D + H)), H, D), b1=uniform(0.05, H),
                  W2=uniform(math.sqrt(3 / H), H, H), b2=uniform(0.05, H),
                  W3=uniform(math.sqrt(6 / (H + C)), C, H), b3=uniform(0.05, C))
    N = case["N"] if "N" in case else case["B"]
    X = torch.randn(N, D, generator=g, device=DEV) * 2
    y = torch.randint(C, (N,), generator=g, device=DEV, dtype=torch.int32)
    return params, X, y


_ALGO = dict(filtered=kpynq.KM_ALGO_FILTERED, lloyd=kpynq.KM_ALGO_LLOYD)
_GROUPING = dict(contiguous=kpynq.KM_GROUP_CONTIGUOUS, clustered=kpynq.KM_GROUP_CLUSTERED)


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case)
    if kind == "fit":
        s["X"], s["C0"] = _points(case, seed)
        s["km"] = kpynq.KMeans(s["X"], s["C0"], case["G"], algo=_ALGO[case["algo"]],
                               grouping=_GROUPING[case["grouping"]])
        s["labels"] = torch.empty(case["N"], dtype=torch.int32, device=DEV)
        s["C"] = torch.empty(case["K"], case["D"], device=DEV)
    elif kind == "oneshot":
        X, C0 = _points(case, seed)
        s["X"], s["C0"] = X.cpu(), C0.cpu()
        s["labels"] = torch.empty(case["N"], dtype=torch.int32)
        s["C"] = torch.empty(case["K"], case["D"])
        if case["pinned"]:
            for k in ("X", "C0", "labels", "C"):
                s[k] = s[k].pin_memory()
    elif kind == "batch":
        probs = _problems(case, seed)
        s["batch"] = kpynq.KMeansBatch(probs)
        s["sizes"] = [X.shape[0] for X, _, _ in probs]
        s["cents"] = [C0.numel() for _, C0, _ in probs]
        s["labels"] = torch.empty(sum(s["sizes"]), dtype=torch.int32, device=DEV)
        s["C"] = torch.empty(sum(s["cents"]), device=DEV)
    elif kind == "step":
        s["X"], s["C0"] = _points(case, seed)
        s["labels"] = torch.empty(case["N"], dtype=torch.int32, device=DEV)
        s["C"] = torch.empty(case["K"], case["D"], device=DEV)
        s["objective"] = torch.empty(1, dtype=torch.float64, device=DEV)
    elif kind == "seeding":
        s["X"], _ = _points(case, seed)
        s["u"] = torch.rand(case["K"], generator=_gen(seed + 1), device=DEV, dtype=torch.float64).cpu()
        s["C"] = torch.empty(case["K"], case["D"], device=DEV)
        s["idx"] = torch.empty(case["K"], dtype=torch.int64, device=DEV)
    else:
        params, s["X"], s["y"] = _network(case, seed)
        s["net"] = kpynq.MLP(case["D"], case["H"], case["C"])
        s["net"].set_params(params)
        if kind == "gradient":
            s["grad"] = torch.empty(s["net"].n_params(), device=DEV)
        else:
            s["pred"] = torch.empty(case["N"], dtype=torch.int32, device=DEV)
    return s


def run(s):
    kind = s["kind"]
    if kind == "fit":
        s["km"].reset(s["C0"])
        r = s["km"].fit(s["iters"], s["tol"], s["labels"], s["C"], with_stats=False)
        return dict(labels=s["labels"], centroids=s["C"], objective=r.objective, n_iter=r.n_iter)
    if kind == "oneshot":
        km = kpynq.KMeans(s["X"], s["C0"], s["G"], grouping=_GROUPING[s["grouping"]])
        r = km.fit(s["iters"], s["tol"], s["labels"], s["C"], with_stats=False)
        km.close()
        return dict(labels=s["labels"], centroids=s["C"], objective=r.objective, n_iter=r.n_iter)
    if kind == "batch":
        b = s["batch"]
        b.reset()
        b.fit(s["iters"], 0.0)
        J, its, n0, c0 = [], [], 0, 0
        for i, (n, c) in enumerate(zip(s["sizes"], s["cents"])):
            j, it = b.get(i, s["labels"][n0:n0 + n], s["C"][c0:c0 + c])
            J.append(j)
            its.append(it)
            n0, c0 = n0 + n, c0 + c
        return dict(labels=s["labels"], centroids=s["C"], objective=torch.tensor(J, dtype=torch.float64),
                    n_iter=torch.tensor(its))
    if kind == "step":
        kpynq.kmeans_lloyd_step_noalloc(s["X"], s["N"], s["D"], s["C0"], s["K"], s["labels"], s["C"], s["objective"])
        return dict(labels=s["labels"], centroids=s["C"], objective=s["objective"])
    if kind == "seeding":
        kpynq.kmeans_init_kmeanspp(s["X"], s["N"], s["D"], s["K"], s["u"], s["C"], s["idx"])
        return dict(centroids=s["C"], indices=s["idx"])
    if kind == "gradient":
        loss = s["net"].gradient(s["X"], s["y"], s["grad"])
        return dict(grad=s["grad"], loss=loss)
    return dict(pred=s["net"].predict(s["X"], s["pred"]))


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind in ("gradient", "predict"):
        D, H, C = case["D"], case["H"], case["C"]
        params = D * H + H + H * H + H + H * C + C
        mac = D * H + H * H + H * C
        if kind == "predict":
            return dict(bytes=case["N"] * (4 * D + 4) + 4 * params, flops=2 * case["N"] * mac)
        # forward, input gradients (not the first layer's) and weight gradients
        return dict(bytes=case["B"] * (4 * D + 4) + 8 * params, flops=2 * case["B"] * (3 * mac - D * H))
    if kind == "batch":
        sizes = _sizes(case)
        return dict(bytes=sum(n * (4 * d + 4) + 8 * k * d for n, d, k in sizes),
                    flops=sum(2 * n * k * d + n * d for n, d, k in sizes))
    N, D, K = case["N"], case["D"], case["K"]
    size = 2 if case.get("dtype") == "bf16" else 4
    if kind == "seeding":  # every point against every centre (each a difference, a square and a sum)
        return dict(bytes=4 * N * D + 4 * K * D + 16 * K, flops=3 * N * D * K)
    # the points once, the labels and both sets of centroids; one all-pairs
    # contraction and one sum per cluster (a filtered fit cannot skip the
    # first assignment; plain Lloyd contracts in every iteration)
    flops = 2 * N * K * D + N * D
    if case.get("algo") == "lloyd":
        flops *= case["iters"]
    return dict(bytes=size * N * D + 4 * N + 8 * K * D, flops=flops)


# ---------------------------------------------------------------------------
# the same results in FP64
# ---------------------------------------------------------------------------
def _assign64(X, C):
    """argmin_k ||x - c_k||^2 in FP64 (X float32 or bfloat16, C float64)."""
    mu = C.mean(0)
    Cc = C - mu
    cn = (Cc * Cc).sum(1)
    out = torch.empty(X.shape[0], dtype=torch.int64, device=X.device)
    rows = max(1024, (1 << 27) // C.shape[0])
    for a in range(0, X.shape[0], rows):
        d = torch.addmm(cn, X[a:a + rows].double() - mu, Cc.T, alpha=-2.0)
        out[a:a + rows] = d.argmin(1)
    return out


def _objective64(X, lab, C):
    J = torch.zeros((), dtype=torch.float64, device=X.device)
    for a in range(0, X.shape[0], 1 << 20):
        d = X[a:a + (1 << 20)].double() - C[lab[a:a + (1 << 20)]]
        J += (d * d).sum()
    return J


def _update64(X, lab, C):
    S = torch.zeros_like(C)
    for a in range(0, X.shape[0], 1 << 20):
        S.index_add_(0, lab[a:a + (1 << 20)], X[a:a + (1 << 20)].double())
    n = torch.bincount(lab, minlength=C.shape[0]).double().unsqueeze(1)
    return torch.where(n > 0, S / n.clamp(min=1), C)


def _lloyd64(X, C0, iters, tol):
    """(centroids, objective): assignment and update until `iters` iterations,
    no change, or a relative decrease of the objective below tol; the
    objective is that of the final assignment to the returned centroids."""
    C, prev, Jp = C0.double(), None, None
    for _ in range(iters):
        lab = _assign64(X, C)
        J = float(_objective64(X, lab, C)) if tol > 0 else None
        same = prev is not None and bool((lab == prev).all())
        C = _update64(X, lab, C)
        if same or (tol > 0 and Jp is not None and Jp - J < tol * Jp):
            break
        prev, Jp = lab, J
    return C, _objective64(X, _assign64(X, C), C)


def _seeding64(X, K, u):
    """Squared distances summed coordinate by coordinate in FP64, weights as
    integers scaled to the largest, the first point whose running sum exceeds
    floor(u * total)."""
    N, D = X.shape
    cols = X.T.contiguous().double()
    d = None
    idx = []
    for j in range(K):
        W = 0
        if d is not None and float(d.max()) > 0:
            run = torch.cumsum(torch.ldexp(d, torch.tensor(32 - math.frexp(float(d.max()))[1])).floor().long(), 0)
            W = int(run[-1])
        if W == 0:
            pick = min(N - 1, max(0, int(math.floor(float(u[j]) * N))))
        else:
            T = min(int(math.floor(float(u[j]) * float(W))), W - 1)
            pick = int(torch.searchsorted(run, torch.tensor([T], device=X.device), right=True))
        idx.append(pick)
        s = torch.zeros(N, dtype=torch.float64, device=X.device)
        for i in range(D):
            t = cols[i] - cols[i, pick]
            s += t * t
        d = s if d is None else torch.minimum(d, s)
    idx = torch.tensor(idx, device=X.device)
    return dict(centroids=X[idx].double(), indices=idx)


def _gradient64(params, X, y):
    """Mean cross-entropy of the softmax and its gradient; weights and points
    at their bfloat16 values, everything else in FP64."""
    p = {k: (v.to(torch.bfloat16) if k[0] == "W" else v).double().requires_grad_() for k, v in params.items()}
    h = X.to(torch.bfloat16).double()
    for i in (1, 2):
        h = torch.nn.functional.gelu(h @ p["W%d" % i].T + p["b%d" % i])
    loss = torch.nn.functional.cross_entropy(h @ p["W3"].T + p["b3"], y.long())
    names = ("W1", "b1", "W2", "b2", "W3", "b3")
    grads = torch.autograd.grad(loss, [p[k] for k in names])
    return dict(grad=torch.cat([g.reshape(-1) for g in grads]), loss=float(loss))


def exact(case, seed):
    kind = case["kind"]
    if kind == "gradient":
        return _gradient64(*_network(case, seed))
    if kind == "predict":
        return None  # class indices: no computed numbers
    if kind == "seeding":
        X, _ = _points(case, seed)
        u = torch.rand(case["K"], generator=_gen(seed + 1), device=DEV, dtype=torch.float64).cpu()
        return _seeding64(X, case["K"], u)
    if kind == "batch":
        got = [_lloyd64(X, C0, case["iters"], 0.0) for X, C0, _ in _problems(case, seed)]
        return dict(labels=None, centroids=torch.cat([C.reshape(-1) for C, _ in got]),
                    objective=torch.stack([J for _, J in got]).cpu(), n_iter=None)
    if case["N"] * case["K"] * case["D"] * case.get("iters", 1) > 3e12:
        return None  # over about 20 seconds of FP64
    X, C0 = _points(case, seed)
    if kind == "step":
        C = C0.double()
        lab = _assign64(X, C)
        return dict(labels=lab, centroids=_update64(X, lab, C), objective=_objective64(X, lab, C).reshape(1))
    C, J = _lloyd64(X, C0, case["iters"], case["tol"])
    return dict(labels=None, centroids=C, objective=float(J), n_iter=None)
