"""Near-ties of survivors on the filtered path: points within a few FP32 roundings
of the midpoint of two centroids, in every iteration, so that the FP32 scan often
prefers the wrong one and the ordered pair corrects it (the point's own bounds
with it).  The two centroids share a group or not; odd and even row widths.
Labels, update, objective and bounds against the FP64 oracle as in
test_gpu_parity (same tolerances)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from test_gpu_parity import kp, lockstep  # noqa: E402,F401

pytestmark = pytest.mark.gpu


def pairs(D, P, seed):
    """P pairs of centroids at -1 and +1 of coordinate 0, the pairs 64 apart in
    coordinate 1.  Anchors sit on them; the other points lie beside the plane
    between, mirrored in all other coordinates and in coordinate 0, so that the
    means of the two clusters stay mirror images."""
    rng = np.random.default_rng(seed)
    X, C = [], []
    for i in range(P):
        y = rng.normal(size=(40, D - 2)) * 0.5
        x0 = rng.integers(1, 9, size=40) * 2.0 ** -26
        for s in (-1.0, 1.0):
            anchor = np.zeros((60, D))
            anchor[:, 0], anchor[:, 1] = s, 64.0 * i
            C.append(anchor[0])
            X.append(anchor)
            for m in (-1.0, 1.0):
                z = np.empty((40, D))
                z[:, 0], z[:, 1], z[:, 2:] = s * x0, 64.0 * i, m * y
                X.append(z)
    X = np.concatenate(X).astype(np.float32)
    return X[rng.permutation(len(X))], np.array(C, np.float32)


@pytest.mark.parametrize("D", [12, 17, 20, 28, 48, 64, 96, 128])
@pytest.mark.parametrize("together", [True, False])
def test_filtered_near_ties(kp, D, together):  # noqa: F811
    P = 6
    X, C0 = pairs(D, P, D)
    if not together:  # all of the one side, then all of the other
        C0 = np.concatenate([C0[0::2], C0[1::2]])
    st = lockstep(kp, X, C0, P, 5, check_bounds=True, dense_switch=1.0)
    assert all(s["n_recheck"] > 0 and s["path"] == kp.KM_PATH_FILTERED for s in st[1:]), st


@pytest.mark.parametrize("D", [5, 64, 96, 128])
@pytest.mark.parametrize("dense_switch", [0.0, 1.0])
def test_copies_of_every_centroid(kp, D, dense_switch):  # noqa: F811
    """Every centroid twice, in different groups, and clusters symmetric about
    it: each point has two nearest ones in each iteration, the lower index wins."""
    rng = np.random.default_rng(D)
    P = 7
    c = rng.integers(-20, 21, size=(P, D)) * 4.0
    d = rng.integers(-3, 4, size=(P, 40, D))
    X = np.concatenate([c[:, None] + d, c[:, None] - d], 1).reshape(-1, D).astype(np.float32)
    C0 = np.concatenate([c, c]).astype(np.float32)
    st = lockstep(kp, X[rng.permutation(len(X))], C0, 4, 4, check_bounds=True, dense_switch=dense_switch)
    assert all(s["n_recheck"] == len(X) for s in st)
