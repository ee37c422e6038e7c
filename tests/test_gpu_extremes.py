"""Finite rows whose squared norms leave the range of fp32: fast scores are infinities, NaN or zeros there, and
every label has to come from the exact pass.  Against the CPU oracle (fp64)."""
import numpy as np
import pytest
import torch

from oracle import cat_oracle as O
from paper_2509_26277_b200 import binding as B
from tests.parity import close, labels_match

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a)).cuda()


def host(t):
    return t.detach().cpu().numpy()


@pytest.fixture(params=[3, 0], ids=["small kernels", "general path"])
def small_kernels(request):
    old = B.cat_get_small_problem_kernels()
    B.cat_set_small_problem_kernels(request.param)
    yield request.param
    B.cat_set_small_problem_kernels(old)


def _clusters(n, d, k, mag):
    """Rows around k points (the first k rows one of each), and the points' magnitudes."""
    rng = np.random.default_rng(n + 7 * d + k)
    size = {"huge": np.full(k, 1e19), "one huge": np.where(np.arange(k) == k // 2, 1e19, 1.0),
            "overflow in the products": np.full(k, 1.2e19 / np.sqrt(d)), "tiny": np.full(k, 1e-24)}[mag]
    cen = rng.normal(size=(k, d)) * size[:, None]
    pick = np.concatenate([np.arange(k), rng.integers(0, k, size=n - k)])
    Yq = cen[pick] + 0.4 * size[pick][:, None] * rng.normal(size=(n, d))
    return Yq.astype(np.float32), cen.astype(np.float32), size


MAGS = ["huge", "one huge", "overflow in the products", "tiny"]


@pytest.mark.parametrize("n,d", [(9001, 256), (700, 516), (8500, 513), (300, 64)])
@pytest.mark.parametrize("k", [2, 3, 4, 5, 9])
@pytest.mark.parametrize("mag", MAGS)
def test_fit(n, d, k, mag, small_kernels):
    Yq, _, size = _clusters(n, d, k, mag)
    Yfp = (0.9 * Yq).astype(np.float32)
    ora = O.fit(Yq, Yfp, k, 3)
    assert int(ora.near.sum()) == 0
    for diag in (False, True):
        C, G, Bt, lab = B.cat_fit(dev(Yq), dev(Yfp), k, 3, want_diag=diag)[:4]
        assert np.array_equal(host(lab), ora.labels), f"{int((host(lab) != ora.labels).sum())} labels differ"
        scale = np.abs(ora.centroids).max(axis=1, keepdims=True)
        close(host(C) / scale, ora.centroids / scale, "centroids")


@pytest.mark.parametrize("n,d", [(513, 256), (513, 264), (500, 1001), (300, 64), (300, 10)])
@pytest.mark.parametrize("k", [2, 3, 4, 5, 9])
@pytest.mark.parametrize("mag", MAGS)
def test_inference(n, d, k, mag, small_kernels):
    Yq, C, size = _clusters(n, d, k, mag)
    g = np.linspace(0.5, 1.5, k * d, dtype=np.float32).reshape(k, d)
    b = (g * size[:, None]).astype(np.float32)
    want, lab, best, second = O.apply(Yq, C, g, b)
    assert np.array_equal(host(B.cat_assign(dev(Yq), dev(C))), lab)
    out, glab = B.cat_apply(dev(Yq), dev(C), dev(g), dev(b), want_labels=True)
    assert np.array_equal(host(glab), lab)
    np.testing.assert_array_equal(host(out), O.affine_with_labels(Yq, lab, g, b))


@pytest.mark.parametrize("stray", [[], [3], [5, 64, 120]])
@pytest.mark.parametrize("value", [1e30, -3e38, np.inf, np.nan])
def test_stray_rows_do_not_reach_the_others(stray, value):
    """Rows of huge or non-finite entries among the first 128, which the fp16 copies take their common point from: the
    other rows are still decided by their fast scores (exact labels either way)."""
    n, d, k = 4000, 1001, 20
    rng = np.random.default_rng(9)
    C = rng.normal(size=(k, d)).astype(np.float32)
    Yq = (C[rng.integers(0, k, size=n)] + 0.4 * rng.normal(size=(n, d))).astype(np.float32)
    Yq[stray] = value
    ws = B.workspace("apply", n, d, k, "cuda")
    labels = host(B.cat_assign(dev(Yq), dev(C), ws=ws))
    rest = np.setdiff1d(np.arange(n), stray)
    assert np.array_equal(labels[rest], O.assign(Yq[rest], C)[0])
    assert ((labels >= 0) & (labels < k)).all()
    assert len(stray) <= B.cat_workspace_report(ws)["refined_rows_last"] < 100


@pytest.mark.parametrize("n,d", [(6000, 60), (3000, 1000), (3000, 301)])
def test_scores_around_the_lowest_finite_one(n, d, small_kernels):
    """Two near centroids and ten far ones, placed so that the scores ||y - c||^2 - ||y - m||^2 (m: the centroids'
    mean) of the two near ones pass the lowest finite fp32 number while every norm is finite: one of
    the two may come out as an infinity, the other not."""
    k = 12
    rng = np.random.default_rng(d)
    u, w = np.linalg.qr(rng.normal(size=(d, 2)))[0].T
    C = np.concatenate([[1.7e19 * u + 3e16 * w, 1.7e19 * u - 3e16 * w], np.tile(-4.6e18 * u, (k - 2, 1))])
    C[2:] += 1e17 * rng.normal(size=(k - 2, d)) / np.sqrt(d)
    C = C.astype(np.float32)
    m = C.astype(np.float64).mean(0)
    # along u: score(h) = |h u - c|^2 - |h u - m|^2 = 2 h (m - c).u + |c|^2 - |m|^2
    c = 1.7e19 * u
    h = (-3.4028235e38 - c @ c + m @ m) / (2 * (m - c) @ u)
    Yq = (h * (1 + 1e-5 * rng.normal(size=n)))[:, None] * u + (1e14 * rng.normal(size=n))[:, None] * w
    Yq = Yq.astype(np.float32)
    assert np.isfinite((Yq * Yq).sum(1)).all()
    lab, best, second = O.assign(Yq, C)
    g, b = rng.normal(size=(k, d)).astype(np.float32), rng.normal(size=(k, d)).astype(np.float32)
    labels_match(host(B.cat_assign(dev(Yq), dev(C))), lab, best, second, "labels")
    out, glab = B.cat_apply(dev(Yq), dev(C), dev(g), dev(b), want_labels=True)
    labels_match(host(glab), lab, best, second, "labels")


def _visitors(n, d, k):
    """Ordinary rows, and one huge row for each of the first k centroids.  The huge row of the most populated cluster
    is drawn to another cluster's centroid in the second round, while all ordinary rows gather in the cluster it leaves."""
    rng = np.random.default_rng(n + d + k)
    cen = np.eye(k, d) * 3.0
    cen[1] = 3.0 * np.array([0.75, np.sqrt(1 - 0.75 ** 2)] + [0.0] * (d - 2))
    pick = np.where(rng.random(n) < 0.9, 0, rng.integers(0, k, size=n))
    pick[:k] = np.arange(k)
    Yq = cen[pick] + 0.05 * rng.normal(size=(n, d))
    big = np.zeros((k, d))
    big[:] = 2e14 * cen / 3.0
    big[1] *= (pick == 1).sum() + 1                          # its cluster's mean is about as long as big[0]
    Yq = np.concatenate([Yq, big]).astype(np.float32)
    return Yq


@pytest.mark.parametrize("n,d,k", [(1000, 64, 8), (3000, 32, 16), (600, 128, 8)])
def test_sums_survive_the_visit_of_a_huge_row(n, d, k):
    Yq = _visitors(n, d, k)
    ora = O.fit(Yq, Yq, k, 2)
    assert ora.centroids[0].max() < 10
    C, G, Bt, lab = B.cat_fit(dev(Yq), dev(Yq), k, 2)
    assert np.array_equal(host(lab), ora.labels)
    scale = np.abs(ora.centroids).max(axis=1, keepdims=True)
    # both are means in fp64, rounded once to fp32
    close(host(C) / scale, ora.centroids / scale, "centroids", abs_tol=2.0 ** -23, rel_tol=0.0)
