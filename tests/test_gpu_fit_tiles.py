"""Fits of many rows of few columns in one launch (rows held as fp16 operand fragments) against the oracle."""
import numpy as np
import pytest
import torch

from oracle import cat_oracle as O
from paper_2509_26277_b200 import binding as B
from tests.parity import close, labels_match
from tests.test_gpu_extremes import MAGS, _clusters, _visitors

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def host(t):
    return t.detach().cpu().numpy()


# one and two steps of columns, one chunk of centroids and two, aligned rows and not, a last group and a last CTA that are
# not full, one group per CTA, the most rows a CTA holds
SHAPES = [(8193, 4, 2), (8200, 10, 100), (9001, 17, 33), (8193 + 148, 63, 64), (20_001, 64, 65), (30_000, 50, 128), (12_000, 256, 32),
          (10_007, 255, 30), (40_003, 129, 16), (100_003, 32, 128), (200_704, 64, 64)]


@pytest.mark.parametrize("n,d,k", SHAPES)
@pytest.mark.parametrize("kind", ["cloud", "repeated"])
def test_fit(n, d, k, kind):
    assert B.cat_kernel_for("fit", n, d, k) == "fit_tiles_kernel"
    rng = np.random.default_rng(n + 3 * d + k)
    Yq = rng.normal(size=(n, d)).astype(np.float32)
    if kind == "repeated":
        Yq = Yq[rng.integers(0, max(2, k // 2), size=n)].copy()
    Yfp = (0.9 * Yq + 0.1 * rng.normal(size=(n, d))).astype(np.float32)
    for init in (None, (Yq[rng.permutation(n)[:k]] + 0.25).astype(np.float32)):
        ora = O.fit(Yq, Yfp, k, 5, init=init)
        args = dict(init_centroids=None if init is None else dev(init))
        C, G, Bt, lab = B.cat_fit(dev(Yq), dev(Yfp), k, 5, **args)
        again = B.cat_fit(dev(Yq), dev(Yfp), k, 5, **args)
        assert all(torch.equal(a, b) for a, b in zip((C, G, Bt, lab), again))
        want, best, second = O.assign(Yq, host(C))
        labels_match(host(lab), want, best, second, "labels")
        if int(ora.near.sum()) == 0 or kind == "repeated":
            close(host(C), ora.centroids, "centroids")
            assert np.array_equal(host(lab), ora.labels)
        g, b = O.solve_gamma_beta(Yq, Yfp, host(lab), k)
        close(host(G), g, "gamma")
        close(host(Bt), b, "beta")
    assert B.cat_workspace_report(B.workspace("fit", n, d, k, "cuda"))["device_status"] == 0


@pytest.mark.parametrize("iters", [0, 1, 2, 40])
def test_rounds(iters):
    """None, both parities, and more than the labels need to come to rest; a common offset far above the rows' spread."""
    n, d, k = 9000, 48, 12
    rng = np.random.default_rng(2)
    cen = 20.0 * rng.normal(size=(k, d))
    Yq = (cen[np.arange(n) % k] + rng.normal(size=(n, d)) + 300.0).astype(np.float32)
    ora = O.fit(Yq, Yq, k, iters)
    C, G, Bt, lab = B.cat_fit(dev(Yq), dev(Yq), k, iters)
    assert np.array_equal(host(lab), ora.labels)
    close(host(C), ora.centroids, "centroids")


@pytest.mark.parametrize("n,d,k", [(9001, 4, 60), (9000, 10, 100), (20_000, 32, 40)])
def test_counters_do_not_depend_on_the_early_end(n, d, k):
    """Labels that come to rest leave the total as if every assignment had run: each one more adds the rows of the last."""
    Yq = np.random.default_rng(n).normal(size=(1500, d)).astype(np.float32)[np.arange(n) % 1500]   # one cloud of repeated rows
    ws = B.workspace("fit", n, d, k, "cuda")
    reps, labels = {}, {}
    for iters in (150, 151, 165):
        labels[iters] = B.cat_fit(dev(Yq), dev(Yq), k, iters, ws=ws)[3]
        reps[iters] = B.cat_workspace_report(ws)
    assert torch.equal(labels[150], labels[165])
    last = reps[150]["refined_rows_last"]
    assert last > 0 and reps[165]["refined_rows_last"] == last
    assert reps[151]["refined_rows_total"] - reps[150]["refined_rows_total"] == last
    assert reps[165]["refined_rows_total"] - reps[150]["refined_rows_total"] == 15 * last


@pytest.mark.parametrize("k", [2, 9, 70])
@pytest.mark.parametrize("mag", MAGS)
def test_magnitudes_at_the_ends_of_fp32(k, mag):
    Yq, _, size = _clusters(9001, 64, k, mag)
    ora = O.fit(Yq, Yq, k, 3)
    C, G, Bt, lab = B.cat_fit(dev(Yq), dev(Yq), k, 3)
    assert np.array_equal(host(lab), ora.labels)
    scale = np.abs(ora.centroids).max(axis=1, keepdims=True)
    close(host(C) / scale, ora.centroids / scale, "centroids")


@pytest.mark.parametrize("n,d,k", [(9000, 64, 8), (9000, 32, 16), (12_000, 128, 8)])
def test_sums_survive_the_visit_of_a_huge_row(n, d, k):
    """Every centroid is the mean of the rows that carried its label, whatever rows were there before.  (The labels are the
    kernel's own: the distances between the huge rows and the centroids differ by less than fp64 resolves.)"""
    Yq = _visitors(n, d, k)
    assert B.cat_kernel_for("fit", len(Yq), d, k) == "fit_tiles_kernel"
    y = Yq.astype(np.float64)
    before = y[:k]
    for t in range(4):
        lab = host(B.cat_fit(dev(Yq), dev(Yq), k, t)[3])
        C = host(B.cat_fit(dev(Yq), dev(Yq), k, t + 1)[0])
        want = np.stack([y[lab == j].mean(0) if (lab == j).any() else before[j] for j in range(k)])
        scale = np.abs(want).max(axis=1, keepdims=True)
        # both are means in fp64, rounded once to fp32
        close(C / scale, want / scale, f"centroids of round {t + 1}", abs_tol=2.0 ** -23, rel_tol=0.0)
        before = C.astype(np.float64)
