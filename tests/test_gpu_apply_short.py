"""Inference on short rows that stay in registers, fp32 and bf16 output, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import cat_oracle as O
from paper_2509_26277_b200 import binding as B
from tests.parity import labels_match
from tests.test_gpu_extremes import MAGS, _clusters

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def host(t):
    return t.detach().cpu().numpy()


def _check(Y, C, g, b, alpha=1.0):
    n, d = Y.shape
    k = len(C)
    assert B.cat_kernel_for("apply", n, d, k) == B.cat_kernel_for("apply_bf16", n, d, k) == "apply_short_kernel"
    olab, best, second = O.assign(Y, C)
    out, lab = B.cat_apply(dev(Y), dev(C), dev(g), dev(b), want_labels=True)
    labels_match(host(lab), olab, best, second, "labels")
    np.testing.assert_array_equal(host(out), O.affine_with_labels(Y, host(lab), g, b))
    half, lab2 = B.cat_apply_bf16(dev(Y), dev(C), dev(g), dev(b), want_labels=True)
    assert torch.equal(lab, lab2)
    np.testing.assert_array_equal(host(half.float()), host(out.to(torch.bfloat16).float()))
    ws = B.workspace("apply", n, d, k, "cuda")
    out3 = B.cat_apply(dev(Y), dev(C), dev(g), dev(b), ws=ws)
    assert torch.equal(out, out3)
    return B.cat_workspace_report(ws)


# every number of column steps, one chunk of centroids and two, tiles of centroids that are not full, a last group of one row
SHAPES = [(8192, 32, 8), (8193, 32, 128), (8207, 48, 17), (9000, 48, 100), (20_001, 64, 64), (8208, 64, 65), (20_011, 64, 81), (8195, 64, 128), (9003, 80, 8), (8211, 80, 81), (10_001, 96, 33),
          (9001, 96, 96), (8197, 32, 113), (8193, 112, 64), (20_003, 112, 90), (8199, 128, 9), (30_005, 128, 64), (8209, 128, 100), (200_704, 64, 64)]


@pytest.mark.parametrize("n,d,k", SHAPES)
@pytest.mark.parametrize("kind", ["cloud", "near ties", "far apart"])
def test_matches_the_oracle(n, d, k, kind):
    rng = np.random.default_rng(n + d + k)
    C = (rng.normal(size=(k, d)) * (30.0 if kind == "far apart" else 1.0)).astype(np.float32)
    Y = (C[rng.integers(0, k, size=n)] + rng.normal(size=(n, d), scale=1.0)).astype(np.float32)
    if kind == "near ties":
        C[k // 2] = C[0]                                         # equal centroids: the lower index
        i, j = rng.integers(0, k, size=n), rng.integers(0, k, size=n)
        Y = (0.5 * (C[i] + C[j]) + 1e-3 * rng.normal(size=(n, d))).astype(np.float32)
        Y[::3] = 0.25 * C.sum(0) / k                             # every centroid is a candidate
        Y[1::7] = C[j[1::7]]
    g, b = rng.normal(size=(k, d)).astype(np.float32), rng.normal(size=(k, d)).astype(np.float32)
    rep = _check(Y, C, g, b)
    assert rep["device_status"] == 0 and rep["refined_rows_last"] <= n
    if kind == "far apart":
        assert rep["refined_rows_last"] < n // 100


@pytest.mark.parametrize("d", [32, 64, 128])
@pytest.mark.parametrize("k", [8, 9, 70])
@pytest.mark.parametrize("mag", MAGS)
def test_magnitudes_at_the_ends_of_fp32(d, k, mag):
    Y, C, size = _clusters(8300, d, k, mag)
    g = np.linspace(0.5, 1.5, k * d, dtype=np.float32).reshape(k, d)
    b = (g * size[:, None]).astype(np.float32)
    _, lab, _, _ = O.apply(Y, C, g, b)
    out, glab = B.cat_apply(dev(Y), dev(C), dev(g), dev(b), want_labels=True)
    assert np.array_equal(host(glab), lab)
    np.testing.assert_array_equal(host(out), O.affine_with_labels(Y, lab, g, b))


def test_rows_that_are_not_finite_leave_the_others_alone():
    rng = np.random.default_rng(4)
    n, d, k = 8200, 64, 20
    C = rng.normal(size=(k, d)).astype(np.float32)
    Y = (C[rng.integers(0, k, size=n)] + 0.3 * rng.normal(size=(n, d))).astype(np.float32)
    Y[5, 3], Y[17, 60], Y[18, 0] = np.nan, np.inf, -np.inf
    g, b = rng.normal(size=(k, d)).astype(np.float32), rng.normal(size=(k, d)).astype(np.float32)
    out, lab = B.cat_apply(dev(Y), dev(C), dev(g), dev(b), want_labels=True)
    rest = np.setdiff1d(np.arange(n), [5, 17, 18])
    assert np.array_equal(host(lab)[rest], O.assign(Y[rest], C)[0])
    np.testing.assert_array_equal(host(out)[rest], O.affine_with_labels(Y[rest], host(lab)[rest], g, b))
    assert ((host(lab) >= 0) & (host(lab) < k)).all()
