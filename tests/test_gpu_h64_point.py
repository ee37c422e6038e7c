"""64-row-tile inference with centroids taken relative to a point among them: far-off clouds, stray and equal centroids."""
import numpy as np
import pytest
import torch

from oracle import cat_oracle as O
from paper_2509_26277_b200 import binding as B
from tests.parity import labels_match

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def host(t):
    return t.detach().cpu().numpy()


@pytest.mark.parametrize("d,k", [(640, 65), (1000, 161), (1024, 256), (2048, 97)])
@pytest.mark.parametrize("kind", ["cloud far from the origin", "first centroid stray", "two of three stray", "equal first three", "infinite centroid",
                                  "zero point"])
def test_matches_the_oracle(d, k, kind):
    n = 4096 + 77
    rng = np.random.default_rng(d + k)
    C = rng.normal(size=(k, d)).astype(np.float32)
    if kind == "cloud far from the origin":
        C = (0.05 * C + 20.0 * rng.normal(size=d)).astype(np.float32)
    elif kind == "first centroid stray":
        C[0] *= 3e4
    elif kind == "two of three stray":
        C[:2] = C[:2] * 1e3 + 1e4
    elif kind == "equal first three":
        C[1] = C[2] = C[0]
    elif kind == "zero point":
        C[:3] = 0.0
    Y = (C[rng.integers(0, k, size=n)] + 0.5 * (0.05 if "cloud" in kind else 1.0) * rng.normal(size=(n, d))).astype(np.float32)
    Y[::5] = (0.5 * (C[rng.integers(3, k, size=len(Y[::5]))] + C[rng.integers(3, k, size=len(Y[::5]))])).astype(np.float32)
    if kind == "infinite centroid":
        C[k - 1, 7] = np.inf
    g, b = rng.normal(size=(k, d)).astype(np.float32), rng.normal(size=(k, d)).astype(np.float32)
    B.cat_set_apply_column_split(64)
    try:
        olab, best, second = O.assign(Y, C)
        out, lab = B.cat_apply(dev(Y), dev(C), dev(g), dev(b), want_labels=True)
        labels_match(host(lab), olab, best, second, "labels")
        np.testing.assert_array_equal(host(out), O.affine_with_labels(Y, host(lab), g, b))
    finally:
        B.cat_set_apply_column_split(0)
