"""cat_apply_pca in the kernel that keeps rows in shared memory (scores of the projected rows without the projection)
against the oracle, and against the three-step path it takes the place of."""
import numpy as np
import pytest
import torch

from oracle import cat_oracle as O
from oracle import cat_pca_oracle as P
from paper_2509_26277_b200 import binding as B
from tests.parity import labels_match

pytestmark = pytest.mark.gpu


def host(t):
    return t.detach().cpu().numpy()


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a)).cuda()


def _case(seed, n, d, p, k, offset, scale):
    rng = np.random.default_rng(seed)
    Y = (rng.normal(size=(n, d)) * scale + offset).astype(np.float32)
    V = np.linalg.qr(rng.normal(size=(d, p)))[0].T.astype(np.float32)
    mean = (np.full(d, offset) + 0.1 * scale * rng.normal(size=d)).astype(np.float32)
    C = (scale * rng.normal(size=(k, p))).astype(np.float32)
    g, b = rng.normal(size=(k, d)).astype(np.float32), rng.normal(size=(k, d)).astype(np.float32)
    return Y, mean, V, C, g, b


def _check(Y, mean, V, C, g, b, one_kernel=None):
    """one_kernel: whether the call takes that kernel (preparation, rows, open rows: three launches; the other way has more)."""
    args = [dev(a) for a in (Y, mean, V, C, g, b)]
    before = B.cat_kernel_launches()
    out, lab = B.cat_apply_pca(*args, want_labels=True)
    if one_kernel is not None:
        assert (B.cat_kernel_launches() - before == 3) == one_kernel
    want, olab, best, second = P.apply_pca(Y, mean, V, C, g, b)
    labels_match(host(lab), olab, best, second, "labels of the projected rows")
    np.testing.assert_array_equal(host(out), O.affine_with_labels(Y, host(lab), g, b))
    return host(lab)


# (one warp a team, two and four; each number of centroid groups; aligned rows and not; the fewest rows of a length; fragments in shared
# memory and out of L2; a last group that is not full)
@pytest.mark.parametrize("n,d,p,k,offset,scale", [
    (64, 1024, 3, 2, 0.0, 1.0), (65, 1023, 1, 2, 0.0, 1.0), (65_536, 1, 1, 2, 0.0, 1.0), (13_108, 5, 5, 3, 0.0, 1.0), (1024, 64, 8, 16, 0.0, 1.0),
    (2001, 63, 20, 30, 0.0, 1.0), (2003, 33, 9, 48, 2.0, 1.0), (1001, 127, 33, 64, 0.0, 1.0), (3001, 60, 12, 32, 0.0, 1.0), (3003, 100, 50, 40, 0.0, 1.0),
    (1500, 44, 44, 64, 0.0, 10.0), (1003, 201, 30, 16, 0.0, 1.0), (1005, 203, 30, 64, 0.0, 1.0), (1007, 204, 60, 9, 0.0, 1.0), (999, 132, 8, 64, 0.0, 1.0),
    (1003, 501, 16, 16, 0.0, 1.0), (1003, 502, 16, 30, 0.0, 1.0), (1003, 300, 16, 64, 0.0, 1.0), (999, 300, 16, 10, 0.0, 1.0), (999, 1000, 20, 30, 0.0, 1.0),
    (999, 204, 12, 20, 0.0, 1.0), (1001, 201, 12, 40, 0.0, 1.0), (1001, 1001, 12, 40, 0.0, 1.0), (999, 300, 20, 40, 0.0, 1.0), (999, 1000, 50, 40, 0.0, 1.0),
    (1001, 301, 50, 64, 0.0, 1.0),
    (1001, 128, 33, 17, 3.0, 1.0), (997, 129, 50, 32, 0.0, 1e-3), (2003, 256, 50, 33, 100.0, 1.0), (2003, 257, 4, 48, 0.0, 1e3),
    (3001, 1000, 50, 64, 1.0, 1.0), (3001, 1001, 50, 64, 0.0, 1.0), (513, 1024, 300, 5, 0.0, 1.0), (515, 1023, 64, 49, 50.0, 1.0),
])
def test_labels_and_outputs_match_the_oracle(n, d, p, k, offset, scale):
    case = _case(n + d + p + k, n, d, p, k, offset, scale)
    lab = _check(*case, one_kernel=True)
    old = B.cat_get_small_problem_kernels()
    B.cat_set_small_problem_kernels(0)
    try:
        assert (lab != _check(*case, one_kernel=False)).mean() <= 2e-3   # (a row within fp32 rounding of a bisector)
    finally:
        B.cat_set_small_problem_kernels(old)


def test_equal_centroids_and_rows_between_two():
    """Rows on the bisector of two centroids, and centroids that coincide: lowest index, as the exact distances have it."""
    rng = np.random.default_rng(5)
    d, p, k, n = 300, 12, 20, 4000
    V = np.eye(p, d, dtype=np.float32)   # the projection is exact: the first p columns
    C = rng.integers(-8, 8, size=(k, p)).astype(np.float32)
    C[7] = C[3]
    C[19] = C[3]
    i, j = rng.integers(0, k, size=n), rng.integers(0, k, size=n)
    Y = rng.normal(size=(n, d)).astype(np.float32)
    Y[:, :p] = (C[i] + C[j]) / 2
    Y[::2, :p] = C[i[::2]]
    g, b = rng.normal(size=(k, d)).astype(np.float32), rng.normal(size=(k, d)).astype(np.float32)
    mean = np.zeros(d, np.float32)
    _, lab = B.cat_apply_pca(dev(Y), dev(mean), dev(V), dev(C), dev(g), dev(b), want_labels=True)
    olab, _, _ = O.assign(np.ascontiguousarray(Y[:, :p]), C)
    np.testing.assert_array_equal(host(lab), olab)


@pytest.mark.parametrize("n,d,k", [(3000, 300, 40), (3001, 301, 64), (4000, 64, 7), (2003, 100, 33)])
def test_centroids_that_coincide(n, d, k):
    """Every row but those of a few clusters is left to the kernel behind; the lowest of the equal centroids has it, and rows on the
    bisector of two such groups are decided by the projection."""
    rng = np.random.default_rng(n + k)
    half = (k + 1) // 2
    Y, mean, V, C, g, b = _case(n + k, n, d, 12, k, 1.0, 1.0)
    C[half:] = C[rng.permutation(half)[:k - half]]
    i, j = rng.integers(0, k, size=n), rng.integers(0, k, size=n)
    z = np.where((np.arange(n) % 3 == 0)[:, None], 0.5 * (C[i] + C[j]), C[i] + 0.05 * rng.normal(size=(n, 12)))
    Y = (z @ V + mean + 1e-6 * rng.normal(size=(n, d))).astype(np.float32)
    ws = B.pca_workspace("apply_pca", n, d, 12, "cuda", k)
    out, lab = B.cat_apply_pca(dev(Y), dev(mean), dev(V), dev(C), dev(g), dev(b), want_labels=True, ws=ws)
    assert int(ws[:4].view(torch.int32)) > n // 2   # (the control block's first word: rows listed for that kernel)
    assert host(lab).max() < half
    _, olab, best, second = P.apply_pca(Y, mean, V, C[:half], g, b)
    labels_match(host(lab), olab, best, second, "labels")
    np.testing.assert_array_equal(host(out), O.affine_with_labels(Y, host(lab), g, b))


def test_components_that_are_not_unit_vectors_and_rows_out_of_range():
    rng = np.random.default_rng(6)
    Y, mean, V, C, g, b = _case(6, 1200, 200, 10, 24, 0.0, 1.0)
    V = (V * np.logspace(-3, 3, 10)[:, None]).astype(np.float32)
    C = (C * np.logspace(-3, 3, 10)[None]).astype(np.float32)
    Y[3] *= 1e18
    Y[4] *= 1e-25
    Y[5] = 0.0
    _check(Y, mean, V, C, g, b)
    Y[6, 11] = np.nan
    Y[7, 12] = np.inf
    old = B.cat_get_small_problem_kernels()
    got = []
    try:
        for mask in (old, 0):
            B.cat_set_small_problem_kernels(mask)
            got.append([host(t) for t in B.cat_apply_pca(dev(Y), dev(mean), dev(V), dev(C), dev(g), dev(b), want_labels=True)])
    finally:
        B.cat_set_small_problem_kernels(old)
    rest = np.setdiff1d(np.arange(1200), [6, 7])
    np.testing.assert_array_equal(got[0][1][rest], got[1][1][rest])
    np.testing.assert_array_equal(got[0][0][rest], got[1][0][rest])
    assert all(0 <= l < 24 for l in got[0][1][[6, 7]])


@pytest.mark.parametrize("n,d,k", [(3000, 300, 20), (3001, 301, 20), (4000, 64, 7), (1000, 1001, 40)])
def test_output_in_the_place_of_the_input(n, d, k):
    """Rows on bisectors, which the kernel for open rows reads once more, with Y_out = Yq."""
    rng = np.random.default_rng(n + d)
    p = 12
    V = np.linalg.qr(rng.normal(size=(d, p)))[0].T.astype(np.float32)
    C = rng.normal(size=(k, p)).astype(np.float32)
    i, j = rng.integers(0, k, size=n), rng.integers(0, k, size=n)
    Y = ((0.5 * (C[i] + C[j])) @ V + 1e-7 * rng.normal(size=(n, d))).astype(np.float32)
    g, b = rng.normal(size=(k, d)).astype(np.float32), rng.normal(size=(k, d)).astype(np.float32)
    mean = np.zeros(d, np.float32)
    ws = B.pca_workspace("apply_pca", n, d, p, "cuda", k)
    want, lab = B.cat_apply_pca(dev(Y), dev(mean), dev(V), dev(C), dev(g), dev(b), want_labels=True, ws=ws)
    np.testing.assert_array_equal(host(want), O.affine_with_labels(Y, host(lab), g, b))
    assert int(ws[:4].view(torch.int32)) > 100   # (the control block's first word: rows listed for that kernel)
    y = dev(Y)
    _, lab2 = B.cat_apply_pca(y, dev(mean), dev(V), dev(C), dev(g), dev(b), out=y, want_labels=True)
    assert torch.equal(lab, lab2)
    assert torch.equal(y, want)
