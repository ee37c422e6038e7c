"""The inference kernel that keeps groups of eight rows in shared memory (any row length), through the C ABI,
against the CPU oracle: edges of the group, of the sixteen-column steps, of the parts a warp takes and of the
groups of sixteen centroids; rows the fast scores cannot decide; ties; extreme magnitudes."""
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


def _check(Yq, C, g, b):
    _, lab, best, second = O.apply(Yq, C, g, b)
    ws = B.workspace("apply", *Yq.shape, C.shape[0], "cuda")
    out, glab = B.cat_apply(dev(Yq), dev(C), dev(g), dev(b), want_labels=True, ws=ws)
    report = B.cat_workspace_report(ws)
    assert report["device_status"] == 0
    labels_match(host(glab), lab, best, second, "labels")
    # the corrected row is one fused multiply-add of the label's coefficients: the same bits
    np.testing.assert_array_equal(host(out), O.affine_with_labels(Yq, host(glab), g, b))
    o16, l16 = B.cat_apply_bf16(dev(Yq), dev(C), dev(g), dev(b), want_labels=True)
    assert torch.equal(l16, glab) and torch.equal(o16, out.to(torch.bfloat16))
    return host(glab), report["refined_rows_last"]


SHAPES = [(1, 1000, 8), (7, 1001, 2), (8, 16, 3), (9, 17, 16), (65, 31, 17), (100, 128, 33), (301, 129, 48), (77, 144, 64),
          (513, 256, 65), (200, 257, 128), (90, 512, 24), (130, 513, 24), (1187, 528, 9), (4000, 1000, 16), (333, 1001, 50),
          (129, 1024, 32), (71, 1999, 5), (40, 2048, 16), (2500, 100, 100), (50, 3001, 4),
          (1300, 10, 16), (333, 3, 2), (700, 1000, 64), (450, 1001, 128), (300, 1023, 33), (260, 2047, 64), (90, 2048, 20)]


@pytest.mark.parametrize("n,d,k", SHAPES)
@pytest.mark.parametrize("kind", ["spread", "close"])
def test_rows_kernel_matches_the_oracle(n, d, k, kind):
    rng = np.random.default_rng(n * 31 + d + k)
    Yq = (rng.normal(size=(n, d)) + 2.0).astype(np.float32)
    g, b = rng.normal(size=(k, d)).astype(np.float32), rng.normal(size=(k, d)).astype(np.float32)
    if kind == "spread":
        C = (rng.normal(size=(k, d)) + 2.0).astype(np.float32)
    else:
        # a tight bunch far from the origin, two of them equal (always left to the exact decision)
        C = (2.0 + 2e-3 * rng.normal(size=(k, d))).astype(np.float32)
        C[-1] = C[0]
    lab, undecided = _check(Yq, C, g, b)
    if kind == "close":
        assert undecided >= (lab == 0).sum()
        assert not (lab == k - 1).any()


@pytest.mark.parametrize("d,k", [(1000, 16), (1001, 32), (60, 40)])
@pytest.mark.parametrize("scale", [1e-25, 1e-12, 1e15])
def test_rows_kernel_at_extreme_magnitudes(d, k, scale):
    rng = np.random.default_rng(d + k)
    Yq = (rng.normal(size=(200, d)) * scale).astype(np.float32)
    Yq[3] *= 1e-6 if scale < 1 else 1e6                      # a row far off the others' magnitude
    Yq[5, d // 2:] *= 1e4                                    # and one whose parts differ
    C = Yq[rng.choice(np.arange(6, 200), size=k, replace=False)].copy()
    g, b = rng.normal(size=(k, d)).astype(np.float32), (rng.normal(size=(k, d)) * scale).astype(np.float32)
    _check(Yq, C, g, b)


FITS = [(5, 4, 5), (600, 5, 2), (37, 1000, 16), (593, 1001, 7), (1024, 64, 64), (1500, 17, 300), (2300, 130, 33), (4100, 257, 24),
        (8192, 50, 32), (300, 3000, 9), (148 * 4 + 1, 8, 3), (2000, 1999, 60)]


@pytest.mark.parametrize("n,d,k", FITS)
@pytest.mark.parametrize("kind", ["cloud", "repeated"])
def test_fit_with_rows_in_shared_memory(n, d, k, kind):
    """cat_fit on small sets (all rounds in one launch): labels, centroids and closed form against the oracle,
    run-to-run repeatability, explicit start; a set with few distinct rows (zero distances, exact ties, empty
    clusters, early fixed point)."""
    rng = np.random.default_rng(n + 3 * d + k)
    Yq = rng.normal(size=(n, d)).astype(np.float32)
    if kind == "repeated":
        Yq = Yq[rng.integers(0, max(2, min(n, k) // 2), size=n)].copy()
    Yfp = (0.9 * Yq + 0.1 * rng.normal(size=(n, d))).astype(np.float32)
    for init in (None, (Yq[rng.permutation(n)[:k]] + 0.25).astype(np.float32)):
        ora = O.fit(Yq, Yfp, k, 6, init=init)
        args = dict(init_centroids=None if init is None else dev(init))
        C, G, Bt, lab = B.cat_fit(dev(Yq), dev(Yfp), k, 6, **args)
        C2, G2, B2, lab2 = B.cat_fit(dev(Yq), dev(Yfp), k, 6, **args)
        assert torch.equal(C, C2) and torch.equal(G, G2) and torch.equal(Bt, B2) and torch.equal(lab, lab2)
        want, best, second = O.assign(Yq, host(C))
        labels_match(host(lab), want, best, second, "labels")
        if int(ora.near.sum()) == 0 or kind == "repeated":
            close(host(C), ora.centroids, "centroids")
            assert np.array_equal(host(lab), ora.labels)
        g, b = O.solve_gamma_beta(Yq, Yfp, host(lab), k)
        close(host(G), g, "gamma")
        close(host(Bt), b, "beta")
    assert B.cat_workspace_report(B.workspace("fit", n, d, k, "cuda"))["device_status"] == 0


# Several groups of rows for every team of every CTA (148 CTAs of T teams take 8 rows each at a time), and a last group
# that is not full: slots that are loaded again, barriers' phases, the prefetch into the other slot.  Teams of 1, 2, 4
# and 8 warps, aligned and ragged rows, fragments in shared memory and in L2.
MANY = [(75_001, 10, 16), (75_003, 60, 12), (36_001, 200, 9), (36_003, 201, 33), (24_001, 528, 9), (24_003, 1000, 16),
        (20_003, 1001, 50), (20_001, 1004, 60), (20_005, 131, 100), (9_003, 1600, 20), (9_001, 2047, 64)]


@pytest.mark.parametrize("n,d,k", MANY)
def test_teams_that_take_many_groups(n, d, k):
    rng = np.random.default_rng(n + d)
    C = rng.normal(size=(k, d)).astype(np.float32)
    Yq = (C[rng.integers(0, k, size=n)] + rng.normal(size=(n, d), scale=0.7)).astype(np.float32)
    Yq[::97] = 0.5 * (C[0] + C[1])                           # undecided rows all over the matrix
    g, b = rng.normal(size=(k, d)).astype(np.float32), rng.normal(size=(k, d)).astype(np.float32)
    assert B.cat_kernel_for("apply", n, d, k) == B.cat_kernel_for("apply_bf16", n, d, k) == "apply_rows_kernel"
    _check(Yq, C, g, b)
    first = B.cat_apply(dev(Yq), dev(C), dev(g), dev(b))
    for _ in range(3):
        assert torch.equal(B.cat_apply(dev(Yq), dev(C), dev(g), dev(b)), first)


@pytest.mark.parametrize("call,n,d,k,kernel", [
    ("apply", 4095, 1004, 128, "apply_rows_kernel"), ("apply", 4096, 1004, 128, "assign_tc_kernel"),
    ("apply", 4096, 256, 128, "apply_rows_kernel"), ("apply", 4096, 264, 65, "assign_tc_kernel"),
    ("apply", 4096, 120, 65, "assign_tc_kernel"), ("apply_bf16", 4096, 120, 65, "apply_rows_kernel"),
    ("apply_bf16", 4096, 132, 65, "assign_tc_kernel"), ("apply", 4096, 132, 65, "apply_rows_kernel"),
    ("apply", 4096, 512, 64, "apply_rows_kernel"), ("apply", 4096, 1000, 33, "apply_h64_kernel"),
    ("apply", 4096, 1000, 32, "apply_rows_kernel"), ("apply", 4096, 1504, 64, "apply_h64_kernel"),
    ("apply", 4096, 1544, 64, "apply_rows_kernel"), ("apply", 4096, 1001, 128, "apply_rows_kernel"),
    ("apply", 4096, 48, 65, "assign_tc_kernel"), ("apply", 4096, 64, 64, "small_kernel"),
    ("fit", 4096, 1000, 32, "fit_rows_kernel"), ("fit", 8192, 256, 32, "fit_rows_kernel"),
    ("fit", 8192, 256, 64, "assign_tc_kernel, fp16 copies"), ("fit", 6144, 256, 128, "assign_tc_kernel, fp16 copies"),
    ("fit", 8192, 50, 64, "fit_rows_kernel"), ("fit", 5000, 64, 64, "small_kernel"), ("fit", 4096, 64, 64, "fit_rows_kernel"),
    ("apply", 8191, 64, 64, "small_kernel"), ("apply", 8192, 64, 64, "apply_short_kernel"), ("apply_bf16", 8191, 64, 64, "apply_rows_kernel"),
    ("apply_bf16", 8192, 112, 64, "apply_short_kernel"), ("apply", 8192, 144, 64, "apply_rows_kernel"),
    ("apply", 9000, 128, 112, "apply_short_kernel"), ("apply", 9000, 128, 113, "small_kernel"),
    ("fit", 8192, 64, 64, "small_kernel"), ("fit", 8193, 64, 64, "fit_tiles_kernel"),
    ("fit", 201_280, 64, 64, "fit_tiles_kernel"), ("fit", 201_281, 64, 64, "small_kernel"),
    ("fit", 40_256, 256, 32, "fit_tiles_kernel"), ("fit", 40_257, 256, 32, "assign_tc_kernel, fp16 copies"),
])
def test_lines_of_the_dispatch(call, n, d, k, kernel):
    """One shape on each side of the lines; results of either side against the oracle."""
    assert B.cat_kernel_for(call, n, d, k) == kernel
    rng = np.random.default_rng(n + d + k)
    cen = rng.normal(size=(k, d)).astype(np.float32)
    Yq = (cen[rng.integers(0, k, size=n)] + rng.normal(size=(n, d))).astype(np.float32)
    if call == "fit":
        C, G, Bt, lab = B.cat_fit(dev(Yq), dev(Yq), k, 3)
        want, best, second = O.assign(Yq, host(C))
        labels_match(host(lab), want, best, second, "labels")
        ora = O.fit(Yq, Yq, k, 3)
        if int(ora.near.sum()) == 0:
            close(host(C), ora.centroids, "centroids")
    else:
        g, b = rng.normal(size=(k, d)).astype(np.float32), rng.normal(size=(k, d)).astype(np.float32)
        _check(Yq, cen, g, b)
