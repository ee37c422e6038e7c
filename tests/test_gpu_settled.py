"""Fits on the multi-launch path whose labels come to rest before the last round: the rounds behind that one do no
work, and the result is that of running them."""
import numpy as np
import pytest
import torch

from oracle import cat_oracle as O
from paper_2509_26277_b200 import binding as B
from tests.parity import labels_match

pytestmark = pytest.mark.gpu


def _clusters(seed, n, d, k, spread):
    rng = np.random.default_rng(seed)
    cen = rng.normal(size=(k, d)) * spread
    Yq = (cen[np.arange(n) % k] + rng.normal(size=(n, d))).astype(np.float32)
    return Yq, (0.9 * Yq + 0.05 * rng.normal(size=(n, d))).astype(np.float32)


@pytest.mark.parametrize("n,d,k,spread", [(9001, 64, 16, 20.0), (9001, 63, 20, 20.0), (20_000, 256, 40, 1.0), (9000, 40, 3, 20.0),
                                          (9000, 16, 300, 20.0), (9000, 64, 1, 20.0)])
def test_rounds_after_a_fixed_point_change_nothing(n, d, k, spread):
    Yq, Yfp = _clusters(3, n, d, k, spread)
    q, f = torch.from_numpy(Yq).cuda(), torch.from_numpy(Yfp).cuda()
    old = B.cat_get_small_problem_kernels()
    B.cat_set_small_problem_kernels(0)
    try:
        ws = torch.empty(B.lib().cat_fit_workspace_bytes(n, d, k), dtype=torch.uint8, device="cuda")
        want = O.fit(Yq, Yfp, k, 60, near_rel=1e-6)
        labels = [torch.full((n,), -1, dtype=torch.int32, device="cuda")] + [B.cat_fit(q, f, k, t)[3] for t in range(60)]
        rounds = next((t for t in range(1, 61) if torch.equal(labels[t], labels[t - 1])), 61)   # the first that moves nothing
        got = {}
        for iters in (60, 59, 12, 0, 60):   # both parities of the label buffers; a fit that settles, then others on its workspace
            C, G, Bt, lab = B.cat_fit(q, f, k, iters, ws=ws)
            # (the ninth word of the control block: a round has moved nothing)
            assert bool(ws[32:36].view(torch.int32)) == (iters >= rounds)
            got.setdefault(iters, []).append([t.cpu() for t in (C, G, Bt, lab)])
        sums, counts = B.cat_cluster_sums(q, got[60][0][3].cuda(), k, ws=ws)
    finally:
        B.cat_set_small_problem_kernels(old)
    assert all(torch.equal(a, b) for a, b in zip(got[60][0], got[60][1]))
    if np.array_equal(want.labels, O.fit(Yq, Yfp, k, 59).labels):
        assert all(torch.equal(a, b) for a, b in zip(got[60][0], got[59][0]))
    if want.near.sum() == 0:
        assert np.array_equal(got[60][0][3].numpy(), want.labels)
        np.testing.assert_allclose(got[60][0][0].numpy(), want.centroids, rtol=1e-5, atol=1e-6)
    first = O.fit(Yq, Yfp, k, 0)
    assert (got[0][0][3].numpy() != first.labels).mean() < 1e-3
    np.testing.assert_array_equal(counts.cpu().numpy(), np.bincount(got[60][0][3].numpy(), minlength=k))


# (aligned rows and not; a tile of rows a CTA, several, a last one that is not full; clusters whose entries fill more than a chunk; most
# clusters and fewest)
@pytest.mark.parametrize("n,d,k", [(200_000, 1028, 8), (50_003, 33, 512), (303_104, 16, 200), (303_105, 9, 200), (700_001, 12, 200)])
def test_rounds_in_which_many_rows_move(n, d, k):
    """One cloud of rows, which keeps moving: from the fourth round on the update follows a list of the moved rows."""
    Yq = np.random.default_rng(n).normal(size=(n, d)).astype(np.float32)
    q = torch.from_numpy(Yq).cuda()
    old = B.cat_get_small_problem_kernels()
    B.cat_set_small_problem_kernels(0)
    try:
        res = {t: [x.cpu().numpy() for x in B.cat_fit(q, q, k, t)] for t in (4, 5, 6)}
        again = B.cat_fit(q, q, k, 6)
    finally:
        B.cat_set_small_problem_kernels(old)
    assert all(np.array_equal(a, b.cpu().numpy()) for a, b in zip(res[6], again))
    for t in (4, 5):
        moved = res[t][3] != res[t + 1][3]
        entries = np.bincount(np.concatenate([res[t][3][moved], res[t + 1][3][moved]]), minlength=k)
        assert moved.sum() > n // 200 and (k > 8 or entries.max() > 2048)
    for t in (4, 5):
        want, _ = O.update_centroids(Yq, res[t][3], res[t][0])
        # (both are fp32 roundings of fp64 means)
        np.testing.assert_allclose(res[t + 1][0], want, rtol=2.0 ** -23, atol=1e-12)
    lab, best, second = O.assign(Yq, res[6][0])
    labels_match(res[6][3], lab, best, second, "labels")


@pytest.mark.parametrize("n,d,k", [(2000, 64, 16), (2001, 100, 5), (1000, 1601, 9), (3000, 30, 3), (3000, 16, 20), (1500, 1000, 8)])
def test_counters_of_the_exact_pass_do_not_depend_on_the_early_end(n, d, k):
    """One cloud of rows, some of which are undecided in every round; its labels come to rest within 90 rounds.  With
    diagnostics every assignment runs, and the counters are those of that fit."""
    Yq = (np.random.default_rng(4).normal(size=(n, d)) * np.linspace(3.0, 0.3, d)).astype(np.float32)
    q = torch.from_numpy(Yq).cuda()
    old = B.cat_get_small_problem_kernels()
    B.cat_set_small_problem_kernels(0)
    try:
        ws = torch.empty(B.lib().cat_fit_workspace_bytes(n, d, k), dtype=torch.uint8, device="cuda")
        for kw in (dict(), dict(init_centroids=torch.from_numpy(Yq[n - k:]).cuda())):
            diag = B.cat_fit(q, q, k, 120, want_diag=True, ws=ws, **kw)[-1]
            B.cat_fit(q, q, k, 120, ws=ws, **kw)
            rep = B.cat_workspace_report(ws)
            assert diag["refined_rows_total"] > 0 or k == 3   # (fp32 scores leave hardly a row open)
            assert rep["refined_rows_last"] == diag["refined_rows_final"]
            assert rep["refined_rows_total"] == diag["refined_rows_total"]
    finally:
        B.cat_set_small_problem_kernels(old)
