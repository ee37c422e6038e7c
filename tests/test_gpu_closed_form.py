"""gamma and beta of small sets, which one launch forms, at the ends of its range, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import cat_oracle as O
from paper_2509_26277_b200 import binding as B
from tests.parity import close

pytestmark = pytest.mark.gpu


# one row a cluster, a last block of columns that is not full, rows that are not aligned, the most rows either takes and one more,
# the fewest clusters for them and one less
@pytest.mark.parametrize("n,d,k", [(2, 4, 2), (5, 7, 5), (33, 100, 3), (2048, 33, 4), (2049, 33, 5), (2048, 33, 3), (8192, 36, 16), (8192, 36, 15),
                                   (8193, 36, 17), (1000, 1000, 16)])
@pytest.mark.parametrize("kind", ["even", "one cluster has nearly all"])
def test_small_sets(n, d, k, kind):
    rng = np.random.default_rng(n + d + k)
    far = 50.0 * rng.normal(size=(k, d))
    pick = np.concatenate([np.arange(k), rng.integers(0, k, size=n - k) if kind == "even" else np.zeros(n - k, np.int64)])
    Yq = (far[pick] + rng.normal(size=(n, d))).astype(np.float32)
    Yfp = (0.8 * Yq + 0.1 * rng.normal(size=(n, d)) + 3.0).astype(np.float32)
    q, f = torch.from_numpy(Yq).cuda(), torch.from_numpy(Yfp).cuda()
    C, G, Bt, lab = B.cat_fit(q, f, k, 2)
    g, b = O.solve_gamma_beta(Yq, Yfp, lab.cpu().numpy(), k)
    close(G.cpu().numpy(), g, "gamma")
    close(Bt.cpu().numpy(), b, "beta")
    # fit_pca forms the sums themselves, too
    if d > 4 and n > k:
        r = B.cat_fit_pca(q, f, k, 2, min(d, 6))
        g, b = O.solve_gamma_beta(Yq, Yfp, r["labels"].cpu().numpy(), k)
        close(r["gamma"].cpu().numpy(), g, "gamma")
        close(r["beta"].cpu().numpy(), b, "beta")
