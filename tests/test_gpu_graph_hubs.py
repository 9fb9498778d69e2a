"""The fuzzy union of neighbour lists with hubs: in-lists of every length that
takes its own path (up to a warp, ranked by a warp, sorted by a CTA, beyond the
CTA's sort), list lengths around the templates' widths, against the oracle on
the same lists."""
import numpy as np
import pytest

from gpu_util import drgb_module
from oracle import fuzzy as ofuzzy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k,hubs", [(9, 1, 0), (40, 8, 0), (3000, 9, 2), (2000, 16, 3), (2000, 17, 1), (700, 32, 1),
                                      (20000, 5, 4), (12000, 2, 1)])
def test_union_with_hubs_matches_oracle(n, k, hubs):
    import torch
    drgb = drgb_module()
    rng = np.random.default_rng(n + k)
    # hubs: the first few points are in most lists, the next ones in fewer and fewer
    share = np.concatenate([[0.9, 0.5, 0.06, 0.02][:hubs], np.full(n - hubs, 0.0)])
    idx = np.empty((n, k), np.int32)
    for i in range(n):
        take = [h for h in range(hubs) if h != i and rng.uniform() < share[h]][:k]
        rest = set(take)
        while len(rest) < k:
            j = int(rng.integers(0, n)) if rng.uniform() < 0.7 else int(rng.integers(0, min(n, 300)))
            if j != i:
                rest.add(j)
        idx[i] = rng.permutation(sorted(rest))
    dist = np.sort(rng.uniform(0.5, 3.0, (n, k)).astype(np.float32), axis=1)
    dist[::7] = dist[::7, :1]  # rows of equal distances
    T = 100
    g = drgb.fuzzy_weights(torch.from_numpy(idx).cuda(), torch.from_numpy(dist).cuda(), T, with_rho_sigma=True)
    o = ofuzzy.build_csr(idx.astype(np.int64), dist.astype(np.float64), T, k)
    np.testing.assert_array_equal(g.rho.cpu().numpy(), o["rho"])
    rp, col, q = (x.cpu().numpy().astype(np.int64) for x in (g.row_ptr, g.col, g.q))
    w = g.w.cpu().numpy().astype(np.float64)
    np.testing.assert_array_equal(q, np.rint(2.0 ** 24 * w).astype(np.int64))
    S = o["union"].tocsr()
    heads = np.repeat(np.arange(n), np.diff(rp))
    assert np.all((np.diff(col) > 0) | (np.diff(heads) > 0))
    # weights of FP32 bisection and exponentials: 1e-5, as for the k-NN graphs
    np.testing.assert_allclose(w, np.asarray(S[heads, col]).ravel(), atol=1e-5)
    ours, theirs = set(zip(heads.tolist(), col.tolist())), set(
        zip(np.repeat(np.arange(n), np.diff(o["row_ptr"])).tolist(), o["col"].tolist()))
    for i, j in ours ^ theirs:
        assert abs(S[i, j] - 1.0 / T) <= 1e-5 + 2.0 ** -23
