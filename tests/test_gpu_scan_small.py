"""The scan of a small database, a warp a query, on both sides of its line and at
the edges of its tiles (32 points) and steps (64 dimensions): small integers
against brute force, where equal distances are frequent and the order by
(distance, index) has to hold bit for bit; non-finite and overflowing rows against
the tiled scan of the same points (gpu)."""
import numpy as np
import pytest

from gpu_util import drgb_module
from test_gpu_scan import _d2, _ints, _nearest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,k", [(2, 1, 1), (3, 5, 2), (31, 8, 15), (32, 8, 31), (33, 8, 32), (40, 64, 15), (64, 65, 5),
                                   (97, 127, 16), (200, 128, 32), (400, 70, 15), (401, 70, 15), (1200, 64, 15), (1201, 64, 15),
                                   (1199, 2, 32), (1000, 1, 7)])
def test_graph_orders_by_distance_then_index(n, d, k):
    import torch
    drgb = drgb_module()
    X = _ints(n, d, n + d)
    D = _d2(X, X).astype(np.float64)
    np.fill_diagonal(D, np.inf)
    oi, od = _nearest(D, k)
    idx, dist = drgb.knn_graph(torch.from_numpy(X).cuda(), k, mode=1)
    np.testing.assert_array_equal(idx.cpu().numpy(), oi)
    np.testing.assert_array_equal(dist.cpu().numpy(), od)


@pytest.mark.parametrize("n,m,d,k", [(33, 1, 3, 5), (300, 20000, 20, 10), (300, 20001, 20, 10), (1200, 777, 64, 15), (400, 2000, 66, 16)])
def test_separate_and_listed_queries(n, m, d, k):
    import torch
    drgb = drgb_module()
    X, Y, Q, P = _ints(n, d, 1), _ints(n, 2, 2), _ints(m, d, 3), _ints(m, 2, 4)
    dev = lambda a: torch.from_numpy(a).cuda()
    nx, ny = _nearest(_d2(Q, X), k)[0], _nearest(_d2(P, Y), k)[0]
    hits = int((nx[:, :, None] == ny[:, None, :]).sum())
    assert drgb.eval_recall_heldout(dev(X), dev(Y), dev(Q), dev(P), k) == hits / (k * m)
    q = min(n, 57)  # listed rows of the database itself
    rows = np.arange(q) * n // q
    DX, DY = _d2(X[rows], X).astype(np.float64), _d2(Y[rows], Y).astype(np.float64)
    DX[np.arange(q), rows] = DY[np.arange(q), rows] = np.inf
    hits = int((_nearest(DX, k)[0][:, :, None] == _nearest(DY, k)[0][:, None, :]).sum())
    assert drgb.eval_recall(dev(X), dev(Y), k, q) == hits / (k * q)


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf"), 3e19, 0.0])
def test_rows_without_finite_distances(bad):
    # the same points, padded with far copies to a size that the tiled scan takes, give
    # the small scan's rows wherever the padding is farther than every neighbour
    import torch
    drgb = drgb_module()
    g = torch.Generator(device="cuda").manual_seed(1)
    X = torch.randn((500, 20), generator=g, device="cuda")
    X[7], X[130, 3], X[499] = bad, bad, bad
    Z = torch.cat([X, 1000.0 + torch.randn((2000, 20), generator=g, device="cuda")])
    small, tiled = drgb.knn_graph(X, 15, mode=1), drgb.knn_graph(Z, 15, mode=1)
    assert torch.equal(small[0], tiled[0][:500]) and torch.equal(small[1], tiled[1][:500])
    far = small[0] < 0  # (two copies of an overflowing row still have each other)
    assert bool(far.any()) == (bad != 0.0) and bool(torch.isinf(small[1][far]).all())
