"""The FP32 scan (k nearest, queries against a database, ranks) at the edges of
its tiles, against brute force on small integers: squared distances are then
exact in FP32, equal distances are frequent, and the order by (distance, index)
has to hold bit for bit."""
import numpy as np
import pytest

from gpu_util import drgb_module

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def drgb():
    return drgb_module()


def _ints(n, d, seed):
    return np.random.default_rng(seed).integers(-3, 4, (n, d)).astype(np.float32)


def _d2(Q, X):
    q, x = Q.astype(np.int64), X.astype(np.int64)
    return (q * q).sum(1)[:, None] + (x * x).sum(1)[None, :] - 2 * q @ x.T


def _nearest(D, k):
    order = np.argsort(D, axis=1, kind="stable")[:, :k]
    return order, np.sqrt(np.take_along_axis(D, order, 1).astype(np.float32))


# n around the 64-query block, the 128-point tile and the chunk of two tiles;
# d around the 32-dimension stage and the 64 dimensions kept in shared memory
@pytest.mark.parametrize("n,d,k", [(2, 1, 1), (63, 2, 16), (65, 31, 17), (128, 32, 32), (129, 33, 15), (513, 64, 15),
                                   (1000, 65, 5), (2049, 3, 31), (4095, 50, 15), (700, 130, 16)])
def test_scan_orders_by_distance_then_index(drgb, n, d, k):
    import torch
    X = _ints(n, d, n + d)
    D = _d2(X, X).astype(np.float64)
    np.fill_diagonal(D, np.inf)
    oi, od = _nearest(D, k)
    Xd = torch.from_numpy(X).cuda()
    idx, dist = drgb.knn_graph(Xd, k, mode=1)
    np.testing.assert_array_equal(idx.cpu().numpy(), oi)
    np.testing.assert_array_equal(dist.cpu().numpy(), od)
    ctx = drgb.context()
    lib = drgb._lib.load()
    lib.drgb_set_scratch_limit(ctx, 1)  # no room for partial lists: the unsplit scan
    try:
        idx1, dist1 = drgb.knn_graph(Xd, k, mode=1)
        torch.cuda.synchronize()
    finally:
        lib.drgb_set_scratch_limit(ctx, 0)
    assert torch.equal(idx, idx1) and torch.equal(dist, dist1)


@pytest.mark.parametrize("n,m,d,k", [(300, 300, 7, 10), (3001, 777, 40, 15), (2000, 65, 70, 30)])
def test_quality_scores_equal_brute_force(drgb, n, m, d, k):
    import torch
    X, Y = _ints(n, d, 1), _ints(n, 2, 2)
    rows = np.arange(m) * n // m
    DX, DY = _d2(X[rows], X).astype(np.float64), _d2(Y[rows], Y).astype(np.float64)
    DX[np.arange(m), rows] = DY[np.arange(m), rows] = np.inf
    nx, ny = _nearest(DX, k)[0], _nearest(DY, k)[0]
    hits = sum(len(set(a) & set(b)) for a, b in zip(nx, ny))
    rank = np.argsort(np.argsort(DX, axis=1, kind="stable"), axis=1) + 1
    excess = np.maximum(np.take_along_axis(rank, ny, 1) - k, 0).sum()
    Xd, Yd = torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda()
    assert drgb.eval_recall(Xd, Yd, k, m) == hits / (k * m)
    assert drgb.eval_trust(Xd, Yd, k, m) == pytest.approx(1 - 2 / (m * k * (2.0 * n - 3 * k - 1)) * excess, abs=1e-14)
    # queries from another matrix: nothing is excluded
    Q, P = _ints(m, d, 3), _ints(m, 2, 4)
    hits = sum(len(set(a) & set(b)) for a, b in zip(_nearest(_d2(Q, X), k)[0], _nearest(_d2(P, Y), k)[0]))
    got = drgb.eval_recall_heldout(Xd, Yd, torch.from_numpy(Q).cuda(), torch.from_numpy(P).cuda(), k)
    assert got == hits / (k * m)


def test_scan_under_capture_and_on_two_streams(drgb):
    import torch
    X = torch.from_numpy(_ints(1500, 20, 5)).cuda()
    want = drgb.knn_graph(X, 15, mode=1)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        got = drgb.knn_graph(X, 15, mode=1)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(want[0], got[0]) and torch.equal(want[1], got[1])
    streams = [torch.cuda.Stream() for _ in range(2)]
    outs = []
    for i in range(6):
        with torch.cuda.stream(streams[i % 2]):
            outs.append(drgb.knn_graph(X, 15, mode=1))
    torch.cuda.synchronize()
    assert all(torch.equal(want[0], o[0]) for o in outs)
