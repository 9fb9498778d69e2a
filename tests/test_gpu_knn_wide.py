"""The tensor-core search for wide rows and for separate queries returns the
FP32 scan's result bit for bit, at the edges of its tiles, K steps and splits."""
import numpy as np
import pytest

from gpu_util import drgb_module

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def drgb():
    return drgb_module()


def _points(torch, n, d, seed, kind):
    g = torch.Generator(device="cuda").manual_seed(seed)
    if kind == "ties":  # small integers: many equal distances, copies of points
        X = torch.randint(-2, 3, (n, d), generator=g, device="cuda").float()
        X[n // 2:n // 2 + 40] = X[7]
        return X
    c = 5.0 * torch.randn((30, d), generator=g, device="cuda")
    return c[torch.randint(0, 30, (n,), generator=g, device="cuda")] + torch.randn((n, d), generator=g, device="cuda") + 100.0


# d + 3 columns around the 64-column K step (62: the first width past the
# cell-ordered kernel; 253 and 254: 4 and 5 steps; 1021: the last width taken,
# 1022: the scan); n ragged against the 128-query block and 256-row tile
@pytest.mark.parametrize("kind", ["clusters", "ties"])
@pytest.mark.parametrize("n,d,k", [(7001, 62, 15), (6913, 125, 1), (4000, 253, 31), (4097, 254, 16), (2050, 784, 15),
                                   (1800, 1021, 10), (1800, 1022, 10), (5000, 200, 32), (1733, 50, 15), (4096, 16, 15),
                                   (13999, 61, 15)])
def test_wide_graph_equals_scan(drgb, n, d, k, kind):
    import torch
    X = _points(torch, n, d, n + d, kind)
    got, want = drgb.knn_graph(X, k), drgb.knn_graph(X, k, mode=1)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


@pytest.mark.parametrize("kind", ["clusters", "ties"])
@pytest.mark.parametrize("n,m,d,k", [(60001, 1025, 50, 15), (70000, 3000, 16, 31), (1024, 60000, 61, 5),
                                     (5000, 4000, 200, 15)])
def test_held_out_recall_of_wide_queries(drgb, n, m, d, k, kind):
    import torch
    X, Q = _points(torch, n, d, 1, kind), _points(torch, m, d, 2, kind)
    Y, P = X[:, :2].contiguous(), Q[:, :2].contiguous()
    rows = torch.arange(m, device="cuda")
    # neighbours in 64 bits: exact for the integers; for the clusters a near-tie may differ
    hits = 0
    for r in rows.split(1000):
        nx = torch.cdist(Q[r].double(), X.double(), compute_mode="donot_use_mm_for_euclid_dist").sort(dim=1, stable=True).indices[:, :k]
        ny = torch.cdist(P[r].double(), Y.double(), compute_mode="donot_use_mm_for_euclid_dist").sort(dim=1, stable=True).indices[:, :k]
        hits += int((nx[:, :, None] == ny[:, None, :]).sum())
    got = drgb.eval_recall_heldout(X, Y, Q, P, k)
    assert abs(got - hits / (k * m)) <= (0 if kind == "ties" else 8.0 / (k * m))


def test_wide_graph_without_room_or_finite_values(drgb):
    import torch
    X = _points(torch, 5000, 150, 3, "clusters")
    want = drgb.knn_graph(X, 15, mode=1)
    lib, ctx = drgb._lib.load(), drgb.context()
    lib.drgb_set_scratch_limit(ctx, 1)
    try:
        got = drgb.knn_graph(X, 15)
        torch.cuda.synchronize()
    finally:
        lib.drgb_set_scratch_limit(ctx, 0)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    for bad in (float("nan"), float("inf"), 1e30):
        Xb = X.clone()
        Xb[17, 3] = bad
        got, want = drgb.knn_graph(Xb, 15), drgb.knn_graph(Xb, 15, mode=1)
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    g = torch.cuda.CUDAGraph()
    want = drgb.knn_graph(X, 15, mode=1)
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        got = drgb.knn_graph(X, 15)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(got[0], want[0])
