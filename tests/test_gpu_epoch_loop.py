"""A loop of epochs in one launch gives the bits of the same epochs run one by
one (embed_epoch, whose kernel has its own tests against the oracle): windows
with no, one and many groups, rows longer than a round, empty rows, negative
counts around the compile-time one, odd and even numbers of epochs."""
import numpy as np
import pytest

from gpu_util import drgb_module

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def drgb():
    return drgb_module()


def _graph(drgb, n, degrees, seed, full=0.3):
    """Random CSR with the given row degrees; a share `full` of the entries fires every epoch."""
    import torch
    rng = np.random.default_rng(seed)
    rp = np.concatenate([[0], np.cumsum(degrees)]).astype(np.int32)
    nnz = int(rp[-1])
    col = rng.integers(0, n, nnz).astype(np.int32)
    q = np.where(rng.uniform(size=nnz) < full, 1 << 24, rng.integers(1 << 16, 1 << 24, nnz)).astype(np.int32)
    dev = lambda a: torch.from_numpy(a).cuda()
    return drgb.Graph(dev(rp), dev(col), dev(np.ones(max(nnz, 1), np.float32)[:nnz]), dev(q))


def _degrees(kind, n, rng):
    d = rng.integers(0, 30, n)
    if kind == "hubs":
        d[n // 3] = 2000   # several rounds, all of its groups one run
        d[n // 2] = 769
        d[n // 2 + 1:n // 2 + 40] = 0
        d[-1] = 600
    elif kind == "sparse":
        d = (rng.uniform(size=n) < 0.01).astype(np.int64)
        d[:5] = 0
        d[-50:] = 0
    elif kind == "full":
        d = np.full(n, 32)
    return d


@pytest.mark.parametrize("kind,n,neg,t0,t1", [
    ("mixed", 3, 5, 0, 7), ("mixed", 700, 5, 0, 40), ("mixed", 700, 0, 3, 20), ("mixed", 900, 4, 0, 15), ("mixed", 900, 9, 0, 15),
    ("mixed", 900, 64, 0, 4), ("hubs", 3000, 5, 0, 33), ("hubs", 9000, 3, 10, 30), ("sparse", 4000, 5, 0, 20), ("full", 5000, 5, 0, 12),
    ("mixed", 30000, 5, 100, 112), ("hubs", 70000, 5, 0, 6), ("mixed", 2000, 5, 0, 300)])
def test_loop_equals_single_epochs(drgb, kind, n, neg, t0, t1):
    import torch
    rng = np.random.default_rng(n + neg)
    g = _graph(drgb, n, _degrees(kind, n, rng), n)
    Y0 = torch.from_numpy(rng.uniform(-10, 10, (n, 2)).astype(np.float32)).cuda()
    T = 300
    got = drgb.embed_epochs(Y0.clone(), g, 1.577, 0.895, 1.0, neg, t0, t1, T, 12345678901)
    want = Y0
    for t in range(t0, t1):
        want = drgb.embed_epoch(want, g, 1.577, 0.895, float(np.float32(1.0 * (1.0 - t / T))), neg, t, 12345678901)
    assert torch.equal(got, want)


def test_loop_without_entries_and_with_malformed_rows(drgb):
    import torch
    Y0 = torch.randn(100, 2, device="cuda")
    g = drgb.Graph(*(torch.zeros(k, dtype=t, device="cuda") for k, t in
                     ((101, torch.int32), (1, torch.int32), (1, torch.float32), (1, torch.int32))))
    assert torch.equal(drgb.embed_epochs(Y0.clone(), g, 1.577, 0.895, 1.0, 5, 0, 3, 10, 1), Y0)
    rng = np.random.default_rng(0)
    bad = _graph(drgb, 500, rng.integers(1, 20, 500), 1, full=1.0)
    bad.col[7] = 500  # not a row
    drgb.embed_epochs(torch.randn(500, 2, device="cuda"), bad, 1.577, 0.895, 1.0, 5, 0, 4, 10, 1)
    lib, ctx = drgb._lib.load(), drgb.context()
    assert lib.drgb_sync(ctx, None) != 0  # reported by the next synchronising call
    assert lib.drgb_sync(ctx, None) == 0
