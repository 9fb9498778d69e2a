"""The tensor-core search of separate queries against the FP32 scan, bit for bit
through transform(), whose start and forces follow from the neighbours and
their distances: with too little scratch for the product the same call scans.
Matrices whose base is only 4- or 8-byte aligned take narrower copies (gpu)."""
import pytest

from gpu_util import drgb_module

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def drgb():
    return drgb_module()


def _points(n, d, seed, kind, shift=0):
    """n x d points whose base lies `shift` floats past a 256-byte boundary."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    if kind == "ties":  # small integers: many equal distances, copies of points
        X = torch.randint(-2, 3, (n, d), generator=g, device="cuda").float()
        X[n // 2:n // 2 + 40] = X[7]
    else:
        c = 5.0 * torch.randn((30, d), generator=torch.Generator(device="cuda").manual_seed(d), device="cuda")
        X = c[torch.randint(0, 30, (n,), generator=g, device="cuda")] + torch.randn((n, d), generator=g, device="cuda") + 100.0
    out = torch.empty(n * d + shift, device="cuda")[shift:].view(n, d)
    out.copy_(X)
    assert out.is_contiguous() and out.data_ptr() % 16 == 4 * shift % 16
    return out


def _scanned(drgb, f):
    """f() with room for its own buffers but not for the product's (64 MB of lists and more)."""
    lib, ctx = drgb._lib.load(), drgb.context()
    assert lib.drgb_set_scratch_limit(ctx, 48 << 20) == 0
    try:
        return f()
    finally:
        lib.drgb_set_scratch_limit(ctx, 0)


@pytest.mark.parametrize("kind", ["clusters", "ties"])
@pytest.mark.parametrize("n,m,d,k,sx,sq", [(60001, 1025, 50, 15, 0, 0), (70000, 3000, 16, 31, 1, 0), (1024, 20000, 61, 5, 0, 1),
                                           (5000, 4000, 200, 15, 0, 0), (5000, 4000, 200, 15, 1, 0), (5000, 4000, 200, 15, 0, 3),
                                           (5000, 4000, 200, 15, 2, 0), (5000, 4000, 200, 15, 2, 2), (9000, 700, 62, 1, 2, 1),
                                           (2100, 2100, 1021, 16, 0, 0)])
def test_separate_queries_equal_the_scan(drgb, n, m, d, k, kind, sx, sq):
    import torch
    X, Q = _points(n, d, 1, kind, sx), _points(m, d, 2, kind, sq)
    Y = torch.randn(n, 2, device="cuda")
    run = lambda: drgb.transform(X, Y, Q, k=k, n_epochs=3)
    got = run()
    assert torch.equal(got, _scanned(drgb, run))


@pytest.mark.parametrize("d,shift", [(200, 1), (200, 2), (202, 1), (64, 3)])
def test_graph_of_a_matrix_off_the_boundary(drgb, d, shift):
    import torch
    X = _points(4100, d, 3, "clusters", shift)
    got, want = drgb.knn_graph(X, 15), drgb.knn_graph(X, 15, mode=1)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


@pytest.mark.parametrize("n", [16383, 16384, 20001])
@pytest.mark.parametrize("d,k", [(3, 15), (16, 30), (61, 5)])
def test_uncertified_rows_on_both_sides_of_the_cells_line(drgb, n, d, k):
    # many copies of a point leave rows uncertified: scanned over all points, or
    # over the cells they reach
    import torch
    g = torch.Generator(device="cuda").manual_seed(n + d)
    X = torch.randn(n // 20, d, generator=g, device="cuda")[torch.randint(0, n // 20, (n,), generator=g, device="cuda")]
    got = drgb.knn_graph(X, k, mode=3)
    assert drgb.knn_uncertified() > 0
    want = drgb.knn_graph(X, k, mode=1)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
