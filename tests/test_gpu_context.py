"""What a context promises around the kernels: its memory cap covers every
buffer it keeps, searches that were enqueued return before they run and do not
wait for other streams', every kernel is counted, and the stage times of a fit
stay the fit's (gpu)."""
import ctypes as C

import pytest

from gpu_util import drgb_module

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture
def drgb():
    """The module with a context of its own."""
    m = drgb_module()
    m.context()
    lib = m._lib.load()
    own = C.c_void_p()
    assert lib.drgb_ctx_create(0, C.byref(own)) == 0
    saved, m._contexts[0] = m._contexts[0], own.value
    yield m
    m._contexts[0] = saved
    lib.drgb_ctx_destroy(own)


def _points(n, d, seed=0):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    c = 5.0 * torch.randn((20, d), generator=g, device="cuda")
    return c[torch.randint(0, 20, (n,), generator=g, device="cuda")] + torch.randn((n, d), generator=g, device="cuda")


def _render(drgb, side):
    """A call whose scratch is 16 bytes a pixel."""
    import torch
    Y, rgb = torch.rand(10, 2, device="cuda"), torch.rand(10, 3, device="cuda")
    return drgb.render(Y, rgb, width=side, height=side, radius=2.0)


# ------------------------------------------------------------------ memory
@pytest.mark.parametrize("mode", [0, 1])
def test_held_memory_is_reported_and_capped(drgb, mode):
    import torch
    lib, ctx = drgb._lib.load(), drgb.context()
    X = _points(20000, 150)
    want = drgb.knn_graph(X, 15, mode=mode)  # (outputs and modules are loaded once)
    torch.cuda.synchronize()
    own = C.c_void_p()
    assert lib.drgb_ctx_create(0, C.byref(own)) == 0
    saved, drgb._contexts[0] = drgb._contexts[0], own.value
    try:
        torch.cuda.synchronize()
        free0 = torch.cuda.mem_get_info()[0]
        got = drgb.knn_graph(X, 15, mode=mode)
        torch.cuda.synchronize()
        lost = free0 - torch.cuda.mem_get_info()[0]
        assert lib.drgb_ctx_scratch_bytes(own) >= lost - 4 * MB
        assert lib.drgb_set_scratch_limit(own, 1 * MB) == 0
        assert lib.drgb_ctx_scratch_bytes(own) <= 1 * MB
        assert free0 - torch.cuda.mem_get_info()[0] <= 4 * MB
        again = drgb.knn_graph(X, 15, mode=mode)  # without room for lists: the same result
        torch.cuda.synchronize()
        assert lib.drgb_ctx_scratch_bytes(own) <= 1 * MB
    finally:
        drgb._contexts[0] = saved
        lib.drgb_ctx_destroy(own)
    for r in (got, again):
        assert torch.equal(r[0], want[0]) and torch.equal(r[1], want[1])


def test_buffers_of_two_kinds_share_one_cap(drgb):
    import torch
    lib, ctx = drgb._lib.load(), drgb.context()
    held = lambda: lib.drgb_ctx_scratch_bytes(ctx)
    cap = 200 * MB
    X = _points(5000, 150)
    want = drgb.knn_graph(X, 15)
    _render(drgb, 3400)  # 176 MB beside the search's buffer
    torch.cuda.synchronize()
    assert held() > cap
    assert lib.drgb_set_scratch_limit(ctx, cap) == 0
    assert held() <= cap
    for _ in range(2):  # each needs less than the cap by itself
        _render(drgb, 3400)
        assert held() <= cap
        got = drgb.knn_graph(X, 15)
        torch.cuda.synchronize()
        assert held() <= cap
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    assert lib.drgb_set_scratch_limit(ctx, 0) == 0


# ------------------------------------------------------------------ streams
# sizes at which auto mode takes the product over all points, below and above
# the cell-ordered form's width, and the scan
SEARCHES = [(2000, 50, 0), (9000, 50, 0), (3000, 200, 0), (2000, 50, 1), (3000, 200, 1), (900, 20, 0)]


def _busy(stream):
    """About half a second of a one-thread kernel on `stream`; an event after it."""
    import torch
    with torch.cuda.stream(stream):
        torch.cuda._sleep(1_000_000_000)
        ev = torch.cuda.Event()
        ev.record(stream)
    return ev


@pytest.mark.parametrize("n,d,mode", SEARCHES)
def test_search_returns_before_it_runs(drgb, n, d, mode):
    import torch
    X = _points(n, d)
    want = drgb.knn_graph(X, 15, mode=mode)
    torch.cuda.synchronize()
    busy = _busy(torch.cuda.current_stream())
    got = drgb.knn_graph(X, 15, mode=mode)
    assert not busy.query()  # enqueued behind it
    torch.cuda.synchronize()
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


@pytest.mark.parametrize("n,d,mode", SEARCHES)
def test_searches_on_two_streams_do_not_wait_for_each_other(drgb, n, d, mode):
    import torch
    X = _points(n, d)
    want = drgb.knn_graph(X, 15, mode=mode)
    torch.cuda.synchronize()
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(2):  # (the second time nothing grows)
        busy = _busy(s1)
        with torch.cuda.stream(s1):
            a = drgb.knn_graph(X, 15, mode=mode)
        with torch.cuda.stream(s2):
            b = drgb.knn_graph(X, 15, mode=mode)
        s2.synchronize()
        assert not busy.query()
        torch.cuda.synchronize()
        for r in (a, b):
            assert torch.equal(r[0], want[0]) and torch.equal(r[1], want[1])


def test_counters_wait_for_the_search(drgb):
    # asked on another stream than the search's, which is still behind other work
    import torch
    X = _points(3000, 200)
    X[100:200] = X[:1]  # copies: more than the candidate lists hold
    drgb.knn_graph(X, 15)
    want = (drgb.knn_uncertified(), drgb.knn_tiles())
    assert want[0] >= 100
    drgb.knn_graph(_points(2000, 50), 15)
    assert (drgb.knn_uncertified(), drgb.knn_tiles()) != want
    s1 = torch.cuda.Stream()
    _busy(s1)
    with torch.cuda.stream(s1):
        drgb.knn_graph(X, 15)
    assert (drgb.knn_uncertified(), drgb.knn_tiles()) == want


def test_searches_on_many_streams_with_growth(drgb):
    # more streams than the context keeps buffers, sizes that grow in between
    import torch
    sets = [_points(n, d, n) for n, d in ((1500, 70), (3000, 200), (6000, 90), (2000, 50))]
    want = [drgb.knn_graph(X, 15, mode=1) for X in sets]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(12)]
    outs = []
    for i in range(48):
        with torch.cuda.stream(streams[i % 12]):
            outs.append((i % 4, drgb.knn_graph(sets[i % 4], 15)))
    torch.cuda.synchronize()
    for k, r in outs:
        assert torch.equal(r[0], want[k][0]) and torch.equal(r[1], want[k][1])


def test_search_beside_a_capture_on_another_stream(drgb):
    # a stream being captured in the global mode forbids what may synchronise the
    # device; a search enqueued on another stream meanwhile still runs
    import torch
    lib, ctx = drgb._lib.load(), drgb.context()
    X = _points(2000, 50)
    want = drgb.knn_graph(X, 15)
    X2 = _points(2600, 50)
    want2 = drgb.knn_graph(X2, 15, mode=1)
    idx, dist = torch.empty_like(want2[0]), torch.empty_like(want2[1])
    lib.drgb_set_scratch_limit(ctx, 1)  # (the buffer has to be allocated again)
    lib.drgb_set_scratch_limit(ctx, 0)
    other = torch.cuda.Stream()
    z = torch.zeros(8, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        z.add_(1.0)
        rc = lib.drgb_knn_graph(ctx, C.c_void_p(X2.data_ptr()), 2600, 50, 15, 0, C.c_void_p(idx.data_ptr()),
                                C.c_void_p(dist.data_ptr()), C.c_void_p(other.cuda_stream))
    g.replay()
    torch.cuda.synchronize()
    assert rc == 0 and float(z[0]) == 1.0
    assert torch.equal(idx, want2[0]) and torch.equal(dist, want2[1])


# ------------------------------------------------------------------ counters
def _counted(drgb, f):
    before = drgb.launch_count()
    f()
    return drgb.launch_count() - before


def test_every_kernel_is_counted(drgb):
    import torch
    X = _points(3000, 50)
    P = drgb.mlp_init(50, seed=1)
    rows = torch.randint(0, 3000, (64 * 7,), dtype=torch.int32, device="cuda")
    # weights, gather, two layers, head, layer 3 backward, three weight
    # gradients, dH1, column sums, gradient
    assert _counted(drgb, lambda: drgb.mlp_grad(P, X, rows, 64, 5, 1.577, 0.895)) == 12
    g = drgb.fuzzy_weights(*drgb.knn_graph(X, 15), 200)

    def train(steps):
        Q = P.clone()
        drgb.mlp_train(X, g, 1.577, 0.895, Q, torch.zeros_like(Q), torch.zeros_like(Q), steps, batch_edges=64)
    few, more = (_counted(drgb, lambda s=s: train(s)) for s in (3, 8))
    # a step: a gradient's ten without weights and gather, the next batch's two
    assert more - few == 5 * 12
    assert few == 3 * 12 + 4  # and before the first: heads, weights, batch
    # at least the start's three orthonormalisations of three kernels and one
    # Rayleigh-Ritz step of six beside means, covariance and projection
    assert _counted(drgb, lambda: drgb.pca(_points(2000, 100), 5)) >= 9 + 6 + 8


def test_stage_times_stay_the_fits(drgb):
    import torch
    X = _points(5000, 50)
    drgb.set_profiling(True)
    try:
        Y = drgb.fit_transform(X, n_epochs=20)
        t = drgb.stage_times()
        drgb.transform(X, Y, _points(4000, 50, 1), n_epochs=9)
        drgb.eval_recall(X, Y, 15, 1000)
        drgb.eval_recall_heldout(X, Y, X[:4000].contiguous(), Y[:4000].contiguous(), 15)
        drgb.knn_graph(_points(3000, 50, 2), 15)
        drgb.knn_graph(_points(3000, 200, 2), 15)
        torch.cuda.synchronize()
        assert drgb.stage_times() == t
    finally:
        drgb.set_profiling(False)
