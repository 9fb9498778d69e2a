"""How windows are dealt over the warps of an epoch's grid does not show in
the result: the pipelined form (dealt over all CTAs) and the flat form (CTAs of
consecutive windows) give the same bits (gpu)."""
import numpy as np
import pytest

from gpu_util import drgb_module

pytestmark = pytest.mark.gpu


@pytest.fixture
def drgb():
    """The module with a context of its own (a form once chosen stays chosen)."""
    import ctypes as C
    m = drgb_module()
    m.context()
    lib = m._lib.load()
    own = C.c_void_p()
    assert lib.drgb_ctx_create(0, C.byref(own)) == 0
    saved, m._contexts[0] = m._contexts[0], own.value
    yield m
    m._contexts[0] = saved
    lib.drgb_ctx_destroy(own)


# windows of 512 entries: fewer than the CTAs, one more than they, one a warp and one more, two rounds and a rest
@pytest.mark.parametrize("windows", [1, 7, 455, 457, 1000, 3648, 3649, 7500])
@pytest.mark.parametrize("warps", [4, 8])
def test_forms_agree(drgb, windows, warps):
    import torch
    rng = np.random.default_rng(windows)
    n = max(2, windows * 512 // 16 - 5)
    deg = np.full(n, 16)
    deg[rng.integers(0, n, n // 50)] = 0
    deg[n // 2] = 900
    rp = np.concatenate([[0], np.cumsum(deg)]).astype(np.int32)
    nnz = int(rp[-1])
    dev = lambda a: torch.from_numpy(a).cuda()
    g = drgb.Graph(dev(rp), dev(rng.integers(0, n, nnz).astype(np.int32)), dev(np.ones(nnz, np.float32)),
                   dev(rng.integers(1 << 16, 1 << 24, nnz).astype(np.int32)))
    Y = dev(rng.uniform(-10, 10, (n, 2)).astype(np.float32))
    drgb.set_tuning(1, warps)
    out = []
    for pipe in (1, 0):
        drgb.set_tuning(2, pipe)
        out.append(drgb.embed_epoch(Y, g, 1.577, 0.895, 0.7, 5, 11, 5))
    assert torch.equal(*out)
