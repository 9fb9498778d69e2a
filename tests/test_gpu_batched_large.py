"""Batches on both sides of the line between the one-launch loop of epochs (11
windows of 512 entries an SM) and a launch an epoch: each instance keeps the
bits of its own fit, for every force-kernel setting (gpu)."""
import ctypes as C

import numpy as np
import pytest

import datagen
from gpu_util import drgb_module

pytestmark = pytest.mark.gpu


@pytest.fixture
def drgb():
    """The module with a context of its own (a form once chosen stays chosen)."""
    m = drgb_module()
    m.context()
    lib = m._lib.load()
    own = C.c_void_p()
    assert lib.drgb_ctx_create(0, C.byref(own)) == 0
    saved, m._contexts[0] = m._contexts[0], own.value
    yield m
    m._contexts[0] = saved
    lib.drgb_ctx_destroy(own)


def _instances(sizes):
    parts = [datagen.mixture(int(nb), 20, 5 + b % 7, seed=70 + b)[0] for b, nb in enumerate(sizes)]
    return np.ascontiguousarray(np.concatenate(parts)), np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)


def _check(drgb, sizes, settings, **params):
    import torch
    X, off = _instances(sizes)
    Xd = torch.from_numpy(X).cuda()
    si, sn = [11 + 7 * b for b in range(len(sizes))], [101 + 13 * b for b in range(len(sizes))]
    want = [drgb.fit_transform(Xd[off[b]:off[b + 1]].contiguous(), seed_init=si[b], seed_neg=sn[b], **params)
            for b in range(len(sizes))]
    for s in settings:
        if s:
            drgb.set_tuning(1, s[0])
            drgb.set_tuning(2, s[1])
        Y = drgb.fit_transform_batched(Xd, off, si, sn, **params)
        for b in range(len(sizes)):
            assert torch.equal(Y[off[b]:off[b + 1]], want[b]), f"instance {b} (n={sizes[b]}), setting {s}"


@pytest.mark.parametrize("neg", [5, 3, 9])
def test_a_launch_an_epoch(drgb, neg):
    # 43,609 rows of 15 neighbours: 2,563 windows
    _check(drgb, [16, 500, 20000, 60, 14000, 9000, 33], [None, (4, 1), (4, 0), (8, 1), (8, 0)], n_epochs=12, neg=neg)


@pytest.mark.parametrize("past", [0, 1])
def test_both_sides_of_the_line(drgb, past):
    import torch
    limit = 11 * torch.cuda.get_device_properties(0).multi_processor_count
    sizes = [700, 16, 5000, 40]
    # capacity: ceil(2 n k / 512) windows and one an instance
    n = (limit - 5) * 512 // 30 + past
    sizes.append(n - sum(sizes))
    assert (-(-30 * n // 512) + 5 <= limit) == (past == 0)
    _check(drgb, sizes, [None, (8, 0)], n_epochs=11)
