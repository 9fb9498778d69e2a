"""Contexts of their own in two host threads, calls of different shared-memory
sizes at the same time: what a kernel may use is a setting of the process, so no
call may lower it under another's launch (gpu)."""
import ctypes as C
import threading

import pytest

from gpu_util import drgb_module

pytestmark = pytest.mark.gpu


def _run(drgb, jobs, rounds):
    """jobs: one function of a context and a stream per thread; the return codes that are not 0."""
    import torch
    lib, bad = drgb._lib.load(), []
    ready = threading.Barrier(len(jobs))

    def work(job):
        torch.cuda.set_device(0)
        ctx, stream = C.c_void_p(), torch.cuda.Stream()
        assert lib.drgb_ctx_create(0, C.byref(ctx)) == 0
        ready.wait()
        for _ in range(rounds):
            rc = job(lib, ctx, C.c_void_p(stream.cuda_stream))
            if rc:
                bad.append((rc, lib.drgb_last_error(ctx).decode()))
        stream.synchronize()
        lib.drgb_ctx_destroy(ctx)
    threads = [threading.Thread(target=work, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return bad


def _p(t):
    return C.c_void_p(t.data_ptr())


def test_scans_of_different_sizes():
    import torch
    drgb = drgb_module()

    def scan(n, d, k):
        X = torch.randn(n, d, device="cuda")
        idx, dist = torch.empty(n, k, dtype=torch.int32, device="cuda"), torch.empty(n, k, device="cuda")
        torch.cuda.synchronize()
        return lambda lib, ctx, st: lib.drgb_knn_graph(ctx, _p(X), n, d, k, 1, _p(idx), _p(dist), st)
    assert _run(drgb, [scan(200, 64, 32), scan(200, 3, 5), scan(200, 20, 16)], 3000) == []


def test_fuzzy_rows_of_different_lengths():
    import torch
    drgb = drgb_module()

    def fuzzy(n, k):
        idx = (torch.arange(n, device="cuda")[:, None] + torch.arange(1, k + 1, device="cuda")) % n
        idx = idx.int().contiguous()
        dist = torch.rand(n, k, device="cuda").sort(1).values
        rp = torch.empty(n + 1, dtype=torch.int32, device="cuda")
        col, q = (torch.empty(2 * n * k, dtype=torch.int32, device="cuda") for _ in range(2))
        w = torch.empty(2 * n * k, device="cuda")
        torch.cuda.synchronize()
        return lambda lib, ctx, st: lib.drgb_fuzzy_weights(ctx, _p(idx), _p(dist), n, k, 200, _p(rp), _p(col), _p(w), _p(q),
                                                          2 * n * k, None, None, st)
    assert _run(drgb, [fuzzy(300, 32), fuzzy(300, 17), fuzzy(300, 31)], 2000) == []
