"""Fits, layouts and transforms of small data on a stream that may use only some
of the SMs (a green context's): there the loop of epochs in one cooperative
launch may be refused, and a launch an epoch runs instead (gpu)."""
import ctypes as C

import pytest

from gpu_util import drgb_module

pytestmark = pytest.mark.gpu


class _Resource(C.Structure):  # CUdevResource
    _fields_ = [("type", C.c_int), ("padding", C.c_ubyte * 92), ("sm_count", C.c_uint), ("rest", C.c_ubyte * 256)]


def _limited_stream(sms):
    """A stream of a green context of about `sms` SMs, and how many it got."""
    cu = C.CDLL("libcuda.so.1")

    def ok(rc, what):
        if rc:
            pytest.skip(f"{what}: CUDA error {rc}")
    dev, whole, part, rest = C.c_int(), _Resource(), _Resource(), _Resource()
    ok(cu.cuDeviceGet(C.byref(dev), 0), "device")
    ok(cu.cuDeviceGetDevResource(dev, C.byref(whole), 1), "resources")  # CU_DEV_RESOURCE_TYPE_SM
    groups = C.c_uint(1)
    ok(cu.cuDevSmResourceSplitByCount(C.byref(part), C.byref(groups), C.byref(whole), C.byref(rest), C.c_uint(0), C.c_uint(sms)),
       "split")
    desc, green, stream = C.c_void_p(), C.c_void_p(), C.c_void_p()
    ok(cu.cuDevResourceGenerateDesc(C.byref(desc), C.byref(part), C.c_uint(1)), "descriptor")
    ok(cu.cuGreenCtxCreate(C.byref(green), desc, dev, C.c_uint(1)), "green context")  # CU_GREEN_CTX_DEFAULT_STREAM
    ok(cu.cuGreenCtxStreamCreate(C.byref(stream), green, C.c_uint(1), C.c_int(0)), "stream")  # CU_STREAM_NON_BLOCKING
    return stream.value, part.sm_count


def test_small_work_on_a_few_sms():
    import torch
    drgb = drgb_module()
    X, X_new = torch.randn(9000, 30, device="cuda"), torch.randn(4000, 30, device="cuda")
    idx, dist = drgb.knn_graph(X, 15)
    g = drgb.fuzzy_weights(idx, dist, 200)
    Y0 = drgb.init_embedding(9000, seed=3)

    def run():
        return (drgb.fit_transform(X, n_epochs=30), drgb.transform(X, Y0, X_new, n_epochs=30),
                drgb.embed_epochs(Y0.clone(), g, 1.577, 0.895, 1.0, 5, 0, 7, 200, 5))
    want = run()
    torch.cuda.synchronize()
    handle, sms = _limited_stream(16)
    assert sms < torch.cuda.get_device_properties(0).multi_processor_count
    stream = torch.cuda.ExternalStream(handle)
    with torch.cuda.stream(stream):
        got = run()
    torch.cuda.synchronize()
    for a, b in zip(got, want):
        assert torch.equal(a, b)
