"""The bound that the tensor-core k-NN's certificate puts on the rounding of its
products (gpu): the accumulators of the kernels' operands [x, C, C, C] and
[-2 y, n / C in three parts] against sums in 64 bits (exact products, at most
1,024 of them), over the widths the kernels take and operands chosen to round
badly.  The certificate assumes at most 34 units of 2^-23 (|x|^2 + |y|^2) for
each step of 16 columns."""
import ctypes as C

import pytest

from gpu_util import drgb_module

pytestmark = pytest.mark.gpu

ROWS = 1024


def _rows(d, top, seed):
    """ROWS x d values of magnitude up to `top`, several kinds of rows."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = lambda *s: torch.rand(*s, generator=g, device="cuda", dtype=torch.float64)
    kinds = []
    m = ROWS // 8
    kinds.append(top * (2 * r(m, d) - 1))                                    # even
    kinds.append(top / 4 * torch.randn(m, d, generator=g, device="cuda").double().clamp(-4, 4))
    kinds.append(top * torch.sign(r(m, d) - 0.5) * 2.0 ** (-20 * r(m, d)))   # magnitudes over 20 binary orders
    kinds.append(top * (1 - 2.0 ** -11 * (1 + r(m, d))))                     # one sign, full significands
    kinds.append(-kinds[-1].clone())                                         # against it: every term of one sign
    k = top * 2.0 ** -10 * (1 + r(m, d))                                     # large terms first, then many small ones
    k[:, : max(1, d // 16)] = top
    kinds.append(k)
    kinds.append(k.flip(1).clone())                                          # and last
    base = top / 2 * torch.randn(1, d, generator=g, device="cuda").double().clamp(-2, 2)
    kinds.append(base * (1 + 2.0 ** -9 * (r(m, d) - 0.5)))                   # near-copies: the sum cancels
    return torch.cat(kinds)


@pytest.mark.parametrize("f16,d", [(1, 16), (1, 50), (1, 61), (1, 62), (1, 200), (1, 509), (1, 784), (1, 1021), (0, 16), (0, 61)])
def test_sums_stay_within_the_certificates_bound(f16, d):
    import torch
    drgb = drgb_module()
    lib, ctx = drgb._lib.load(), drgb.context()
    op = torch.float16 if f16 else torch.bfloat16
    top, scale = (1024.0, 32768.0) if f16 else (100.0, 1.0)
    K = (d + 3 + 63) // 64 * 64
    worst = 0.0
    for seed in range(4):
        x = _rows(d, top, 7 * d + seed).to(op)
        y = x if seed % 2 else _rows(d, top, 7 * d + 100 + seed).to(op)
        A, B = (torch.zeros(ROWS, K, dtype=op, device="cuda") for _ in range(2))
        A[:, :d], A[:, d:d + 3] = x, scale
        B[:, :d] = -2.0 * y
        n = (y.float() ** 2).sum(1) / scale
        for part in range(3):
            B[:, d + part] = n.to(op)
            n = n - B[:, d + part].float()
        out = torch.empty(ROWS, ROWS, device="cuda")
        ptr = lambda t: C.c_void_p(t.data_ptr())
        stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
        assert lib.drgb_product_selftest(ctx, ptr(A), ptr(B), ROWS, ROWS, K, f16, ptr(out), stream) == 0
        assert lib.drgb_sync(ctx, stream) == 0
        want = A.double() @ B.double().T
        norms = (x.double() ** 2).sum(1)[:, None] + (y.double() ** 2).sum(1)[None, :]
        bound = K / 16 * 34 * 2.0 ** -23 * norms
        worst = max(worst, float(((out.double() - want).abs() / bound).max()))
    print(f"f16 {f16} d {d}: {worst:.3f} of the bound")
    assert worst <= 1.0


def test_sizes_are_checked():
    import torch
    drgb = drgb_module()
    lib, ctx = drgb._lib.load(), drgb.context()
    t = torch.zeros(256 * 64 + 1, dtype=torch.float16, device="cuda")
    o = torch.zeros(128 * 128, device="cuda")
    p, q = C.c_void_p(t.data_ptr()), C.c_void_p(o.data_ptr())
    E = drgb._lib.ERR_INVALID
    assert lib.drgb_product_selftest(ctx, p, p, 128, 128, 65, 1, q, None) == E
    assert lib.drgb_product_selftest(ctx, p, p, 100, 128, 64, 1, q, None) == E
    assert lib.drgb_product_selftest(ctx, p, p, 128, 64, 64, 1, q, None) == E
    assert lib.drgb_product_selftest(ctx, C.c_void_p(t.data_ptr() + 2), p, 128, 128, 64, 1, q, None) == E
    assert lib.drgb_product_selftest(None, p, p, 128, 128, 64, 1, q, None) == E
