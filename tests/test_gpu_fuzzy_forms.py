"""The two forms of the fuzzy rows' bisection agree bit for bit (gpu): rows whose
quotients stay among the normal numbers divide by a correctly rounded reciprocal
and decide most steps by hardware exponentials; a row with a smaller excess takes
plain divides and exponentials.  An excess of 1e-30 instead of 0 sends a row to
the plain form and changes no exponential (exp(-1e-30 / sigma) is 1)."""
import numpy as np
import pytest

from gpu_util import drgb_module

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [2, 3, 5, 8, 9, 15, 16, 17, 31, 32])
@pytest.mark.parametrize("spread", [0.05, 1.0, 10.0])
def test_forms_of_the_bisection_agree(k, spread):
    import torch
    drgb = drgb_module()
    rng = np.random.default_rng(1000 * k + int(spread))
    n = 30000
    idx = ((np.arange(n)[:, None] + np.arange(1, k + 1)) % n).astype(np.int32)
    # excesses over `spread` decades about a scale between 1e-9 and 1e15
    scale = 10.0 ** rng.uniform(-9, 15, (n, 1))
    d = np.sort(scale * 10.0 ** (spread * rng.uniform(-0.5, 0.5, (n, k))), axis=1)
    d = np.clip(d, 1e-15, 1e17).astype(np.float32)
    d[::5, k // 2:] = d[::5, k // 2:k // 2 + 1]  # ties
    d[:, 0] = 0.0
    out = []
    for tiny in (0.0, 1e-30):
        d[:, 1] = tiny
        g = drgb.fuzzy_weights(torch.from_numpy(idx).cuda(), torch.from_numpy(d).cuda(), 200, with_rho_sigma=True)
        torch.cuda.synchronize()
        out.append(g)
    a, b = out
    assert torch.equal(a.sigma, b.sigma)
    assert torch.equal(a.row_ptr, b.row_ptr) and torch.equal(a.col, b.col) and torch.equal(a.w, b.w) and torch.equal(a.q, b.q)
