"""New points without neighbours (NaN, overflowing distances) in transform() (gpu)."""
import pytest

from gpu_util import drgb_module

pytestmark = pytest.mark.gpu


def test_new_points_without_neighbours_are_reported():
    # NaN and overflowing rows have no neighbours: the call reports them (the rows'
    # start has no coordinates to be averaged from) and the context goes on
    import torch
    drgb = drgb_module()
    g = torch.Generator(device="cuda").manual_seed(1)
    X, Q = (torch.randn((n, 50), generator=g, device="cuda") for n in (3000, 500))
    Y = torch.randn(3000, 2, device="cuda")
    want = drgb.transform(X, Y, Q, n_epochs=9)
    for bad in (float("nan"), 1e30):
        Qb = Q.clone()
        Qb[17] = bad
        Qb[499, 3] = bad
        with pytest.raises(drgb.DrgbError):
            drgb.transform(X, Y, Qb, n_epochs=9)
        assert torch.equal(drgb.transform(X, Y, Q, n_epochs=9), want)
