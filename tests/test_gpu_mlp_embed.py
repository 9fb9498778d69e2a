"""The fused forward pass at its edges: one row, whole and ragged tiles, more
tiles than CTAs, input widths from 1 to the operand's 64 columns, against the
oracle; a row's result does not depend on its place."""
import numpy as np
import pytest

from gpu_util import drgb_module
from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d", [(1, 50), (127, 1), (128, 64), (129, 63), (152 * 128 + 1, 7), (2 * 152 * 128 + 77, 33)])
def test_embed_matches_oracle_and_itself(n, d):
    import torch
    drgb = drgb_module()
    rng = np.random.default_rng(n + d)
    X = rng.normal(size=(n, d)).astype(np.float32)
    P = drgb.mlp_init(d, seed=3)
    P += 0.02 * torch.randn(P.shape, generator=torch.Generator(device="cuda").manual_seed(5), device="cuda")
    P[:256 * 64].view(256, 64)[:, d:] = 0  # columns beyond d stay 0, as in training
    Xd = torch.from_numpy(X).cuda()
    Y = drgb.mlp_embed(P, Xd)
    rows = np.unique(np.concatenate([np.arange(0, n, max(1, n // 200)), np.arange(max(0, n - 100), n)]))
    want = omlp.embed(P.cpu().numpy().astype(np.float64), X[rows], d)
    # the tolerance of the forward pass: FP32 sums may flip BF16 roundings
    assert np.abs(Y.cpu().numpy()[rows] - want).max() <= 1e-2 * (np.abs(want).max() + 1.0)
    for i in (0, n // 2, n - 1):
        assert torch.equal(drgb.mlp_embed(P, Xd[i:i + 1].contiguous())[0], Y[i])
