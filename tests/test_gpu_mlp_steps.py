"""Training steps whose batches are prepared one step ahead (gpu)."""
import numpy as np
import pytest

import datagen
from gpu_util import drgb_module
from oracle import fuzzy as ofuzzy, knn as oknn

pytestmark = pytest.mark.gpu


# one edge; fewer rows than a tile; rows just below, at and above tiles of 128; several chunks of 512
@pytest.mark.parametrize("batch,neg,steps", [(1, 0, 2), (1, 8, 3), (63, 0, 3), (64, 0, 3), (65, 0, 3), (37, 2, 5), (700, 5, 3)])
def test_each_step_trains_on_its_own_batch(batch, neg, steps):
    """With a learning rate of 0 every step's loss is the loss that mlp_grad gives for that step's sample."""
    import torch
    drgb = drgb_module()
    X, _ = datagen.mixture(600, 20, 5, seed=3)
    oi, od = oknn.knn(X, 10)
    g = ofuzzy.build_csr(oi, od, 200, 10)
    gd = drgb.Graph(torch.from_numpy(g["row_ptr"].astype(np.int32)).cuda(), torch.from_numpy(g["col"].astype(np.int32)).cuda(),
                    torch.from_numpy(g["w"].astype(np.float32)).cuda(), torch.from_numpy(g["q"].astype(np.int32)).cuda())
    Xd = torch.from_numpy(X).cuda()
    P = drgb.mlp_init(20, seed=4)
    P0 = P.clone()
    m, v = torch.zeros_like(P), torch.zeros_like(P)
    losses = drgb.mlp_train(Xd, gd, 1.577, 0.895, P, m, v, steps=steps, batch_edges=batch, neg=neg, lr=0.0, seed=6)
    assert torch.equal(P, P0)
    mo = np.zeros(P.numel(), np.float64)
    for t in range(steps):
        rows = drgb.mlp_sample(gd, batch, neg, t, 6)
        grad, loss = drgb.mlp_grad(P0, Xd, rows, batch, neg, 1.577, 0.895)
        assert float(losses[t]) == float(loss)
        mo = 0.9 * mo + 0.1 * grad.cpu().numpy().astype(np.float64)
    # first moments: FP32 1 - 0.9 is off by 4 x 2^-24, products and sums by less; a sum is at least a tenth of its largest term
    scale = np.abs(mo).max() + 1e-30
    assert np.abs(m.cpu().numpy() - mo).max() <= steps * 4 * 2.0 ** -24 * scale * 10
