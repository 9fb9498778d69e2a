"""PCA at feature counts around the splits and row ranges of the product C X:
128 rows of X a split, up to the largest count of 1,024 (above it the call is
refused), 8 rows of C a block (gpu)."""
import numpy as np
import pytest

from gpu_util import drgb_module
from test_gpu_pca import _check, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [65, 127, 128, 129, 135, 1023, 1024, 1025, 1160])
def test_sizes_around_the_splits(D):
    g = np.random.default_rng(D)
    n, dim = 1500, 10
    sd = np.concatenate([8 * 0.8 ** np.arange(30), np.zeros(D - 30)]) + 0.02
    Q, _ = np.linalg.qr(g.normal(size=(D, D)))
    X = ((g.normal(size=(n, D)) * sd) @ Q.T + g.normal(size=D)).astype(np.float32)
    drgb = drgb_module()
    if D > 1024:
        with pytest.raises(drgb.DrgbError):
            _run(drgb, X, dim)
        return
    _check(X, dim, *_run(drgb, X, dim), min_unique=dim - 2)
