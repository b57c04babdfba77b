"""Edges of the training products' tiles: fewer rows than the tensor-core path takes, whole and partial
128-row tiles and 64-row stages of the weight gradients, and the wide tiles of large batches."""
import numpy as np
import pytest

from inputs import random_mlp
from oracle import mlp

pytestmark = pytest.mark.gpu

BF16_UNIT = 2.0 ** -7  # of a value: 8 significant bits


def _per_tensor():
    for name, (o, k) in mlp.offsets().items():
        yield name, slice(o, o + k)


@pytest.fixture(scope="module")
def pkg():
    import paper_1611_06765_gb300 as P

    return P


@pytest.mark.parametrize("n", [1, 15, 16, 17, 64, 65, 128, 129, 1025, 8191, 8193])
def test_gradient_at_tile_edges(pkg, n):
    """Within one BF16 unit of each element's absolute-value scale (a rounding decision of an
    activation may differ), the loss within one such unit."""
    blob, X, T = random_mlp(n=n, seed=5, nparam=mlp.NPARAM)
    loss_g, g_g = pkg.mlp_loss_grad(blob, X, T)
    loss_r, g_r = mlp.loss_and_grad(blob, X, T, round_bf16=True)
    _, B_g = mlp.abs_bounds(blob, X, T, round_bf16=True)
    assert abs(loss_g - loss_r) <= BF16_UNIT * abs(loss_r)
    for name, sl in _per_tensor():
        assert np.all(np.abs(g_g[sl].astype(np.float64) - g_r[sl]) <= BF16_UNIT * B_g[sl]), name
    assert np.all(g_g[:mlp.HEADER] == 0)
