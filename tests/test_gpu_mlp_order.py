"""The order of the training sums.  A gradient is the sum of the partial
gradients of tiles of 64 rows, added one by one in row order in FP32, whatever
grid forms them: one rounding more or less flips BF16 copies of the weights, and a
run of a hundred steps then ends elsewhere.

The test restates that order: a tile's own gradient (a call with its 64 rows, one
tile) scaled by a power of two is its partial in the gradient of all rows, bit for
bit, so the whole must equal the partials added in order."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TILE = 64


def rows(n, seed):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((n, 12)).astype(np.float32)
    y = (X[:, 1] - X[:, 4] + 0.5 * X[:, 7] * X[:, 0] > 0.3).astype(np.float32)
    return X, y


def start_params(seed):
    from paper_1904_08553_gb300 import dcd

    return (np.random.default_rng(seed).standard_normal(dcd.MLP_PARAMS) * 0.3).astype(np.float32)


# tiles: one wave of CTAs, one more than the GPU has SMs, several a CTA, more than there is room for at once
@pytest.mark.parametrize("tiles", [1, 2, 128, 256, 1024, 2048])
def test_gradient_adds_the_tiles_in_order(tiles):
    from paper_1904_08553_gb300 import dcd

    n = TILE * tiles  # a power of two times 64: scaling by 1 / tiles is exact
    X, y = rows(n, tiles)
    dX, dy = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda()
    net = dcd.Mlp(seed=3)
    net.params = start_params(tiles)
    whole, loss = net.grad(dX, dy, n)
    expect, eloss = np.zeros(dcd.MLP_PARAMS, np.float32), 0.0
    for t in range(tiles):
        g, l = net.grad(dX[t * TILE:(t + 1) * TILE], dy[t * TILE:(t + 1) * TILE], TILE)
        expect += g * np.float32(1.0 / tiles)
        eloss += l * TILE
    assert np.array_equal(whole, expect)
    assert loss == eloss * (1.0 / n)
