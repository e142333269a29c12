"""The order of the training sums.  A gradient is the sum of the partial
gradients of tiles of 64 rows, added one by one in row order in FP32, whatever
grid forms them: one rounding more or less flips BF16 copies of the weights, and a
run of a hundred steps then ends elsewhere.

The first test restates that order: a tile's own gradient (a call with its 64
rows, one tile) scaled by a power of two is its partial in the gradient of all
rows, bit for bit, so the whole must equal the partials added in order.  The second
holds training runs to the parameters recorded from a kernel of one CTA a tile and
a sum over the CTAs in order, on the GB300."""
import hashlib

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


# (n, batch, epochs, lr): SHA-256 of the parameters after the run, and its loss
RECORDED = {
    (1, 1, 1, 1e-3): ('7b17a7f964e6499e', '0x1.9df7420000000p-1'),
    (65, 64, 3, 1e-3): ('11695ae37fde0bbf', '0x1.6398340000000p-7'),
    (300, 7, 2, 2e-3): ('22acfbfac5a03edc', '0x1.7fe92aaaaaaaap-3'),
    (5000, 1, 1, 1e-3): ('1744e580c6d9fc8b', '0x1.9468c00000000p-12'),
    (20000, 1024, 6, 2e-3): ('f15c68668ced34cd', '0x1.9be591f4b4b4bp-4'),
    (262144, 8192, 1, 2e-3): ('1f9e17f2eeee8bab', '0x1.0fb7031400000p-2'),
    (524288, 4096, 1, 2e-3): ('009018e623b44919', '0x1.83c13efd40000p-4'),
    (25000, 10000, 8, 2e-3): ('27ce4bf6773a2b7c', '0x1.43a1936666667p-2'),
    (700000, 10000, 1, 2e-3): ('13d35a82e7fd13a4', '0x1.00357667381d8p-2'),
    (100000, 30011, 10, 1e-3): ('3c7d8d017a319f05', '0x1.c344daed60e8ap-2'),
    (150001, 150001, 20, 1e-3): ('db3ad8f6eacd0577', '0x1.56b2297c4d3acp-1'),
}


def run(n, batch, epochs, lr):
    from paper_1904_08553_gb300 import dcd

    X, y = rows(n, n + batch)
    net = dcd.Mlp(seed=1)
    net.params = start_params(n - batch)
    loss = net.train(torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda(), n, batch=batch, epochs=epochs, lr=lr)
    return hashlib.sha256(np.ascontiguousarray(net.params, np.float32).tobytes()).hexdigest()[:16], float(loss).hex()


@pytest.mark.parametrize("case", list(RECORDED), ids=str)
def test_training_runs_end_where_they_did(case):
    assert run(*case) == RECORDED[case]
