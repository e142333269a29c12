"""The training kernel against its definition: mini-batches in row order, the
mean gradient of the batch (dcd_mlp_grad on the same rows), Adam.  Sizes around
one tile, a partial last batch, more tiles than CTAs, several epochs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

B1, B2, EPS = np.float32(0.9), np.float32(0.999), np.float32(1e-8)


def adam(P, m, v, g, t, lr):
    f = np.float32
    m[:] = B1 * m + (f(1) - B1) * g
    v[:] = B2 * v + (f(1) - B2) * g * g
    c1, c2 = f(1) - f(B1) ** f(t), f(1) - f(B2) ** f(t)
    P -= f(lr) * (m / c1) / (np.sqrt(v / c2) + EPS)


@pytest.mark.parametrize("n,batch,epochs", [(1, 1, 1), (63, 64, 1), (65, 64, 2), (1000, 1024, 3), (5000, 4096, 1),
                                            (25_000, 12_000, 1), (300, 7, 1)])
def test_train_is_adam_on_the_gradients(n, batch, epochs):
    import torch

    from paper_1904_08553_gb300 import dcd

    rng = np.random.default_rng(n + batch)
    X = rng.standard_normal((n, 12)).astype(np.float32)
    y = (X[:, 1] - X[:, 4] > 0.3).astype(np.float32)
    P = (rng.standard_normal(dcd.MLP_PARAMS) * 0.3).astype(np.float32)
    dX, dy = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda()
    lr = 1e-3
    net, ref = dcd.Mlp(seed=1), dcd.Mlp(seed=2)
    net.params = P
    loss = net.train(dX, dy, n, batch=batch, epochs=epochs, lr=lr)
    Q, m, v = P.copy(), np.zeros_like(P), np.zeros_like(P)
    t = 0
    for _ in range(epochs):
        for r in range(0, n, batch):
            k = min(batch, n - r)
            ref.params = Q
            g, last = ref.grad(dX[r:r + k].contiguous(), dy[r:r + k].contiguous(), k)
            t += 1
            adam(Q, m, v, g, t, lr)
    got = net.params
    step = np.linalg.norm(Q - P)
    # one step: the same gradient bits, FP32 arithmetic of a few roundings (2^-22
    # relative); later steps: an ulp of a parameter can flip its BF16 copy (2^-8),
    # and Adam divides a gradient by its own size
    bound = 4e-6 if t == 1 else 2e-2
    assert np.linalg.norm(got - Q) <= bound * step + 1e-7 * np.linalg.norm(P)
    assert abs(loss - last) <= 1e-4 * max(1.0, abs(last))
