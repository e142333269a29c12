"""A training run that fails leaves the network as it was, optimiser state
included: every checked CUDA call of a run is made to fail in turn, and the wait
between the CTAs of its first and second launch is made to run out (with a short
limit, for CTAs that do not exist).  Afterwards the parameters are those of before,
and training goes on as in a network that never failed."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 5000  # steps of one row: more than one launch of the training kernel


@pytest.fixture
def nets():
    from paper_1904_08553_gb300 import dcd

    rng = np.random.default_rng(5)
    X = rng.standard_normal((N, 12)).astype(np.float32)
    y = (X[:, 0] > X[:, 3]).astype(np.float32)
    dX, dy = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda()
    out = []
    for _ in range(2):
        net = dcd.Mlp(seed=9)
        net.train(dX, dy, N, batch=700, epochs=1, lr=2e-3)  # moments and step count not zero
        out.append(net)
    dcd.dcd_set_fault(None)
    yield dcd, out[0], out[1], dX, dy
    dcd.dcd_set_fault(None)


def check_after(dcd, net, ref, dX, dy, before):
    dcd.dcd_set_fault(None)
    assert np.array_equal(net.params, before)
    for x, y in zip(net.grad(dX, dy, N), ref.grad(dX, dy, N)):  # the BF16 copies too
        assert np.array_equal(x, y)


def test_every_failure_of_a_run_is_undone(nets):
    dcd, net, ref, dX, dy = nets
    before = net.params
    failures = 0
    for k in range(1, 200):
        dcd.dcd_set_fault(f"cuda:{k}")
        try:
            net.train(dX, dy, N, batch=1, epochs=1, lr=2e-3)
        except dcd.DcdError as e:
            assert e.code == dcd.DCD_ECUDA
            failures += 1
            check_after(dcd, net, ref, dX, dy, before)
            continue
        break
    dcd.dcd_set_fault(None)
    assert failures >= 12  # two launches, six calls each
    ref.train(dX, dy, N, batch=1, epochs=1, lr=2e-3)
    assert np.array_equal(net.params, ref.params)


@pytest.mark.parametrize("launch", [1, 2])
def test_a_wait_that_runs_out_is_undone(nets, launch):
    dcd, net, ref, dX, dy = nets
    before = net.params
    dcd.dcd_set_fault(f"wait:{launch}")
    with pytest.raises(dcd.DcdError) as e:
        net.train(dX, dy, N, batch=1, epochs=1, lr=2e-3)
    assert e.value.code == dcd.DCD_ETIMEOUT
    check_after(dcd, net, ref, dX, dy, before)
    for x in (net, ref):
        x.train(dX, dy, N, batch=512, epochs=2, lr=2e-3)
    assert np.array_equal(net.params, ref.params)


def test_launches_share_one_run():
    """Steps beyond one launch go on where it stopped: the same rows as one call and as two."""
    from paper_1904_08553_gb300 import dcd

    rng = np.random.default_rng(6)
    X = rng.standard_normal((N, 12)).astype(np.float32)
    y = (X[:, 0] > X[:, 3]).astype(np.float32)
    dX, dy = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda()
    one, two = dcd.Mlp(seed=4), dcd.Mlp(seed=4)
    one.train(dX, dy, N, batch=1, epochs=1, lr=1e-3)
    for a, b in ((0, 2000), (2000, 4096), (4096, N)):
        two.train(dX[a:b].contiguous(), dy[a:b].contiguous(), b - a, batch=1, epochs=1, lr=1e-3)
    assert np.array_equal(one.params, two.params)


@pytest.mark.parametrize("n,batch,most", [(3000, 1000, 79), (30_000, 10_000, 100), (30_000, 10_000, 1), (64, 64, 3)])
def test_a_grid_too_large_for_the_device_is_made_smaller(n, batch, most):
    """On a part of the GPU fewer CTAs run at once: the launch is refused, and half as many, down to
    one, end in the same parameters."""
    from paper_1904_08553_gb300 import dcd

    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, 12)).astype(np.float32)
    y = (X[:, 2] > X[:, 5]).astype(np.float32)
    dX, dy = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda()
    net, ref = dcd.Mlp(seed=4), dcd.Mlp(seed=4)
    ref.train(dX, dy, n, batch=batch, epochs=2, lr=1e-3)
    try:
        dcd.dcd_set_fault(f"grid:{most}")
        assert net.train(dX, dy, n, batch=batch, epochs=2, lr=1e-3) > 0
    finally:
        dcd.dcd_set_fault(None)
    assert np.array_equal(net.params, ref.params)
