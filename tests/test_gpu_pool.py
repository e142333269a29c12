"""The learned screen's pool and features, against the oracle, on both sides of
the choice between marking from the vertices with pairs and looking for one from
the others: batches that touch few vertices, about half of the entries, all of
them; repeated records, hubs with hundreds of pairs, vertices without edges."""
import numpy as np
import pytest

from test_gpu_parity import dcd  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("share", [0.01, 0.3, 0.5, 1.0])
@pytest.mark.parametrize("n", [33, 1500])
def test_pool_and_features(dcd, orc, n, share):  # noqa: F811
    rng = np.random.default_rng(n + int(100 * share))
    live = n - n // 8  # the rest has no edges
    m = 6 * live
    e = np.stack([rng.integers(0, live, m), np.minimum(rng.integers(0, live, m), rng.integers(0, live, m))], 1)
    e = e[e[:, 0] != e[:, 1]]
    first = np.concatenate([e, rng.integers(1, 5, (len(e), 1))], 1).astype(np.int32)
    touched = max(2, int(share * live))
    k = 4 * touched
    u, v = rng.integers(0, touched, k), rng.integers(0, touched, k)
    u[: k // 4] = 0  # a hub's pairs
    ins = np.stack([u, v, rng.integers(1, 4, k)], 1)[u != v].astype(np.int32)
    ins = np.concatenate([ins, ins[: len(ins) // 3]])
    dels = np.concatenate([first[(first[:, :2] < touched).all(1)][::3, :2], [[0, live - 1]]]).astype(np.int32)
    none = np.zeros((0, 2), np.int32)
    with dcd.Context(n, mode=dcd.MODE_BASE) as ctx:
        ctx.set_collect(True)
        ctx.apply_batch(first, none)
        lab, _, _ = ctx.update()
        ctx.apply_batch(ins, dels)
        _, _, st = ctx.update()
        X, y, v = ctx.screen_data()
    g0, err0 = orc.Graph.empty(n).apply(first, none)
    g1, err1 = g0.apply(ins, dels)
    assert err0 == 0 and err1 == 0
    rds = orc.screen(g0, g1, lab, ins, dels)
    pool, Xr = orc.screen_features(g0, g1, lab, ins, dels, rds)
    assert sorted(v.tolist()) == np.nonzero(pool)[0].tolist() and st.pool == len(v)
    # the features are single-precision functions of whole numbers: two roundings
    # and a log1p of at most two units in the last place
    np.testing.assert_allclose(X, Xr[v], rtol=2e-6, atol=1e-7)
