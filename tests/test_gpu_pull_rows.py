"""Marking by pull over rows of every length: rows whose only marked neighbour is
first, last, at the edges of what a warp reads and of the chunks of the rest, and
long rows without one.  R_t and the learned screen's pool against the oracle."""
import numpy as np
import pytest

from test_gpu_parity import dcd  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("length", [1, 32, 63, 64, 65, 127, 2111, 2112, 2113, 4160, 4161, 9000])
def test_where_the_neighbour_lies(dcd, orc, length):  # noqa: F811
    """Vertices 0..5 see `length` quiet vertices, and some of them one source among these, at a chosen place."""
    k = 6
    quiet = np.arange(k, k + 10_000)       # no batch touches them
    busy = np.arange(20_000, 30_000)       # the batch does: they hold most entries
    places = [0, length // 2, length - 1, min(63, length - 1), min(64, length - 1), None]
    src = 15_000 + np.arange(k)            # a source for vertex i: its id decides its place in the row
    n = 40_000
    rng = np.random.default_rng(length)
    e = []
    for i, at in enumerate(places):
        if at is None:
            sinks = quiet[:length]
        else:                              # `at` sinks below the source, the others above all quiet ones
            sinks = np.concatenate([quiet[:at], [src[i]], 30_000 + np.arange(length - at - 1)])
        e.append(np.stack([np.full(len(sinks), i), sinks], 1))
    a = rng.choice(busy, 120_000)
    b = rng.choice(busy, 120_000)
    e = np.concatenate(e + [np.stack([a, b], 1)[a != b]])
    first = np.concatenate([e, np.ones((len(e), 1), int)], 1).astype(np.int32)
    x, y = rng.choice(busy, 40_000), rng.choice(busy, 40_000)
    touch = np.concatenate([np.stack([x, y], 1)[x != y], np.stack([src, 31_000 + np.zeros(k, int) + 8999 + 0 * src], 1)])
    touch = np.concatenate([touch, np.ones((len(touch), 1), int)], 1).astype(np.int32)
    none = np.zeros((0, 2), np.int32)
    with dcd.Context(n, mode=dcd.MODE_DELTA) as c:
        c.set_collect(True)
        c.apply_batch(first, none)
        lab, _, _ = c.update()
        c.apply_batch(touch, none)
        _, _, st = c.update()
        _, _, v = c.screen_data()
        rset = c.rset()
    g0, err0 = orc.Graph.empty(n).apply(first, none)
    g1, err1 = g0.apply(touch, none)
    assert err0 == 0 and err1 == 0
    rds = orc.screen(g0, g1, lab, touch, none)
    pool, _ = orc.screen_features(g0, g1, lab, touch, none, rds)
    assert np.array_equal(rset, rds) and st.r_size == rds.sum()
    assert sorted(v.tolist()) == np.nonzero(pool)[0].tolist()
    want = [p is not None for p in places]
    assert [bool(pool[i]) or not w for i, w in enumerate(want)] == [True] * k  # the sources reach their vertices
