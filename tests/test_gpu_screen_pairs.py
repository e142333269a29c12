"""Sources with many pairs and short rows: vertices that lose most of their edges,
and edges that a batch repeats.  The screening walks over a source's pairs, with as
many threads as its row or its pairs want; equal to the oracle at the lengths where
the kernel changes, and not much slower than as many pairs spread evenly."""
import numpy as np
import pytest

from test_gpu_parity import assert_step_equal, dcd  # noqa: F401

pytestmark = pytest.mark.gpu
NONE = np.zeros((0, 2), np.int32)


@pytest.mark.parametrize("pairs", [16, 17, 32, 33, 64, 65, 129, 257, 513, 1025, 2049, 4096, 4097, 6000])
@pytest.mark.parametrize("left", [0, 1, 20, 40])
def test_lost_edges(dcd, orc, pairs, left):  # noqa: F811
    """Vertex 0 loses `pairs` edges and keeps `left`; the next batch repeats one of its edges `pairs` times."""
    n = 7000
    rng = np.random.default_rng(pairs + left)
    star = np.stack([np.zeros(pairs + left, int), 1 + np.arange(pairs + left), rng.integers(1, 4, pairs + left)], 1)
    u = rng.integers(1, n, 12_000)
    near = np.minimum(u // 40 * 40 + rng.integers(0, 40, 12_000), n - 1)
    rest = np.stack([u, near, np.ones(12_000, int)], 1)[u != near]
    rest = rest[rest[:, 1] > 0]
    first = np.concatenate([star, rest]).astype(np.int32)
    again = np.concatenate([np.tile([[0, 1 + pairs + max(left - 1, 0), 1]], (pairs, 1)), [[5, 6, 1]]]).astype(np.int32)
    with dcd.Context(n, mode=dcd.MODE_DELTA) as c:
        ref = orc.Context(n)
        for ins, dels in ((first, NONE), (rest[:50].astype(np.int32), star[:pairs, :2].astype(np.int32)),
                          (again, star[pairs:pairs + 1, :2].astype(np.int32)), (again[:9], NONE)):
            for x in (c, ref):
                x.apply_batch(ins, np.ascontiguousarray(dels))
            lab, q, st = c.update()
            rlab, rq, rst = ref.update(orc.DELTA)
            assert_step_equal(st, rst, lab, rlab, q, rq, c.rset(), ref.rset())


def test_time_of_lost_edges(dcd):  # noqa: F811
    """60,000 deletes on one vertex against 60,000 spread ones: the screening's time, within a factor of 10
    (one thread's walk takes 100 times as long)."""
    n, k = 300_000, 60_000
    rng = np.random.default_rng(1)
    ring = np.stack([np.arange(n), (np.arange(n) + 1) % n, np.ones(n, int)], 1)
    star = np.stack([np.zeros(k, int), 2 + 2 * np.arange(k), np.ones(k, int)], 1)
    pairs = np.stack([n // 2 + np.arange(k), 2 + 2 * np.arange(k), np.ones(k, int)], 1)
    ms = {}
    for name, e in (("hub", star), ("spread", pairs)):
        best = []
        for _ in range(4):
            with dcd.Context(n, mode=dcd.MODE_DELTA) as c:
                c.apply_batch(np.concatenate([ring, e]).astype(np.int32), NONE)
                c.update(labels_out=None)
                c.apply_batch(ring[:10].astype(np.int32), np.ascontiguousarray(e[:, :2].astype(np.int32)))
                best.append(c.update(labels_out=None)[2].ms_screen)
        ms[name] = min(best)
    assert ms["hub"] < 10 * ms["spread"], ms
