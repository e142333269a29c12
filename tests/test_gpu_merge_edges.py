"""The CSR merge at the edges of its classes: segments of records around the
lengths at which a batch record's sorting changes, repeated pairs, and merged
sequences around whole tiles.  Compared with a dictionary model of the merge
(deletes remove whole edges, then inserts add weight)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def model_step(edges, ins, dels):
    for u, v in dels:
        edges.pop((min(u, v), max(u, v)), None)
    for u, v, w in ins:
        k = (min(u, v), max(u, v))
        edges[k] = edges.get(k, 0) + int(w)


def model_csr(edges, n):
    a = np.array([(u, v, w) for (u, v), w in edges.items()] + [(v, u, w) for (u, v), w in edges.items()],
                 np.int64).reshape(-1, 3)
    a = a[np.lexsort((a[:, 1], a[:, 0]))]
    rp = np.zeros(n + 1, np.int64)
    rp[1:] = np.cumsum(np.bincount(a[:, 0], minlength=n))
    return rp, a[:, 1], a[:, 2]


def check(ctx, edges, n):
    rp, col, w = ctx.graph()
    mrp, mcol, mw = model_csr(edges, n)
    assert np.array_equal(rp, mrp)
    assert np.array_equal(col, mcol)
    assert np.array_equal(w, mw)


@pytest.mark.parametrize("length", [1, 63, 64, 65, 511, 512, 513, 4095, 4096, 4097, 9001])
def test_segment_lengths(length):
    from paper_1904_08553_gb300 import dcd

    n = 12_000
    rng = np.random.default_rng(length)
    edges = {}
    with dcd.Context(n, mode=dcd.MODE_BASE) as ctx:
        for t in range(3):
            # the hub's segment holds `length` records, a fifth of them repeats
            sinks = 1 + rng.integers(0, max(1, (4 * length) // 5), length)
            ins = np.stack([np.zeros(length, np.int64), sinks, rng.integers(1, 9, length)], 1)
            flip = rng.random(length) < 0.5
            ins[flip, :2] = ins[flip, 1::-1]
            dels = np.zeros((0, 2), np.int64)
            if t and len(edges):
                present = np.array(list(edges))[rng.integers(0, len(edges), max(1, length // 4))]
                absent = np.stack([np.zeros(5, np.int64), n - 1 - np.arange(5)], 1)
                dels = np.concatenate([present, absent, present[:1]])
            if t == 2:  # deletes alone, the whole row among them
                ins, dels = ins[:0], np.array(list(edges))
            ctx.apply_batch(ins.astype(np.int32), dels.astype(np.int32))
            ctx.update(labels_out=None)
            model_step(edges, ins, dels)
            check(ctx, edges, n)
            st_m2 = ctx.update(labels_out=None)[2].m2  # an empty step keeps 2m and the degrees
            assert st_m2 == 2 * sum(edges.values())


@pytest.mark.parametrize("entries", [2046, 2048, 2050, 4096])
@pytest.mark.parametrize("pairs", [2, 4, 2048])
def test_tile_boundaries(entries, pairs):
    from paper_1904_08553_gb300 import dcd

    n = 3000
    rng = np.random.default_rng(entries * 7 + pairs)
    m = entries // 2
    first = np.stack([np.arange(m), np.arange(m) + 1, np.ones(m, np.int64)], 1)  # a path: row u is u-1, u+1
    edges = {}
    with dcd.Context(n, mode=dcd.MODE_DELTA) as ctx:
        ctx.apply_batch(first.astype(np.int32))
        ctx.update(labels_out=None)
        model_step(edges, first, [])
        check(ctx, edges, n)
        for at in (0, 1022, 1023, 1024, m - 1):  # changes next to a tile's first and last entry
            k = pairs // 2
            keys = list(edges)
            dels = np.array([keys[(at + i) % len(keys)] for i in range(0, k, 2)])
            u = (at + rng.integers(0, 3, k)) % (n - 2000)
            ins = np.stack([u, u + 1 + rng.integers(0, 1500, k), rng.integers(1, 5, k)], 1)
            ctx.apply_batch(ins.astype(np.int32), dels.astype(np.int32))
            ctx.update(labels_out=None)
            model_step(edges, ins, dels)
            check(ctx, edges, n)


def test_bad_device_record_leaves_the_graph():
    from paper_1904_08553_gb300 import dcd

    n = 200
    rng = np.random.default_rng(1)
    u = rng.integers(0, n - 1, 5000)
    ins = np.stack([u, u + 1 + rng.integers(0, n, 5000) % (n - 1 - u), np.ones(5000, np.int64)], 1).astype(np.int32)
    with dcd.Context(n, mode=dcd.MODE_DELTA) as ctx:
        ctx.apply_batch(ins)
        ctx.update(labels_out=None)
        before = ctx.graph()
        bad = ins.copy()
        bad[::7, 1] = n + 3      # out of range
        bad[3::7, 1] = bad[3::7, 0]  # self-loop
        bad[5::7, 2] = 0         # no weight
        d = torch.from_numpy(bad).cuda()
        ctx.apply_batch_device(d, len(d), None, 0)
        with pytest.raises(dcd.DcdError) as e:
            ctx.update(labels_out=None)
        assert e.value.code == dcd.DCD_EINVAL
        for x, y in zip(before, ctx.graph()):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("records", [400, 60_000, 200_000])
def test_sources_per_tile(records):
    """A large graph with batches of few, about one, and several records a
    source: tiles of 128, 64 and 32 sources, some of them with more records than a
    tile stages (runs of sources with 60 each) or with rows too long to stage."""
    from paper_1904_08553_gb300 import dcd

    n = 90_000
    rng = np.random.default_rng(records)
    edges = {}
    with dcd.Context(n, mode=dcd.MODE_BASE) as ctx:
        for t in range(3):
            u, v = rng.integers(0, n, records), rng.integers(0, n, records)
            if t == 0:  # long rows
                u[: records // 4] = rng.integers(0, 3, records // 4) * 40
            if t == 1:  # crowded tiles
                m = min(records // 2, 130 * 58)
                u[:m] = 5000 + np.arange(m) // 58
                v[:m] = rng.integers(0, 4, m) + 60_000 + 9 * (np.arange(m) // 58)
            ok = u != v
            ins = np.stack([u, v, rng.integers(1, 9, records)], 1)[ok]
            dels = np.zeros((0, 2), np.int64)
            if t:
                dels = np.array(list(edges))[rng.integers(0, len(edges), records // 3)]
            ctx.apply_batch(ins.astype(np.int32), dels.astype(np.int32))
            ctx.update(labels_out=None)
            model_step(edges, ins, dels)
            check(ctx, edges, n)
