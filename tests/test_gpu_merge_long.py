"""Batches that put many records on one source: segments longer than a CTA
sorts are sorted over the whole device.  Their pairs must be those
of the same batch with its repeats added up beforehand (which has short segments),
in every mode, and the merged rows those of a dictionary model."""
import numpy as np
import pytest

from test_gpu_merge_edges import check, model_step
from test_gpu_parity import dcd  # noqa: F401

pytestmark = pytest.mark.gpu
NONE = np.zeros((0, 2), np.int32)
SAME = ["nnz", "m2", "r_size", "levels", "iters_total", "moves_total", "communities", "n_lo", "n_hi", "coarse0_delta",
        "coarse0_entries", "pool", "edges_level0_screen"]


def base_graph(n, seed):
    rng = np.random.default_rng(seed)
    m = 6 * n
    u = rng.integers(0, n, m)
    v = np.where(rng.random(m) < 0.8, u // 50 * 50 + rng.integers(0, 50, m), rng.integers(0, n, m)) % n
    return np.stack([u, v, rng.integers(1, 4, m)], 1)[u != v].astype(np.int32)


def added_up(ins):
    """One record an edge, the weights of its repeats added."""
    a = np.stack([ins[:, :2].min(1), ins[:, :2].max(1)], 1)
    e, at = np.unique(a, axis=0, return_inverse=True)
    return np.concatenate([e, np.bincount(at.ravel(), ins[:, 2])[:, None]], 1).astype(np.int32)


def hub_batch(n, seed, hubs, length):
    """`length` records on each hub, few distinct sinks; some of everything else."""
    rng = np.random.default_rng(seed)
    k = hubs * length
    u = np.repeat(np.arange(hubs) * 7, length)
    v = rng.integers(n // 2, n // 2 + 1000, k)
    flip = rng.random(k) < 0.5
    e = np.stack([np.where(flip, v, u), np.where(flip, u, v), rng.integers(1, 4, k)], 1)
    return rng.permutation(np.concatenate([e, base_graph(n, seed + 1)[:300]])).astype(np.int32)


@pytest.mark.parametrize("hubs,length", [(1, 4097), (2, 32_768), (3, 32_769), (1, 50_000)])
@pytest.mark.parametrize("how", ["STATIC", "BASE", "DELTA", "slm", "collect", "labels"])
def test_same_as_added_up(dcd, how, hubs, length):  # noqa: F811
    n = 6000
    kw = dict(mode=getattr(dcd, "MODE_" + how, dcd.MODE_DELTA))
    if how == "slm":
        kw["alg"] = dcd.ALG_SLM
    one, two = dcd.Context(n, **kw), dcd.Context(n, **kw)
    for t in range(3):
        ins = base_graph(n, 5) if t == 0 else hub_batch(n, t, hubs, length)
        dels = NONE if t == 0 else added_up(base_graph(n, 5))[t::9, :2]
        out = []
        for c, batch in ((one, ins), (two, ins if t == 0 else added_up(ins))):
            if how == "labels" and t:
                c.set_labels((np.arange(n) // (10 * t) * (10 * t)).astype(np.int32))
            if how == "collect":
                c.set_collect(True)
            c.apply_batch(batch, np.ascontiguousarray(dels))
            lab, q, st = c.update()
            out.append((lab, q, {k: getattr(st, k) for k in SAME}, c.rset(), *c.graph()))
        for x, y in zip(*out):
            assert np.array_equal(x, y) if isinstance(x, np.ndarray) else x == y
        if t:
            assert np.bincount(ins[:, :2].ravel()).max() > 4096
    one.close()
    two.close()


@pytest.mark.parametrize("length", [8200, 65_536, 140_001])
def test_rows_of_long_segments(dcd, length):  # noqa: F811
    n = 50_000
    rng = np.random.default_rng(length)
    edges = {}
    with dcd.Context(n, mode=dcd.MODE_BASE) as c:
        for t in range(3):
            hub = rng.integers(0, 2, length)  # two long segments, few repeats
            ins = np.stack([hub, 2 + rng.integers(0, n - 2, length), rng.integers(1, 9, length)], 1)
            rep = np.tile([[3, n - 1, 2]], (length // 2, 1))  # and one edge many times
            ins = rng.permutation(np.concatenate([ins, rep]))
            dels = np.zeros((0, 2), np.int64)
            if t:
                dels = np.array(list(edges))[:: 1 + t]
            if t == 2:  # deletes alone on the hubs
                ins = ins[:10]
            c.apply_batch(ins.astype(np.int32), dels.astype(np.int32))
            st = c.update(labels_out=None)[2]
            model_step(edges, ins, dels)
            check(c, edges, n)
            assert st.m2 == 2 * sum(edges.values())


def test_group_and_errors(dcd):  # noqa: F811
    n = 6000
    grp = dcd.Group([n, 500, n], mode=dcd.MODE_DELTA)
    ctx = [dcd.Context(n, mode=dcd.MODE_DELTA) for _ in range(2)]
    for t in range(3):
        for g in (0, 2):
            ins = base_graph(n, g) if t == 0 else hub_batch(n, t + g, 1 + g, 33_000)
            grp.apply_batch(g, ins, NONE)
            ctx[g // 2].apply_batch(added_up(ins), NONE)
        lab, q, st = grp.update()
        for g in (0, 2):
            rl, rq, rst = ctx[g // 2].update()
            assert np.array_equal(lab[grp.offsets[g]:grp.offsets[g + 1]], rl) and q[g] == rq
            assert (st[g].m2, st[g].nnz, st[g].r_size) == (rst.m2, rst.nnz, rst.r_size)
    grp.close()
    c = ctx[0]
    before = c.graph()
    ins = np.tile(np.array([[1, 2, 1 << 30]], np.int32), (40_000, 1))  # a weight above INT32_MAX
    c.apply_batch(ins, NONE)
    with pytest.raises(dcd.DcdError) as e:
        c.update()
    assert e.value.code == dcd.DCD_EOVERFLOW
    for x, y in zip(before, c.graph()):
        assert np.array_equal(x, y)
    for x in ctx:
        x.close()


@pytest.mark.parametrize("run", [31, 32, 33, 64, 65, 500, 4000, 30_000])
def test_runs_of_one_pair(dcd, run):  # noqa: F811
    """An edge repeated around the lengths its records are added up in another way, in segments of every class."""
    n = 40_000
    rng = np.random.default_rng(run)
    edges = {}
    with dcd.Context(n, mode=dcd.MODE_BASE) as c:
        for t, other in enumerate((0, 40, 600, 6000, 39_000)):  # records of other edges on the same source
            ins = np.stack([np.zeros(run + other, int), np.full(run + other, 77), rng.integers(1, 9, run + other)], 1)
            ins[run:, 1] = 100 + rng.permutation(n - 100)[:other]
            dels = np.array([[0, 77]] * (t % 2) + [[0, 100 + t]])
            ins = rng.permutation(ins)
            c.apply_batch(ins.astype(np.int32), dels.astype(np.int32))
            st = c.update(labels_out=None)[2]
            model_step(edges, ins, dels)
            check(c, edges, n)
            assert st.m2 == 2 * sum(edges.values())
