"""Delta-screening's two directions of marking neighbourhoods and its reverse-
pair lookups, against the oracle: batches of deletes inside communities (they
mark neighbourhoods but flag no community, so every mark counts), from few
listed rows (push) to most (pull), rows whose only listed neighbour lies at the
end, vertices that lose their last edge, repeated inserts, 64- and 128-bit
gains."""
import numpy as np
import pytest

from test_gpu_parity import assert_step_equal, dcd  # noqa: F401

pytestmark = pytest.mark.gpu


def graph(rng, n, blocks, wmax):
    """Dense blocks (communities), long rows (vertices 0..4 see every block's
    low members first), leaf pairs at the end."""
    lab = np.arange(n) % blocks
    e = []
    for b in range(blocks):
        m = np.nonzero(lab == b)[0]
        m = m[m < n - 40]
        i = rng.integers(0, len(m), (12 * len(m), 2))
        e.append(m[i])
    for h in range(5):
        e.append(np.stack([np.full(600 - 100 * h, h), 10 + np.arange(600 - 100 * h)], 1))
        e.append(np.array([[h, n - 50 - h]]))
    leaf = n - 40 + 2 * np.arange(20)
    e.append(np.stack([leaf, leaf + 1], 1))
    e = np.concatenate(e)
    e = e[e[:, 0] != e[:, 1]]
    return np.concatenate([e, rng.integers(1, wmax + 1, (len(e), 1))], 1).astype(np.int32)


@pytest.mark.parametrize("wmax", [1, 300_000])
@pytest.mark.parametrize("share", [0.0005, 0.02, 0.3, 0.9])
def test_mark_directions(dcd, orc, share, wmax):  # noqa: F811
    n, blocks = 4000, 8
    rng = np.random.default_rng(int(share * 1e4) + wmax)
    e = graph(rng, n, blocks, wmax)
    ref = orc.Context(n)
    with dcd.Context(n, mode=dcd.MODE_DELTA) as ctx:
        def step(ins, dels):
            ctx.apply_batch(ins, dels)
            ref.apply_batch(ins, dels)
            lab, q, st = ctx.update()
            rlab, rq, rst = ref.update(orc.DELTA)
            assert_step_equal(st, rst, lab, rlab, q, rq, ctx.rset(), ref.rset())
            return lab

        none = np.zeros((0, 3), np.int32)
        lab = step(e, none[:, :2])
        # deletes inside communities, between vertices of high ids first
        same = e[lab[e[:, 0]] == lab[e[:, 1]]]
        high = same[(same[:, 0] > n // 2) & (same[:, 1] > n // 2)]
        dels = high[rng.integers(0, len(high), max(1, int(share * len(high))))][:, :2]
        dels = np.concatenate([dels, dels[:2, ::-1]])  # repeats, the other way round
        step(none, dels.astype(np.int32))
        # the leaf pairs lose their only edge; a few inserts, some of them twice
        leaf = n - 40 + 2 * np.arange(10)
        ins = rng.integers(0, n - 40, (max(4, int(share * 2000)), 2))
        ins = ins[ins[:, 0] != ins[:, 1]]
        ins = np.concatenate([ins, ins[: len(ins) // 3, ::-1], ins[: len(ins) // 5]])
        ins = np.concatenate([ins, rng.integers(1, wmax + 1, (len(ins), 1))], 1).astype(np.int32)
        step(ins, np.stack([leaf, leaf + 1], 1).astype(np.int32))
        # inserts and deletes of the same edges
        step(ins[::2], ins[1::3, :2])
