"""The local move's lane lists and entry labels at their edges, against the
oracle: rows around the lengths of the short bins with few and with many
foreign entries (a lane's list, and the segment that takes over when it is
full), hub rows around a chunk, 64- and 128-bit gains; and a graph large enough
that level 0 keeps its labels in entry order, through passes that move most and
passes that move few."""
import numpy as np
import pytest

from test_gpu_parity import assert_step_equal, dcd  # noqa: F401

pytestmark = pytest.mark.gpu


def degree_stream(n, degs, wmax, seed):
    """Vertices of the given degrees (the rest is filler), then a batch of
    changes; weights 1..wmax."""
    rng = np.random.default_rng(seed)
    steps = []
    e = []
    for v, d in enumerate(degs):
        to = rng.choice(np.arange(len(degs), n), d, replace=False)
        e.append(np.stack([np.full(d, v), to, rng.integers(1, wmax + 1, d)], 1))
    f = rng.integers(len(degs), n, (2 * n, 2))
    f = f[f[:, 0] != f[:, 1]]
    e.append(np.concatenate([f, rng.integers(1, wmax + 1, (len(f), 1))], 1))
    steps.append((np.concatenate(e).astype(np.int32), np.zeros((0, 2), np.int32)))
    for _ in range(2):
        i = rng.integers(0, n, (n // 4, 2))
        i = i[i[:, 0] != i[:, 1]]
        first = steps[0][0]
        steps.append((np.concatenate([i, rng.integers(1, wmax + 1, (len(i), 1))], 1).astype(np.int32),
                      np.ascontiguousarray(first[rng.integers(0, len(first), n // 8), :2])))
    return steps


@pytest.mark.parametrize("mode", ["DELTA", "BASE", "STATIC"])
@pytest.mark.parametrize("wmax", [1, 9, 400_000])
def test_row_lengths(dcd, orc, mode, wmax):  # noqa: F811
    degs = [1, 2, 3, 4, 5, 15, 16, 17, 18, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 512, 513, 1024, 4096,
            4097, 5119, 5120, 5121] + [16, 17, 32] * 40
    n = 6000
    steps = degree_stream(n, degs, wmax, 7 + wmax)
    ref = orc.Context(n)
    with dcd.Context(n, mode=getattr(dcd, "MODE_" + mode)) as ctx:
        for ins, dels in steps:
            ctx.apply_batch(ins, dels)
            ref.apply_batch(ins, dels)
            lab, q, st = ctx.update()
            rlab, rq, rst = ref.update(getattr(orc, mode))
            assert_step_equal(st, rst, lab, rlab, q, rq, ctx.rset(), ref.rset())
        if wmax > 9:
            assert st.m2 >= 1 << 31  # the 128-bit gains


@pytest.mark.parametrize("mode,host_loop", [("STATIC", False), ("DELTA", False), ("DELTA", True)])
def test_entry_labels(dcd, orc, synth, mode, host_loop):  # noqa: F811
    n = 50_000
    s = synth.lfr(synth.seed_for(1, 5), n, 24 * n + n, steps=3, kmax=5000.0, smax=5000.0)
    big = s.steps[0]
    first = (np.concatenate([st[0] for st in s.steps[:2]]), big[1])  # two steps' events: above the size at which
    ref = orc.Context(n)                                               # labels are kept in entry order
    with dcd.Context(n, mode=getattr(dcd, "MODE_" + mode), pass_loop_host=host_loop) as ctx:
        nnz = []
        for ins, dels in [first, s.steps[2], (s.steps[1][0][:40], s.steps[2][1][:10])]:
            ctx.apply_batch(ins, dels)
            ref.apply_batch(ins, dels)
            lab, q, st = ctx.update()
            rlab, rq, rst = ref.update(getattr(orc, mode))
            assert_step_equal(st, rst, lab, rlab, q, rq, ctx.rset(), ref.rset())
            nnz.append(st.nnz)
        assert nnz[1] >= 1 << 21


@pytest.mark.parametrize("empty,wmax", [(0, 1), (40, 4000), (20, 1)])
def test_entry_labels_resummed(dcd, orc, empty, wmax):  # noqa: F811
    """Passes that move most vertices, with no empty rows, with some among the
    others (few enough to sum the labels' agreement along with their gather), and
    with too many; ragged sizes, 64- and 128-bit gains."""
    n = 70_013
    rng = np.random.default_rng(empty + wmax)
    live = np.arange(n) if not empty else np.nonzero(np.arange(n) % empty)[0]
    m = 19 * n
    u = live[rng.integers(0, len(live), m)]
    v = live[np.minimum(np.searchsorted(live, u) // 60 * 60 + rng.integers(0, 60, m), len(live) - 1)]
    far = rng.random(m) < 0.2
    v[far] = live[rng.integers(0, len(live), int(far.sum()))]
    ok = u != v
    ins = np.stack([u, v, rng.integers(1, wmax + 1, m)], 1)[ok].astype(np.int32)
    none = np.zeros((0, 2), np.int32)
    ref = orc.Context(n)
    with dcd.Context(n, mode=dcd.MODE_STATIC) as ctx:
        for a, b in [(ins, none), (ins[:50], ins[100:160, :2])]:
            ctx.apply_batch(a, b)
            ref.apply_batch(a, b)
            lab, q, st = ctx.update()
            rlab, rq, rst = ref.update(orc.STATIC)
            assert_step_equal(st, rst, lab, rlab, q, rq, ctx.rset(), ref.rset())
        assert st.nnz >= 1 << 21 and (wmax == 1 or st.m2 >= 1 << 31)
