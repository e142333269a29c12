"""Vertices and communities without entries, against the oracle: many isolated
vertices (the coarse graphs leave them out), vertices that get their first
edges, communities whose members lose all of theirs, a graph that loses every
edge; single contexts (with the kept coarse graph and without) and groups."""
import numpy as np
import pytest

from test_gpu_parity import assert_step_equal, dcd  # noqa: F401

pytestmark = pytest.mark.gpu


def stream(n, live, seed):
    """Cliques on the first `live` vertices of n; each step connects some fresh
    vertices, and disconnects some cliques altogether."""
    rng = np.random.default_rng(seed)
    k = 6
    tri = np.array([(i, j) for i in range(k) for j in range(i)])
    cl = lambda b: np.concatenate([b * k + tri, np.ones((len(tri), 1), int)], 1)  # noqa: E731
    m = live // k
    x = rng.integers(0, live, (live // 3, 2))
    x = x[x[:, 0] != x[:, 1]]
    cross = np.concatenate([x, np.ones((len(x), 1), int)], 1)
    steps = [(np.concatenate([cl(b) for b in range(m)] + [cross]), np.zeros((0, 2), int))]
    at = live
    for t in range(4):
        fresh = np.arange(at, at + 9)
        at += 9
        old = rng.integers(0, live, 9)
        ins = np.concatenate([np.stack([fresh, old, np.ones(9, int)], 1), [[fresh[0], fresh[1], 2], [fresh[2], fresh[3], 1]]])
        gone = [t, t + 7]  # two cliques lose their edges (and their crossing ones)
        inside = lambda c: np.isin(c // k, gone)  # noqa: E731
        d = np.concatenate([cl(b)[:, :2] for b in gone] + [cross[inside(cross[:, 0]) | inside(cross[:, 1])][:, :2]])
        steps.append((ins, d))
    every = np.concatenate([s[0][:, :2] for s in steps])
    steps.append((steps[0][0][:0], every))                       # every edge goes
    steps.append((steps[0][0][: 5 * len(tri)], every[:0]))       # and some come back
    return [(i.astype(np.int32), d.astype(np.int32)) for i, d in steps]


@pytest.mark.parametrize("mode", ["DELTA", "BASE"])
@pytest.mark.parametrize("n,full", [(9000, False), (9000, True), (400, False)])
def test_isolated(dcd, orc, mode, n, full):  # noqa: F811
    ref = orc.Context(n)
    took = []
    with dcd.Context(n, mode=getattr(dcd, "MODE_" + mode), coarsen_full=full) as ctx:
        for ins, dels in stream(n, 240, 5):
            ctx.apply_batch(ins, dels)
            ref.apply_batch(ins, dels)
            lab, q, st = ctx.update()
            rlab, rq, rst = ref.update(getattr(orc, mode))
            assert_step_equal(st, rst, lab, rlab, q, rq, ctx.rset(), ref.rset())
            took.append(st.coarse0_delta)
    # 9000 vertices are far more communities than the dense coarse graph holds,
    # but only the connected ones count
    assert any(took) != full


def test_isolated_group(dcd, orc):  # noqa: F811
    sizes = [700, 260, 5000]
    streams = [stream(n, 240 if n > 500 else 120, 11 + n) for n in sizes]
    refs = [orc.Context(n) for n in sizes]
    grp = dcd.Group(sizes, mode=dcd.MODE_DELTA)
    for t in range(len(streams[0])):
        for g, s in enumerate(streams):
            grp.apply_batch(g, *s[t])
            refs[g].apply_batch(*s[t])
        lab, q, st = grp.update()
        for g in range(len(sizes)):
            rlab, rq, rst = refs[g].update(orc.DELTA)
            assert np.array_equal(lab[grp.offsets[g]:grp.offsets[g + 1]], rlab)
            assert abs(q[g] - rq) <= 1e-12 * max(1.0, abs(rq))
            assert st[g].communities == rst.communities and st[g].levels == rst.levels
            assert st[g].N == rst.N and st[g].moves_total == rst.moves_total
    grp.close()
