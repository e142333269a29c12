"""The coarse levels in one launch against the general path (the host enqueues
every pass) and the oracle: community counts around the cluster's slices, the
shared-memory and the size limits, 32- and 64-bit sums, the level and pass caps,
groups of unequal graphs.  Integers throughout: everything is equal."""
import numpy as np
import pytest

from test_gpu_parity import assert_step_equal, dcd  # noqa: F401

pytestmark = pytest.mark.gpu

INTS = ["levels", "iters_total", "iters_level0", "moves_total", "edges_scanned", "verts_scanned", "communities", "N"]


def cliques(b, w, seed):
    """b cliques of 4, joined in a ring and by random links in nearby blocks:
    level 0 leaves about b communities, which merge over several levels."""
    rng = np.random.default_rng(seed)
    i, j = np.tril_indices(4, -1)
    base = 4 * np.arange(b)
    inside = np.stack([(base[:, None] + i).ravel(), (base[:, None] + j).ravel()], 1)
    ring = np.stack([base, 4 * ((np.arange(b) + 1) % b) + 1], 1) if b > 2 else np.array([[0, 5]])[: b - 1]
    x = rng.integers(0, 4 * b, 3 * b)
    y = np.clip(x + rng.integers(-40, 41, 3 * b), 0, 4 * b - 1)
    far = np.stack([x, y], 1)[x // 4 != y // 4]
    e = np.concatenate([inside, ring, far])
    wt = np.concatenate([np.full(len(inside), 6 * w), rng.integers(1, 3, len(ring) + len(far)) * w])
    return np.concatenate([e, wt[:, None]], 1).astype(np.int32)


def steps(b, w):
    first = cliques(b, w, b)
    later = cliques(b, w, b + 1)[6 * b:][: b + 2]
    none = np.zeros((0, 2), np.int32)
    return [(first, none), (later, first[6 * b: 7 * b: 2, :2]), (first[:6], later[:, :2])]


@pytest.mark.parametrize("w", [1, 1 << 22])
@pytest.mark.parametrize("mode", ["DELTA", "STATIC"])
@pytest.mark.parametrize("b", [1, 2, 33, 64, 65, 130, 515, 700, 1530, 2060])
def test_levels(dcd, orc, b, mode, w):  # noqa: F811
    if w > 1 and b * 36 * w < 1 << 31 and b not in (2, 33):
        w = 1 << 26
    ref = orc.Context(4 * b)
    with dcd.Context(4 * b, mode=getattr(dcd, "MODE_" + mode)) as one, \
            dcd.Context(4 * b, mode=getattr(dcd, "MODE_" + mode), pass_loop_host=True) as gen:
        for ins, dels in steps(b, w):
            for c in (one, gen, ref):
                c.apply_batch(ins, dels)
            lab, q, st = one.update()
            glab, gq, gst = gen.update()
            assert np.array_equal(lab, glab) and q == gq
            assert {k: getattr(st, k) for k in INTS} == {k: getattr(gst, k) for k in INTS}
            assert list(st.edges_bin) == list(gst.edges_bin) and list(st.verts_bin) == list(gst.verts_bin)
            rlab, rq, rst = ref.update(getattr(orc, mode))
            assert_step_equal(st, rst, lab, rlab, q, rq, one.rset(), ref.rset())


@pytest.mark.parametrize("cap", [dict(max_levels=2), dict(max_iters=1), dict(tau_inv=3)])
def test_level_caps(dcd, cap):  # noqa: F811
    with dcd.Context(1200, **cap) as one, dcd.Context(1200, pass_loop_host=True, **cap) as gen:
        for ins, dels in steps(300, 1):
            got = []
            for c in (one, gen):
                c.apply_batch(ins, dels)
                lab, q, st = c.update()
                got.append((lab.tolist(), q, {k: getattr(st, k) for k in INTS}))
            assert got[0] == got[1]


@pytest.mark.parametrize("w", [1, 1 << 24])
@pytest.mark.parametrize("blocks", [[1, 70, 300, 5], [40] * 90, [1500, 1900, 30]])
def test_level_groups(dcd, blocks, w):  # noqa: F811
    ctx = [dcd.Context(4 * b, pass_loop_host=True) for b in blocks]
    grp = dcd.Group([4 * b for b in blocks])
    runs = [steps(b, w) for b in blocks]
    for t in range(3):
        for g, r in enumerate(runs):
            grp.apply_batch(g, *r[t])
            ctx[g].apply_batch(*r[t])
        lab, q, st = grp.update()
        for g in range(len(blocks)):
            glab, gq, gst = ctx[g].update()
            assert np.array_equal(lab[grp.offsets[g]:grp.offsets[g + 1]], glab) and q[g] == gq
            for k in ("levels", "iters_total", "moves_total", "communities", "N"):
                assert getattr(st[g], k) == getattr(gst, k)
    grp.close()
    for c in ctx:
        c.close()
