"""Sums over every entry of a graph (degrees and 2m after a checkpoint, the weight
inside communities after set_labels), whatever rows it has: long rows, rows of one
entry, runs of empty rows, against the oracle; and not much slower with one row of
half the entries than with even rows."""
import numpy as np
import pytest

from test_gpu_parity import assert_step_equal, dcd  # noqa: F401

pytestmark = pytest.mark.gpu
NONE = np.zeros((0, 2), np.int32)


def edges(kind, n, seed):
    rng = np.random.default_rng(seed)
    m = 4 * n
    u, v = rng.integers(0, n, m), rng.integers(0, n, m)
    if kind == "hub":
        u[: 2 * n] = min(3, n - 1)
    elif kind == "pairs":  # one entry a row
        u = np.arange(0, n - 1, 2)
        v = u + 1
    elif kind == "sparse":  # most rows empty
        u, v = u // 97 * 97 % n, v // 89 * 89 % n
    elif kind == "ends":
        u, v = np.array([0, n - 1, 0]), np.array([n - 1, n - 2, 1])
    e = np.stack([u, v, rng.integers(1, 9, len(u))], 1)
    return e[u != v].astype(np.int32)


@pytest.mark.parametrize("kind", ["even", "hub", "pairs", "sparse", "ends"])
@pytest.mark.parametrize("n", [3, 64, 5000])
def test_after_checkpoint_and_set_labels(dcd, orc, tmp_path, kind, n):  # noqa: F811
    ref = orc.Context(n)
    c = dcd.Context(n, mode=dcd.MODE_DELTA)
    for t in range(4):
        ins = edges(kind, n, t)[: None if t == 0 else max(1, n // 20)]
        dels = NONE if t == 0 else np.ascontiguousarray(edges(kind, n, t - 1)[::7, :2])
        if t in (1, 3):
            c.save(tmp_path / "c")
            c.close()
            c = dcd.Context.load(tmp_path / "c")
        if t in (2, 3):
            lab = (np.arange(n) // 5 * 5 % n).astype(np.int32)
            c.set_labels(lab)
            ref.set_labels(lab)
        for x in (c, ref):
            x.apply_batch(ins, dels)
        lab, q, st = c.update()
        rlab, rq, rst = ref.update(orc.DELTA)
        assert_step_equal(st, rst, lab, rlab, q, rq, c.rset(), ref.rset())
    c.close()


def test_time_with_a_long_row(dcd, tmp_path):  # noqa: F811
    n, m = 1_000_000, 1_000_000
    rng = np.random.default_rng(2)
    other = np.stack([rng.integers(1, n, m), rng.integers(1, n, m), np.ones(m, int)], 1)
    star = np.stack([np.zeros(m, int), 1 + rng.permutation(n - 1)[: m - 1].repeat(2)[:m], np.ones(m, int)], 1)
    even = np.stack([rng.integers(1, n, m), rng.integers(1, n, m), np.ones(m, int)], 1)
    ms = {}
    for name, e in (("hub", star), ("even", even)):
        e = np.concatenate([e, other])
        e = e[e[:, 0] != e[:, 1]].astype(np.int32)
        best = []
        for _ in range(3):
            c = dcd.Context(n, mode=dcd.MODE_BASE, max_iters=1, max_levels=1)
            c.apply_batch(e)
            c.update(labels_out=None)
            c.save(tmp_path / "c")
            c.close()
            c = dcd.Context.load(tmp_path / "c")
            c.apply_batch(e[:10])
            best.append(c.update(labels_out=None)[2].ms_merge)
            c.close()
        ms[name] = min(best)
    assert ms["hub"] < 4 * ms["even"], ms
