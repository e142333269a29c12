"""Scans of more tiles than are added up one by one: row starts of a graph of 34 M
vertices, pairs of a batch of 17 M records.  Compared with sums on the host."""
import numpy as np
import pytest

from test_gpu_parity import dcd  # noqa: F401

pytestmark = pytest.mark.gpu

TILES = 8192 * 4096  # words


def test_many_vertices(dcd):  # noqa: F811
    n = TILES + 4099
    at = np.array([0, 1, 4095, 4096, 4097, n // 3, TILES - 1, TILES, TILES + 1, n - 4, n - 1])
    e = np.array([(u, v) for i, u in enumerate(at) for v in at[i + 1:]])
    ins = np.concatenate([e, 1 + np.arange(len(e))[:, None]], 1).astype(np.int32)
    with dcd.Context(n, mode=dcd.MODE_DELTA) as c:
        c.apply_batch(ins[::2])
        c.update(labels_out=None)
        c.apply_batch(ins[1::2], np.ascontiguousarray(ins[:8:2, :2]))
        st = c.update(labels_out=None)[2]
        kept = np.ones(len(ins), bool)
        kept[:8:2] = False
        assert (st.nnz, st.m2) == (2 * kept.sum(), 2 * int(ins[kept, 2].sum()))
        rp, col, w = c.graph()
        deg = np.bincount(ins[kept, :2].ravel(), minlength=n)
        assert np.array_equal(np.diff(rp), deg)
        both = np.concatenate([ins[kept], ins[kept][:, [1, 0, 2]]])
        both = both[np.lexsort((both[:, 1], both[:, 0]))]
        assert np.array_equal(col, both[:, 1]) and np.array_equal(w, both[:, 2])
        lab = c.labels()
        assert set(np.flatnonzero(lab != np.arange(n)).tolist()) <= set(at.tolist())


def test_many_records(dcd):  # noqa: F811
    n, m = 2_000_000, TILES // 2 + 300_000
    rng = np.random.default_rng(2)
    ins = np.empty((m, 3), np.int32)
    ins[:, 0] = rng.integers(0, n, m, dtype=np.int32)
    ins[:, 1] = (ins[:, 0] + 1 + rng.integers(0, 2000, m, dtype=np.int32)) % n
    ins[:, 2] = 1 + (ins[:, 0] & 3)
    key = np.sort(ins[:, :2].min(1).astype(np.int64) * n + ins[:, :2].max(1))
    first = key[np.concatenate([[True], key[1:] != key[:-1]])]
    with dcd.Context(n, mode=dcd.MODE_STATIC, max_levels=1, max_iters=1) as c:
        c.apply_batch(ins)
        st = c.update(labels_out=None)[2]
        assert (st.nnz, st.m2) == (2 * len(first), 2 * int(ins[:, 2].sum(dtype=np.int64)))
        rp = c.graph()[0]
    deg = np.bincount(first // n, minlength=n) + np.bincount(first % n, minlength=n)
    assert np.array_equal(np.diff(rp), deg)
