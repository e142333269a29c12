"""dcd_modularity_noalloc at the edges of its row classes: eight lanes a row with
eight entries in flight each, the whole CTA for rows above 512 entries, blocks of 256
rows.  Compared with whole-number sums on the host; Q is the same division, so it
is equal."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EDGES = [0, 1, 7, 8, 9, 63, 64, 65, 127, 511, 512, 513, 767, 5000]


def csr(lengths, seed, wmax):
    n = len(lengths)
    rng = np.random.default_rng(seed)
    rp = np.zeros(n + 1, np.int64)
    rp[1:] = np.cumsum(lengths)
    m = int(rp[-1])
    col = rng.integers(0, n, m).astype(np.int32)
    w = rng.integers(max(1, wmax - 1000), wmax + 1, m).astype(np.int32)
    return rp, col, w, (rng.integers(0, max(1, n // 3), n) * 2 % n).astype(np.int32)


def expect(rp, col, w, lab):
    src = np.repeat(np.arange(len(lab)), np.diff(rp))
    w = w.astype(object)
    m2 = int(w.sum()) if len(w) else 0
    same = int(w[lab[src] == lab[col]].sum()) if len(w) else 0
    a = {}
    for c, x in zip(lab[src].tolist(), w.tolist()):
        a[c] = a.get(c, 0) + x
    N = m2 * same - sum(x * x for x in a.values())
    return (float(N) / (float(m2) * float(m2)) if m2 else 0.0), m2


def layouts():
    rng = np.random.default_rng(3)
    few = rng.integers(0, 12, 1000)
    few[rng.permutation(1000)[: len(EDGES)]] = EDGES
    block = rng.integers(0, 3, 700)
    block[[0, 1, 31, 32, 100, 255, 256, 511]] = [513, 5000, 767, 600, 4096, 513, 1025, 2000]  # several a block
    return {"one": [0], "single long": [5000], "edges": EDGES, "scattered": few, "blocks": block,
            "all long": [513] * 300, "all 512": [512] * 257, "empty": [0] * 300}


@pytest.mark.parametrize("wmax", [1, 2**31 - 1])
@pytest.mark.parametrize("name", list(layouts()))
def test_rows(name, wmax):
    from paper_1904_08553_gb300 import dcd

    g = csr(layouts()[name], len(name), wmax)
    pad = [x if len(x) else np.zeros(1, x.dtype) for x in g]  # no NULL for a graph without entries
    q, m2 = dcd.dcd_modularity_noalloc(len(g[3]), *[torch.from_numpy(x).cuda() for x in pad])
    assert (q, m2) == expect(*g)


@pytest.mark.parametrize("length", [64, 512, 513, 5000])
@pytest.mark.parametrize("what", ["label", "column", "negative"])
def test_bad_values_in_rows(length, what):
    from paper_1904_08553_gb300 import dcd

    n = 700
    lengths = np.full(n, 3)
    lengths[300] = length
    for at in (0, length // 2, length - 1):
        rp, col, w, lab = csr(lengths, length, 5)
        if what == "label":
            lab[300] = n
        else:
            col[rp[300] + at] = n if what == "column" else -1
        with pytest.raises(dcd.DcdError) as e:
            dcd.dcd_modularity_noalloc(n, *[torch.from_numpy(x).cuda() for x in (rp, col, w, lab)])
        assert e.value.code == dcd.DCD_EINVAL
