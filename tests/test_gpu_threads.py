"""Contexts of several threads side by side, one context a thread: each thread's
results are those it gets alone.  The coarse levels of the two sizes need different
amounts of shared memory, which is a setting of the process."""
import threading

import numpy as np
import pytest

from test_gpu_coarse_levels import cliques
from test_gpu_parity import dcd  # noqa: F401

pytestmark = pytest.mark.gpu


def test_contexts_in_threads(dcd):  # noqa: F811
    blocks, rounds = (60, 550) * 4, 1500
    none = np.zeros((0, 2), np.int32)
    ctx, alone = [], []
    for b in blocks:
        c = dcd.Context(4 * b, mode=dcd.MODE_STATIC)
        c.apply_batch(cliques(b, 1, b), none)
        lab, q, st = c.update()
        assert st.levels > 1
        ctx.append(c)
        alone.append((lab, q))
    wrong = []
    go = threading.Barrier(len(blocks))

    def run(i):
        go.wait()
        for t in range(rounds):
            try:
                lab, q, _ = ctx[i].update(None if t % 100 else "host")
            except dcd.DcdError as e:
                wrong.append((i, t, str(e)))
                return
            if q != alone[i][1] or (lab is not None and not np.array_equal(lab, alone[i][0])):
                wrong.append((i, t, "labels"))
                return

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(blocks))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for c in ctx:
        c.close()
    assert not wrong
