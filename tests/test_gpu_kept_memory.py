"""What a context keeps between updates: the coarse graph for the next update's
delta rule is sized by the communities of the result, not by those level 0 left,
of which there can be forty times as many."""
import gc

import numpy as np
import pytest

torch = pytest.importorskip("torch")
from test_gpu_coarse_levels import cliques  # noqa: E402
from test_gpu_parity import dcd  # noqa: E402, F401

pytestmark = pytest.mark.gpu


def test_coarse_graph_is_sized_by_the_result(dcd):  # noqa: F811
    b = 4000
    first, later = cliques(b, 1, b), cliques(b, 1, b + 1)[6 * b:][:200]
    none = np.zeros((0, 2), np.int32)
    kept, labels = {}, {}
    for full in (False, True, False, True):  # the second round counts: the process has loaded its kernels
        gc.collect()
        torch.cuda.synchronize()
        free0 = torch.cuda.mem_get_info()[0]
        # from singletons in every update: level 0 leaves about 4000 communities each time
        with dcd.Context(4 * b, mode=dcd.MODE_STATIC, coarsen_full=full) as c:
            for ins in (first, later[:50], later[50:90]):
                c.apply_batch(ins, none)
                lab, _, st = c.update()
                assert st.levels > 2 and st.communities < 400
                assert st.verts_scanned - st.verts_level0 > 1536  # level 1 has that many vertices
            labels[full] = lab
            kept[full] = free0 - torch.cuda.mem_get_info()[0]
    assert np.array_equal(labels[False], labels[True])
    # beside what the rebuild holds: the level-0 matrix (4000^2 cells of 4 bytes and a quarter, 80 MB); two
    # matrices of 400^2 cells of 8 bytes are 3 MB, of 4000^2 cells 320 MB
    assert kept[False] - kept[True] < 200 << 20
