"""One hook chain of all vertices, which only imported words can make (a
vertex's cut then holds the edge to its successor and no other). A path's own
sketches give chains of tens: every hop needs a sample that falls on the right
one of two edges."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [4096, 4097, 9001, 1 << 17, 1 << 20])
def test_chain_of_all_vertices(V):
    from paper_2509_14433_gb300 import cupc as C
    from tests._dev import Dev

    params = (2, 1, 2, 1 << 20)  # two layers of three buckets
    i = np.arange(V - 1, dtype=np.uint32)
    path = np.stack([i, i + 1], 1)
    parts = []
    for odd in (0, 1):  # every other edge of the path: a vertex then has that edge alone
        dev = Dev(V, 5, params)
        assert dev.update(path[odd::2]) == 0
        parts.append(dev.export())
        dev.close()
    sk = parts[0]
    sk[:, 1::2] = parts[1][:, 1::2]  # vertex i: the edge (i, i + 1)
    sk[1] = 0  # the one component's cut is empty
    dev = Dev(V, 5, params)
    a = np.ascontiguousarray(sk)
    assert C.cupc_import_sketches(dev.h, a, a.nbytes, None) == 0
    st, forest = dev.forest()
    assert st == 0
    assert np.array_equal(forest, i.astype(np.uint64) * np.uint64(V) + i + 1)
    assert not dev.labels().any()
