"""Recoveries whose hook trees are long chains, whose rows are sampled four at
a time with a remainder, and on both sides of the one-cluster limit, against
the oracle: forests, labels, round logs."""
import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _edges(kind, V):
    i = np.arange(V - 1, dtype=np.uint32)
    if kind == "path":
        return np.stack([i, i + 1], 1)
    if kind == "caterpillar":  # a spine with a leaf at every vertex
        h = V // 2
        s = np.arange(h - 1, dtype=np.uint32)
        leaf = np.arange(h, dtype=np.uint32)
        return np.concatenate([np.stack([s, s + 1], 1), np.stack([leaf, leaf + h], 1)])
    if kind == "tree":  # every vertex to its half
        return np.stack([(i + 1) // 2, i + 1], 1)[1:]
    return np.stack([i[::3], i[::3] + 1], 1)  # pairs and single vertices


@pytest.mark.parametrize("V", [4096, 4097, 9001])
@pytest.mark.parametrize("kind", ["path", "caterpillar", "tree", "pairs"])
def test_long_chains_of_hooks(kind, V):
    from tests._dev import Dev

    dev, ref = Dev(V, 11), O.Graph(V, 11)
    e = _edges(kind, V)
    assert dev.update(e) == 0 and ref.update(e) == O.OK
    s_ref, f_ref = ref.spanning_forest()
    s_dev, f_dev = dev.forest()
    assert s_ref == s_dev
    assert np.array_equal(f_ref, f_dev)
    assert np.array_equal(ref.labels(), dev.labels())
    glog, olog = dev.round_log(), ref.round_log()
    assert len(glog) == len(olog)
    for (gl, gi), (ol, oi) in zip(glog, olog):
        assert gl == ol and np.array_equal(np.sort(gi), np.sort(oi))
