"""Batches on both sides of the records per vertex from which the library takes
long chunks by itself, with and without hubs, and with the chunks set."""
import numpy as np
import pytest

import oracle as O
from paper_2509_14433_gb300 import workloads as WL

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("records", [0, 256, 512])
@pytest.mark.parametrize("hubs", [False, True])
@pytest.mark.parametrize("V", [600, 2457, 2458, 2600])  # 12289 edges: 41, 10.003, 9.999 and 9.5 records a vertex
def test_long_chunks(V, hubs, records):
    from paper_2509_14433_gb300 import cupc as C
    from tests._dev import Dev

    dev, ref = Dev(V, 31, (4, 0, 0, 0)), O.Graph(V, 31, 4, 0, 0)
    assert C.cupc_set_tuning(dev.h, records, 0, 0) == 0
    out = np.zeros(4, np.uint32)
    assert C.cupc_get_tuning(dev.h, out) == 0 and out[0] == (records or 256)
    assert C.cupc_set_tuning_bucket(dev.h, 7, records, 8, 2) == 0
    g = WL.rng(V)
    for n in (12289, 16384, 100003):
        e = WL.uniform_pairs(V, n, g)
        if hubs:
            e[: n // 3, 0] = g.integers(0, 3, n // 3)
            e[: n // 3, 1] = np.where(e[: n // 3, 1] < 3, V - 1, e[: n // 3, 1])
            e = e[g.permutation(n)]
        e = np.ascontiguousarray(e, np.uint32)
        assert dev.update(e) == 0 and ref.update(e) == O.OK
    assert dev.sync() == 0
    assert np.array_equal(dev.export(), ref.export())
