"""One-launch batches around the sizes from which the kernel looks for hubs."""
import numpy as np
import pytest

import oracle as O
from paper_2509_14433_gb300 import workloads as WL

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [3071, 3072, 3073, 3500, 4096])
@pytest.mark.parametrize("V", [4096, 4097, 70001])
def test_stars_around_the_limits(V, n):
    from tests._dev import Dev

    dev, ref = Dev(V, 21, (3, 0, 0, 0)), O.Graph(V, 21, 3, 0, 0)
    g = WL.rng(n)
    leaves = 1 + g.permutation(V - 1)[:n - 1].astype(np.uint32)
    star = np.concatenate([np.stack([np.zeros(len(leaves), np.uint32), leaves], 1), WL.uniform_pairs(V, n - len(leaves), g)])
    half = np.concatenate([star[: n // 2], WL.uniform_pairs(V, n - n // 2, g)])
    for e in (star, star[::-1, ::-1], half):
        e = np.ascontiguousarray(e, np.uint32)
        assert len(e) == n and dev.update(e) == 0 and ref.update(e) == O.OK
    assert dev.sync() == 0
    assert np.array_equal(dev.export(), ref.export())
