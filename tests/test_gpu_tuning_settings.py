"""Settings of cupc_set_tuning that are no whole number of record groups, on a
batch long enough that they become the chunk size: every sketch word against
the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2509_14433_gb300 import workloads as WL

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

V, SEED = 3000, 8


@pytest.fixture(scope="module")
def graph():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    E = WL.er_edges(V, 0.05, 5)
    ref = O.Graph(V, SEED)
    assert ref.update(E) == O.OK
    return E, ref.export()


@pytest.mark.parametrize("records", [65, 66, 67, 70, 101, 255, 511])
@pytest.mark.parametrize("per_bucket", [False, True])
def test_settings_that_split_a_group(graph, records, per_bucket):
    from paper_2509_14433_gb300 import autotune as AT
    from paper_2509_14433_gb300 import cupc as C
    from tests._dev import Dev

    E, want = graph
    dev = Dev(V, SEED)
    # one CTA per SM: about 3000 records for each warp of a layer group, so that
    # the setting limits the chunk
    if per_bucket:
        assert C.cupc_set_tuning_bucket(dev.h, AT.bucket_of(len(E)), records, 8, 1) == 0
    else:
        assert C.cupc_set_tuning(dev.h, records, 8, 1) == 0
        out = np.zeros(4, np.uint32)
        assert C.cupc_get_tuning(dev.h, out) == 0 and out[0] == records
    assert dev.update(E) == 0 and dev.sync() == 0
    assert np.array_equal(dev.export(), want)
