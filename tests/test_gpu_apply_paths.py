"""The update's apply kernels at the sizes where a path can go wrong, every
sketch word against the oracle: vertices whose record counts sit at the edges
of the direct path, the padding, a pass and a chunk; every lane layout (1 to 31
columns); rows that end inside the registers, the shared slots or HBM; edge
ids above and below 32 bits; batches around the one-launch limit. The path is
integer, so equality is exact."""
import numpy as np
import pytest

import oracle as O
from paper_2509_14433_gb300 import workloads as WL

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _stars(V, counts, g):
    """A batch in which hub i has counts[i] records, the hubs spread over the
    ids so that both smaller and larger endpoints occur."""
    hubs = (np.arange(len(counts)) * (V // (len(counts) + 1)) + 3).astype(np.int64)
    free = np.setdiff1d(np.arange(V), hubs)
    e = np.concatenate([np.stack([np.full(c, h), g.choice(free, c, replace=False)], 1) for h, c in zip(hubs, counts)])
    return e[g.permutation(len(e))].astype(np.uint32)


COUNTS = (1, 2, 3, 4, 5, 7, 8, 31, 32, 33, 63, 64, 65, 255, 256, 257, 511, 700)


@pytest.mark.parametrize("V,L,C,D", [(3000, 0, 0, 0), (70001, 3, 2, 5), (66000, 2, 7, 20)])
@pytest.mark.parametrize("rows", [1, 8, 16])
def test_record_counts_at_the_edges_of_passes_and_chunks(V, L, C, D, rows):
    from paper_2509_14433_gb300 import cupc as B
    from tests._dev import Dev

    dev, ref = Dev(V, 5, (L, C, D, 0)), O.Graph(V, 5, L, C, D)
    assert B.cupc_set_tuning(dev.h, 64 if rows == 1 else 0, min(rows, dev.D), 0) == 0
    g = WL.rng(V + rows)
    e = np.concatenate([_stars(V, COUNTS * 2, g), WL.uniform_pairs(V, 10000, g)])
    assert len(e) > 12288  # the grouped path
    assert dev.update(e) == 0 and ref.update(e) == O.OK
    assert dev.sync() == 0
    assert np.array_equal(dev.export(), ref.export())


@pytest.mark.parametrize("C", [1, 2, 3, 4, 7, 8, 15, 16, 31])
@pytest.mark.parametrize("D", [1, 2, 3, 4, 7])
def test_every_lane_layout(C, D):
    from tests._dev import Dev

    V, L = 500, 5
    dev, ref = Dev(V, 9, (L, C, D, 0)), O.Graph(V, 9, L, C, D)
    g = WL.rng(C * 10 + D)
    for n in (300, 13000):  # one launch; grouped
        e = WL.uniform_pairs(V, n, g)
        assert dev.update(e) == 0 and ref.update(e) == O.OK
    assert dev.sync() == 0
    assert np.array_equal(dev.export(), ref.export())


@pytest.mark.parametrize("n", [1, 31, 512, 513, 8192, 8193, 12288, 12289])
def test_batches_around_the_one_launch_limit(n):
    from paper_2509_14433_gb300 import cupc as B
    from tests._dev import Dev

    V = 1500
    dev, ref = Dev(V, 2), O.Graph(V, 2)
    g = WL.rng(n)
    e = WL.uniform_pairs(V, n, g)
    e[: n // 2, 0] = 7  # a hub
    e[: n // 2, 1] = np.where(e[: n // 2, 1] == 7, 8, e[: n // 2, 1])
    assert dev.update(e) == 0 and ref.update(e) == O.OK
    for at, bad in ((0, (V, 1)), (n - 1, (3, 3)), (n // 2, (0, V))):  # dropped whole, then the next one applies
        b = e.copy()
        b[at] = bad
        assert dev.update(b) == 0 and dev.sync() == B.CUPC_EINVAL
    ops = np.ones(n, np.int8)
    ops[n - 1] = 0
    assert dev.update(e, ops) == 0 and dev.sync() == B.CUPC_EINVAL
    assert np.array_equal(dev.export(), ref.export())
    assert dev.update(e[:1]) == 0 and ref.update(e[:1]) == O.OK
    assert dev.sync() == 0 and dev.stats()["chunks"] == 2
    assert np.array_equal(dev.export(), ref.export())


def test_a_sharded_count_with_hubs():
    # V above the shared-histogram limit and enough edges for the sharded
    # counters; few layers and columns keep the oracle quick
    from tests._dev import Dev

    V, L, C, D = 30000, 2, 2, 6
    dev, ref = Dev(V, 4, (L, C, D, 1 << 21)), O.Graph(V, 4, L, C, D)
    g = WL.rng(8)
    e = np.concatenate([_stars(V, (20000, 9000, 1, 2, 3), g), WL.uniform_pairs(V, 1 << 20, g)])
    for part in (e, e[: 1 << 20], e[: (1 << 20) - 1]):
        assert dev.update(part) == 0 and ref.update(part) == O.OK
        bad = part.copy()
        bad[5, 0] = V
        assert dev.update(bad) == 0 and dev.sync() != 0  # its counts are cleared
    assert dev.sync() == 0
    assert np.array_equal(dev.export(), ref.export())


@pytest.mark.parametrize("V,n", [(1024, 60000), (24576, 1 << 20)])
def test_invalid_edges_all_over_a_shared_histogram_batch(V, n):
    # every CTA meets bad edges while others start: the batch is dropped whole,
    # its counts are cleared and the next batch applies
    from paper_2509_14433_gb300 import cupc as B
    from tests._dev import Dev

    L, C, D = 3, 2, 6
    dev, ref = Dev(V, 6, (L, C, D, 0)), O.Graph(V, 6, L, C, D)
    g = WL.rng(V)
    e = WL.uniform_pairs(V, n, g)
    bad = e.copy()
    bad[::97, 1] = V + 5
    for part in (bad, e, bad[::-1], bad):
        if part is e:
            assert dev.update(e) == 0 and ref.update(e) == O.OK and dev.sync() == 0
        else:
            assert dev.update(part) == 0 and dev.sync() == B.CUPC_EINVAL
    assert np.array_equal(dev.export(), ref.export())


def _b_words(seed, L, C):
    """The addends b of the columns: words L*(C+1) + 3k of the key stream."""
    j = np.uint64(L * (C + 1)) + np.uint64(3) * np.arange(L * C, dtype=np.uint64)
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + np.uint64(0x9E3779B97F4A7C15) * (j + np.uint64(1))
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


@pytest.mark.parametrize("zeros", [3, 5, 11, 14])
def test_padding_in_columns_whose_hash_of_zero_is_deep(zeros):
    # padding records have the id zero, whose depth in a column is the leading
    # zeros of its b: below, inside and beyond the shared rows
    from tests._dev import Dev

    V, L, C, D = 900, 6, 7, 20
    seed = next(s for s in range(1, 1 << 20)
                if ((_b_words(s, L, C) >> np.uint64(63 - zeros)) == 1).any())
    dev, ref = Dev(V, seed, (L, C, D, 0)), O.Graph(V, seed, L, C, D)
    g = WL.rng(zeros)
    e = np.concatenate([_stars(V, (3, 5, 6, 7, 9, 33, 401), g), WL.uniform_pairs(V, 13000, g)])
    assert dev.update(e) == 0 and ref.update(e) == O.OK
    assert dev.sync() == 0
    assert np.array_equal(dev.export(), ref.export())


@pytest.mark.parametrize("hub_share", [0.0, 0.1, 0.15, 0.9])
@pytest.mark.parametrize("records", [0, 70])
def test_hubs_on_a_small_graph_around_the_share_that_changes_the_chunks(hub_share, records):
    # a hundred records a vertex on average, so that the plan counts the hubs':
    # none, an eighth of all records less and more a little, nearly all
    from paper_2509_14433_gb300 import cupc as B
    from tests._dev import Dev

    V, n, L, C, D = 700, 35000, 9, 7, 18
    dev, ref = Dev(V, 3, (L, C, D, 0)), O.Graph(V, 3, L, C, D)
    assert B.cupc_set_tuning(dev.h, records, 0, 0) == 0
    g = WL.rng(int(100 * hub_share))
    e = WL.uniform_pairs(V, n, g)
    k = int(2 * n * hub_share / 2)  # each edge of the hubs' part gives them one record or two
    e[:k, 0] = g.integers(0, max(1, k // 1500 + 1), k)
    e[:k, 1] = np.where(e[:k, 1] == e[:k, 0], 600, e[:k, 1])
    e = e[g.permutation(n)]
    for part in (e, e[::-1], e[:12500]):
        part = np.ascontiguousarray(part)
        assert dev.update(part) == 0 and ref.update(part) == O.OK
    assert dev.sync() == 0
    assert np.array_equal(dev.export(), ref.export())


@pytest.mark.parametrize("V", [4097, 70001])
@pytest.mark.parametrize("C,D", [(1, 3), (2, 1), (3, 2), (7, 4), (7, 5), (8, 9), (16, 6), (31, 5)])
def test_one_launch_batches_with_hubs(V, C, D):
    # a star whose centre is now the first, now the second end; two stars; an
    # edge toggled twice (its sums cancel); no hub; bad edges; and the sizes
    # around the one from which hubs are looked for and where the CTAs grow
    from paper_2509_14433_gb300 import cupc as B
    from tests._dev import Dev

    L = 3
    dev, ref = Dev(V, 12, (L, C, D, 0)), O.Graph(V, 12, L, C, D)
    g = WL.rng(C * 100 + D)
    leaves = 1 + g.permutation(V - 1)[:4096].astype(np.uint32)
    star = np.stack([np.zeros(4096, np.uint32), leaves], 1)
    star[::3] = star[::3, ::-1]
    two = np.concatenate([star[:2500], np.stack([np.full(2600, V - 1), np.arange(1, 2601)], 1)]).astype(np.uint32)
    for e in (np.concatenate([star, star[:1]]), np.concatenate([star, star]), np.concatenate([two, two[::-1]])[:9000],
              np.concatenate([WL.uniform_pairs(V, 12287, g), star[:1]]), np.tile(star, (3, 1))[:12288],
              np.concatenate([star, WL.uniform_pairs(V, 8193 - 4096, g)])):
        e = np.ascontiguousarray(e, np.uint32)
        assert 4096 < len(e) <= 12288
        assert dev.update(e) == 0 and ref.update(e) == O.OK
        bad = e.copy()
        bad[len(e) // 2, 1] = bad[len(e) // 2, 0]
        assert dev.sync() == 0 and dev.update(bad) == 0 and dev.sync() == B.CUPC_EINVAL
    assert np.array_equal(dev.export(), ref.export())
