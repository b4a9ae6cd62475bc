"""Values spread thinly over wide ranges (64-bit hashes) and values in a few
clusters far apart: results against the oracle, and the width of the row
batches.  Empty stretches cost nothing, so a wide batch saves nothing there
and clears and scans its bitmap for the few values it holds; values spread
over all of a range of a few 2^32 still take wide batches."""
import numpy as np
import pytest

import oracle
from paper_1911_04200_gb300 import jsim

pytestmark = pytest.mark.gpu

TOP = 1 << 64


def collection(n, draw):
    segs = [np.unique(draw(i)) for i in range(n)]
    off = np.zeros(n + 1, dtype=np.uint64)
    off[1:] = np.cumsum([s.size for s in segs])
    return off, np.concatenate(segs)


def hashed(n, per, seed):
    rng = np.random.default_rng(seed)
    pool = rng.integers(0, TOP, 2 * per, dtype=np.uint64)
    return collection(n, lambda i: rng.choice(pool, per))


def clusters(n, per, starts, seed, width=1 << 18):
    rng = np.random.default_rng(seed)
    at = np.array(starts, dtype=np.uint64)
    return collection(n, lambda i: at[rng.integers(0, len(at), per)] + rng.integers(0, width, per, dtype=np.uint64))


def spread(n, per, bits, seed):
    rng = np.random.default_rng(seed)
    return collection(n, lambda i: rng.integers(0, 1 << bits, per, dtype=np.uint64))


CASES = [
    ("hashed", lambda: hashed(8, 150, 1), False),
    ("hashed, a sketch's range of samples", lambda: hashed(300, 200, 2), False),
    ("clusters over 2^40", lambda: clusters(40, 3000, [0, 1 << 33, (1 << 40) - (1 << 18)], 3), False),
    ("clusters over 2^64", lambda: clusters(40, 3000, [5, 1 << 50, TOP - (1 << 18)], 4), False),
    ("clusters over 2^35", lambda: clusters(300, 300, [0, 1 << 34, 1 << 35], 5), False),
    ("clusters over 2^32", lambda: clusters(40, 3000, [0, (1 << 32) - (1 << 18)], 9), False),
    ("one value, then a cluster", lambda: clusters(40, 3000, [1 << 36] * 999 + [0], 6), False),
    ("spread over 2^33", lambda: spread(40, 3000, 33, 7), True),
    ("spread over 2^36", lambda: spread(40, 3000, 36, 8), True),
]


@pytest.mark.parametrize("filter_min", [1, 2])
@pytest.mark.parametrize("name,make,wide", CASES, ids=[c[0] for c in CASES])
def test_width_follows_the_values(gpu, name, make, wide, filter_min):
    off, ids = make()
    Co, so, Jo = oracle.all_pairs(off, ids)
    with jsim.Context(filter_min=filter_min) as ctx:
        C, s, J = ctx.all_pairs(off, ids)
        rows = ctx.stats()["batch_rows"]
    np.testing.assert_array_equal(s, so)
    np.testing.assert_array_equal(C.astype(np.uint64), Co)
    np.testing.assert_array_equal(J.view(np.uint64), Jo.view(np.uint64))
    assert rows > 1 << 28 if wide else rows <= 1 << 28


@pytest.mark.parametrize("name,make,wide", CASES, ids=[c[0] for c in CASES])
def test_block_sparse_over_the_same_ranges(gpu, name, make, wide):
    off, ids = make()
    Co, so, Jo = oracle.all_pairs(off, ids)
    with jsim.Context(variant="sparse") as ctx:
        C, s, J = ctx.all_pairs(off, ids)
        st = ctx.stats()
    assert st["variant"] == "sparse"
    np.testing.assert_array_equal(s, so)
    np.testing.assert_array_equal(C.astype(np.uint64), Co)
    np.testing.assert_array_equal(J.view(np.uint64), Jo.view(np.uint64))
    assert st["batch_rows"] > 1 << 28 if wide else st["batch_rows"] <= 1 << 28


@pytest.mark.parametrize("values", [[0], [TOP - 1], [0, TOP - 1], [7] * 3, [1 << 40, (1 << 40) + 1],
                                    [0, 1 << 32, 1 << 33, TOP - 1]])
def test_fewer_values_than_probes(gpu, values):
    segs = [sorted(values), [], sorted(set(values))[:1]]
    off = np.array([0, len(segs[0]), len(segs[0]), len(segs[0]) + 1], dtype=np.uint64)
    ids = np.array(segs[0] + segs[2], dtype=np.uint64)
    Co, so, Jo = oracle.all_pairs(off, ids)
    for variant in ("auto", "sparse"):
        with jsim.Context(variant=variant) as ctx:
            C, s, J = ctx.all_pairs(off, ids)
        np.testing.assert_array_equal(s, so)
        np.testing.assert_array_equal(C.astype(np.uint64), Co)
        np.testing.assert_array_equal(J.view(np.uint64), Jo.view(np.uint64))
