"""Ranked ingest of the block-sparse path (thin value ranges: tile bitmaps and
classes over the numbered nonzero rows) and the wide batches of the dense path,
against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1911_04200_gb300 import jsim

pytestmark = pytest.mark.gpu


def thin_sets(n, rows, bits, seed, repeats=False):
    """n samples over `rows` distinct values of [0, 2^bits): every value in one
    to four samples, the smallest and the largest value among them."""
    rng = np.random.default_rng(seed)
    vals = np.unique(np.concatenate([rng.integers(0, 1 << bits, rows - 2, dtype=np.uint64),
                                     np.array([0, (1 << bits) - 1], dtype=np.uint64)]))
    while len(vals) < rows:
        vals = np.unique(np.concatenate([vals, rng.integers(0, 1 << bits, rows - len(vals), dtype=np.uint64)]))
    sets = [[] for _ in range(n)]
    first = rng.integers(0, n, rows)
    for k in range(4):
        keep = np.ones(rows, bool) if k == 0 else rng.random(rows) < 0.4
        who = (first + k * rng.integers(0, 3, rows)) % n
        for i in range(n):
            sets[i].append(vals[keep & (who == i)])
    out = [np.unique(np.concatenate(s)) for s in sets]
    if repeats:
        out = [np.sort(np.concatenate([s, s[: len(s) // 3]])) for s in out]
    off = np.zeros(n + 1, dtype=np.uint64)
    off[1:] = np.cumsum([len(s) for s in out])
    return off, np.concatenate(out).astype(np.uint64)


@pytest.mark.parametrize("filter_min", [1, 2])
@pytest.mark.parametrize("n,rows,bits,repeats", [
    (129, 3000, 33, False),               # two tiles, one with a single sample; values beyond 32 bits
    (260, (1 << 18) - 1, 32, False),      # rows at the edge of a scan block
    (260, 1 << 18, 32, False),
    (260, (1 << 18) + 65, 31, True),
    (1030, 50_000, 32, True),
])
def test_thin_ranges_match_the_oracle(gpu, n, rows, bits, repeats, filter_min):
    off, ids = thin_sets(n, rows, bits, seed=n + rows)
    if repeats:
        off, ids = thin_sets(n, rows, bits, seed=n + rows, repeats=True)
    Co, so, Jo = oracle.all_pairs(off, ids)
    for variant in ("sparse", "auto"):
        with jsim.Context(variant=variant, filter_min=filter_min) as ctx:
            C, s, J = ctx.all_pairs(off, ids)
            st = ctx.stats()
        if variant == "sparse":
            assert st["variant"] == "sparse" and st["windows"] == 0
        assert st["batch_rows"] > 1 << 28, "the batches of a thin range are wide"
        np.testing.assert_array_equal(s, so)
        np.testing.assert_array_equal(C, Co.astype(np.uint32))
        np.testing.assert_array_equal(J.view(np.uint64), Jo.view(np.uint64))
