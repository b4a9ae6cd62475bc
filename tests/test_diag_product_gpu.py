"""The diagonal-tile product of the block-sparse path at the edges of its
stages (8 words), tiles (128 samples) and 16-tile launches: samples of one
tile share values no other tile holds, so all counts within it come from that
product.  Counts are integers and J their correctly rounded quotient, so the
comparison with the oracle is exact."""
import numpy as np
import pytest

import oracle
from paper_1911_04200_gb300 import jsim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count_bits", [32, 64])
@pytest.mark.parametrize("n,rows", [(1, 1), (2, 64), (127, 449), (128, 512), (129, 513), (256, 1024), (300, 700),
                                    (1025, 100), (2048, 577)])
def test_tiles_of_their_own_values(gpu, n, rows, count_bits):
    rng = np.random.default_rng(n + rows)
    segs = []
    for i in range(n):
        lo = (i // 128) * (1 << 16)  # each group of 128 samples in a window of its own
        segs.append(lo + np.flatnonzero(rng.random(rows) < 0.5).astype(np.uint64))
    off = np.zeros(n + 1, dtype=np.uint64)
    off[1:] = np.cumsum([s.size for s in segs])
    ids = np.concatenate(segs).astype(np.uint64)
    with jsim.Context(variant="sparse", id_bits=21, count_bits=count_bits) as ctx:
        C, s, J = ctx.all_pairs(off, ids)
    Co, so, Jo = oracle.all_pairs(off, ids)
    np.testing.assert_array_equal(s, so)
    np.testing.assert_array_equal(C.astype(np.uint64), Co)
    np.testing.assert_array_equal(J.view(np.uint64), Jo.view(np.uint64))
