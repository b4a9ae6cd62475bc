"""The SM-pair tensor-core product (variant tc2) at the sizes where its tiles,
units, loads and accumulations have edges, against the CUDA-core product of the
same words (both sums of at most 64 W ones per pair: integers, so equal)."""
import numpy as np
import pytest

from paper_1911_04200_gb300 import jsim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,W,pad,skip", [
    (1, 1, 1, 0),            # one bit-row, one row of one tile
    (127, 15, 1, 0),         # a unit (16 words) less one; rows of 128 less one
    (128, 16, 0, 0),
    (129, 17, 1, 0),         # second CTA's first row, second unit's first word
    (255, 33, 1, 0),         # odd words of a line
    (256, 31, 1, 1),         # 8-byte aligned rows: the copying path (odd stride below, odd base here)
    (257, 48, 0, 0),         # three tiles
    (300, 47, 2, 0),         # odd stride: the copying path
    (513, 200, 0, 1),        # odd base, six tiles, fewer units than clusters
    (700, 5000, 0, 0),
    (1100, 30_000, 8, 0),    # 15 tiles, three chunks of units (the middle one walked backwards)
])
def test_edges(gpu, n, W, pad, skip):
    import torch
    g = torch.Generator(device="cuda").manual_seed(n * 1_000_003 + W)
    stride = W + pad
    bits = torch.randint(-(1 << 63), (1 << 63) - 1, (n * stride + skip,), generator=g, device="cuda")
    bits &= torch.randint(-(1 << 63), (1 << 63) - 1, bits.shape, generator=g, device="cuda")
    with jsim.Context(count_bits=64) as c64, jsim.Context() as c32:
        ref = c64.product(bits[skip:], n, W, stride, variant="popc").view(torch.int64)
        C64 = c64.product(bits[skip:], n, W, stride, variant="tc2").view(torch.int64)
        C32 = c32.product(bits[skip:], n, W, stride, variant="tc2").view(torch.int32)
        torch.cuda.synchronize()
    assert torch.equal(C64, ref)
    assert torch.equal(C32.long(), ref)


def test_accumulation_cap(gpu):
    """All-ones rows past 2^22 bit-rows on several tiles: every accumulation
    ends at its exact cap and the next one starts (counts 64 W above 2^23)."""
    import torch
    n, W = 300, (1 << 17) + 5
    X = torch.full((n, W + 1), -1, dtype=torch.int64, device="cuda")
    with jsim.Context(count_bits=64) as ctx:
        C = ctx.product(X, n, W, W + 1, variant="tc2").view(torch.int64)
        torch.cuda.synchronize()
    np.testing.assert_array_equal(C.cpu().numpy(), np.full((n, n), 64 * W))
