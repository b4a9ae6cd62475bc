"""Products of up to 128 samples (one diagonal tile) and just above, at the edges of
its stages (8 words), with aligned and unaligned rows: exact counts, compared with
the bits multiplied in float64."""
import numpy as np
import pytest

from paper_1911_04200_gb300 import jsim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count_bits", [32, 64])
@pytest.mark.parametrize("pad", [0, 1])
@pytest.mark.parametrize("n,W", [(1, 1), (2, 7), (33, 8), (64, 9), (96, 1217), (97, 64), (127, 511), (128, 1225),
                                 (129, 40), (160, 1000)])
def test_small_products(gpu, n, W, pad, count_bits):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(n * W)
    stride = W + W % 2 + pad  # pad 1: odd, rows not 16-byte aligned
    X = torch.randint(-(1 << 63), (1 << 63) - 1, (n, stride), generator=g, device="cuda")
    X[0, W - 1] = -1
    bits = ((X[:, :W, None] >> torch.arange(64, device="cuda")) & 1).reshape(n, -1).double()
    ref = (bits @ bits.T).long()
    dt = torch.uint64 if count_bits == 64 else torch.uint32
    for variant in ("auto", "tc"):
        C = torch.empty((n, n), dtype=dt, device="cuda")
        with jsim.Context(count_bits=count_bits) as ctx:
            ctx.product(X, n, W, stride, C, variant=variant)
        assert torch.equal(C.view(torch.int64 if count_bits == 64 else torch.int32).long(), ref)
