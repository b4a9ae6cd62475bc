"""The automatic choice for few samples under a tight bound on device waits,
and the diagonal-tile product past the most bit-rows one accumulation takes
(2^22 per CTA): two samples of 1.1e7 words, all ones but the second's first
word."""
import pytest

from paper_1911_04200_gb300 import jsim

pytestmark = pytest.mark.gpu

W = 11_000_000  # 148 CTAs x 8192 stages of 8 words = 9.7e6 words


@pytest.mark.timeout(300)
@pytest.mark.parametrize("variant,timeout_ms", [("auto", 1), ("auto", 2000), ("tc", 2000)])
def test_long_products_of_few_samples(gpu, variant, timeout_ms):
    import torch
    X = torch.full((2, W), -1, dtype=torch.int64, device="cuda")
    X[1, 0] = 0x5
    C = torch.empty((2, 2), dtype=torch.int32, device="cuda").view(torch.uint32)
    with jsim.Context(timeout_ms=timeout_ms) as ctx:
        ctx.product(X, 2, W, W, C, variant=variant)
    b = 64 * (W - 1) + 2
    assert C.view(torch.int32).cpu().tolist() == [[64 * W, b], [b, b]]
