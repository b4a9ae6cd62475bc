"""The 4-bit products of a batched call: more small collections than one launch
takes and one of several tiles, word counts read on the device, against the
oracle; and the tuner's choice of them when a later call's packed matrices are
not 16-byte aligned (an allocator need not align further than 8 bytes)."""
import numpy as np
import pytest

import oracle
from paper_1911_04200_gb300 import jsim

pytestmark = pytest.mark.gpu


class Shifting:
    """PyTorch's caching allocator; requests of `size` bytes come back 8 bytes
    past a 16-byte boundary."""

    def __init__(self):
        import torch
        self.torch = torch
        self.sizes, self.size, self.shifted, self.base = [], 0, 0, {}

    def alloc(self, nbytes, stream):
        self.sizes.append(nbytes)
        shift = 8 if nbytes == self.size else 0
        p = self.torch.cuda.caching_allocator_alloc(nbytes + shift, 0, stream)
        self.shifted += shift != 0
        self.base[p + shift] = p
        return p + shift

    def free(self, ptr, nbytes, stream):
        self.torch.cuda.caching_allocator_delete(self.base.pop(ptr))


def dense_collection(n, per, seed):
    rng = np.random.default_rng(seed)
    segs = [np.unique(rng.integers(0, 1 << 20, per, dtype=np.uint64)) for _ in range(n)]
    off = np.zeros(n + 1, dtype=np.uint64)
    off[1:] = np.cumsum([s.size for s in segs])
    return off, np.concatenate(segs)


@pytest.mark.timeout(300)
@pytest.mark.parametrize("count_bits", [32, 64])
def test_tuned_choice_with_unaligned_matrices(gpu, count_bits):
    import torch
    sizes = [128] * 15 + [1, 2, 127, 129, 200]
    cols = [dense_collection(n, 6000, seed) for seed, n in enumerate(sizes)]
    refs = [oracle.all_pairs(o, i) for o, i in cols]

    def check(outs):
        for (C, s, J), (Co, so, Jo) in zip(outs, refs):
            np.testing.assert_array_equal(s, so)
            np.testing.assert_array_equal(C.astype(np.uint64), Co)
            np.testing.assert_array_equal(J.view(np.uint64), Jo.view(np.uint64))

    a = Shifting()
    with jsim.Context(allocator=a, count_bits=count_bits) as ctx:
        for n in (64, 300):  # the kernels loaded: the tuner times them, not their loading
            X = torch.zeros((n, 64), dtype=torch.int64, device="cuda")
            ctx.product(X, n, 64, 64)
        a.sizes.clear()
        check(ctx.all_pairs_batched(cols))
        first = ctx.stats()["variant"]
        a.size = max(a.sizes)  # the packed matrices
        check(ctx.all_pairs_batched(cols))
        assert a.shifted == 1 and ctx.stats()["variant"] != "tc2"
        a.size = 0
        check(ctx.all_pairs_batched(cols))
        assert ctx.stats()["variant"] == first
    assert not a.base
    if first != "tc2":
        pytest.skip("the tuner did not take the 4-bit products here")
