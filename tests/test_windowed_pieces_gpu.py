"""The windowed ingest's flat lists at their edges: values at every offset
from a 32-byte boundary (the first and last pieces of ids read value by
value), segments of no, one and a few values, one sample filling whole
windows, words of more samples than are gathered at a time, and a segment
listed in more than one round.  Counts are integers and J their correctly
rounded quotient, so every comparison with the oracle is exact."""
import numpy as np
import pytest

import oracle
from paper_1911_04200_gb300 import jsim

pytestmark = pytest.mark.gpu


def collection(segs):
    off = np.zeros(len(segs) + 1, dtype=np.uint64)
    off[1:] = np.cumsum([x.size for x in segs])
    return off, np.concatenate(segs).astype(np.uint64)


def check_device(off, ids, shift, filter_min=1):
    import torch
    buf = torch.zeros(ids.size + 4, dtype=torch.int64, device="cuda")
    base = (-(buf.data_ptr() // 8)) % 4  # to a 32-byte boundary
    view = buf[(base + shift) % 4:][:ids.size]
    view.copy_(torch.from_numpy(ids.view(np.int64)))
    d_off = torch.from_numpy(off.view(np.int64)).cuda()
    with jsim.Context(variant="sparse", id_bits=22, filter_min=filter_min) as ctx:
        C, s, J = ctx.all_pairs(d_off, view)
        assert ctx.stats()["windows"] > 0
        torch.cuda.synchronize()
    Co, so, Jo = oracle.all_pairs(off, ids)
    np.testing.assert_array_equal(s.view(torch.int64).cpu().numpy().view(np.uint64), so)
    np.testing.assert_array_equal(C.view(torch.int32).cpu().numpy().view(np.uint32), Co.astype(np.uint32))
    np.testing.assert_array_equal(J.cpu().numpy().view(np.uint64), Jo.view(np.uint64))


@pytest.mark.parametrize("filter_min", [1, 2])
@pytest.mark.parametrize("shift", [0, 1, 2, 3])
def test_alignment_and_short_segments(gpu, shift, filter_min):
    rng = np.random.default_rng(70 + shift)
    segs = []
    for k in range(150):
        m = int(rng.choice([0, 1, 2, 3, 4, 5, 9, 60, 3000]))
        v = np.unique(rng.integers(0, 1 << 22, m))
        segs.append(np.sort(np.concatenate([v, np.array([k % 5, (1 << 22) - 1 - k % 3])[:m % 3]])))
    off, ids = collection(segs)
    check_device(off, ids, shift, filter_min)


@pytest.mark.parametrize("filter_min", [1, 2])
def test_full_windows_gather_few_samples_at_a_time(gpu, filter_min):
    rng = np.random.default_rng(80)
    full = np.arange(1 << 18, (1 << 18) + (1 << 17))
    segs = [full, full[::2]] + [np.unique(rng.integers(0, 1 << 20, 6000)) for _ in range(140)] + [full[1::2]]
    off, ids = collection(segs)
    check_device(off, ids, 1, filter_min)


@pytest.mark.parametrize("filter_min", [1, 2])
def test_segment_of_more_than_one_round(gpu, filter_min):
    # 2^24 + 5 copies of one value before the window's others: a list holds 2^24 of a segment
    rng = np.random.default_rng(90)
    long = np.concatenate([np.full((1 << 24) + 5, 77), np.arange(78, 5000, 7), np.arange(200_000, 300_000, 11)])
    segs = [np.unique(rng.integers(0, 1 << 20, 3000)) for _ in range(5)] + [long, np.array([77, 5000])]
    off, ids = collection(segs)
    check_device(off, ids, 3, filter_min)
