"""Calls in a workspace that is smaller than what they ask for first: wide
batches and the ranked ingest give way to what takes less, and the result is
the oracle's.  The allocators refuse requests on the host; no device memory is
filled up."""
import numpy as np
import pytest

import oracle
from paper_1911_04200_gb300 import jsim, synth

pytestmark = pytest.mark.gpu


class Capped:
    """Device allocator (PyTorch's caching allocator underneath) that refuses
    a request of more than `each` bytes, one of exactly `never` bytes and one
    that would bring what is live above `total` bytes; `peak` is the most that
    was live at a time."""

    def __init__(self, total=1 << 62, each=1 << 62, never=-1):
        import torch
        self.torch = torch
        self.total, self.each, self.never = total, each, never
        self.live, self.now, self.peak, self.refused = {}, 0, 0, 0

    def alloc(self, nbytes, stream):
        if nbytes > self.each or nbytes == self.never or self.now + nbytes > self.total:
            self.refused += 1
            return 0
        p = self.torch.cuda.caching_allocator_alloc(nbytes, 0, stream)
        self.live[p] = nbytes
        self.now += nbytes
        self.peak = max(self.peak, self.now)
        return p

    def free(self, ptr, nbytes, stream):
        self.now -= self.live.pop(ptr)
        self.torch.cuda.caching_allocator_delete(ptr)


def spread_sets(n, per, bits, seed, pool=None):
    """n samples of up to `per` values spread over [0, 2^bits), the smallest and
    the largest value among them; with `pool`, from that many distinct values
    (samples in groups of 32 share a part of it)."""
    rng = np.random.default_rng(seed)
    vals = np.unique(rng.integers(0, 1 << bits, pool, dtype=np.uint64)) if pool else None
    segs = []
    for i in range(n):
        if pool:
            part = vals[(i // 32) % 4::4]
            s = part[rng.random(part.size) < per / part.size]
        else:
            s = rng.integers(0, 1 << bits, per, dtype=np.uint64)
        ends = [0] if i == 0 else [(1 << bits) - 1] if i == n - 1 else []
        segs.append(np.unique(np.concatenate([s, np.array(ends, dtype=np.uint64)])))
    off = np.zeros(n + 1, dtype=np.uint64)
    off[1:] = np.cumsum([s.size for s in segs])
    return off, np.concatenate(segs)


def assert_same(res, ref):
    (C, s, J), (Co, so, Jo) = res, ref
    np.testing.assert_array_equal(s, so)
    np.testing.assert_array_equal(C.astype(np.uint64), Co)
    np.testing.assert_array_equal(J.view(np.uint64), Jo.view(np.uint64))


def needed(call, ref, **kw):
    """What the call asks for when nothing is refused."""
    a = Capped()
    with jsim.Context(allocator=a, **kw) as ctx:
        assert_same(call(ctx), ref)
    assert not a.live
    return a.peak


@pytest.mark.parametrize("filter_min", [1, 2])
def test_wide_dense_batches_give_way(gpu, filter_min):
    off, ids = spread_sets(40, 3000, 32, seed=1)
    ref = oracle.all_pairs(off, ids)
    a = Capped(each=300 << 20)  # a 2^32-row bitmap takes 512 MiB
    with jsim.Context(allocator=a, filter_min=filter_min) as ctx:
        assert_same(ctx.all_pairs(off, ids), ref)
        assert a.refused and ctx.stats()["batch_rows"] == 1 << 28
    assert not a.live


def thin_collection():
    return spread_sets(260, 2000, 32, seed=2, pool=40_000)


@pytest.mark.parametrize("filter_min", [1, 2])
def test_ranked_ingest_gives_way(gpu, filter_min):
    """The ranked ingest's own buffers are granted and a class matrix is
    refused behind them: the call goes through in what the per-value ingest
    takes."""
    off, ids = thin_collection()
    ref = oracle.all_pairs(off, ids)
    call = lambda ctx: ctx.all_pairs(off, ids)
    kw = dict(variant="sparse", filter_min=filter_min)
    ranked = needed(call, ref, **kw)
    per_value = needed(call, ref, batch_rows=1 << 28, **kw)  # (a chosen width: not ranked)
    assert per_value + (8 << 20) < ranked
    a = Capped(total=per_value + (8 << 20))
    with jsim.Context(allocator=a, **kw) as ctx:
        assert_same(call(ctx), ref)
        assert a.refused and ctx.stats()["variant"] == "sparse"
    assert not a.live


class FailOnce(Capped):
    """Refuses its k-th request."""

    def __init__(self, k):
        super().__init__()
        self.k, self.calls = k, 0

    def alloc(self, nbytes, stream):
        self.calls += 1
        return 0 if self.calls == self.k else super().alloc(nbytes, stream)


def test_any_refused_request_of_the_ranked_ingest(gpu):
    """Whichever request is refused: the result, or JSIM_ERR_OOM with the
    outputs untouched; the latter only for the input's own buffers."""
    off, ids = thin_collection()
    ref = oracle.all_pairs(off, ids)
    n = off.size - 1
    base = FailOnce(0)
    with jsim.Context(allocator=base, variant="sparse") as ctx:
        assert_same(ctx.all_pairs(off, ids), ref)
    oom = 0
    for k in range(2, base.calls + 1):  # (the first is the context's own)
        a = FailOnce(k)
        C = np.full((n, n), 7, dtype=np.uint32)
        s = np.full(n, 7, dtype=np.uint64)
        J = np.full((n, n), -1.0)
        with jsim.Context(allocator=a, variant="sparse") as ctx:
            try:
                assert_same(ctx.all_pairs(off, ids, out=(C, s, J)), ref)
            except jsim.JsimError as e:
                assert e.name == "JSIM_ERR_OOM"
                assert (C == 7).all() and (s == 7).all() and (J == -1.0).all()
                oom += 1
        assert not a.live
    assert oom <= 8


@pytest.mark.timeout(300)
def test_ranked_ingest_of_fed_input_gives_way(gpu):
    """Page-locked input copied in pieces under the batch loop."""
    import torch
    alloc = lambda count: torch.empty(count, dtype=torch.int64, pin_memory=True).numpy().view(np.uint64)
    off, ids = synth.clade1024(n=300, median=2e5, alloc=alloc)
    assert ids.nbytes >= 512 << 20
    with jsim.Context(variant="sparse", id_bits=32) as ctx:
        C, s, J = ctx.all_pairs(off, ids)
        assert ctx.stats()["h2d_pieces"] >= 3
    a = Capped(never=4 * ids.size)  # the row numbers
    with jsim.Context(allocator=a, variant="sparse", id_bits=32) as ctx:
        C2, s2, J2 = ctx.all_pairs(off, ids)
        assert a.refused == 1 and ctx.stats()["h2d_pieces"] >= 3 and ctx.stats()["variant"] == "sparse"
    assert not a.live
    assert (C == C2).all() and (s == s2).all() and (J.view(np.uint64) == J2.view(np.uint64)).all()
    np.testing.assert_array_equal(s, oracle.sizes_of(off, ids))


@pytest.mark.timeout(300)
@pytest.mark.parametrize("filter_min", [1, 2])
def test_wide_batches_of_a_batched_call_give_way(gpu, filter_min):
    """The wide lanes are granted and the last buffer behind them is refused."""
    cols = [spread_sets(n, 30_000, 32, seed=n) for n in (250, 249, 248, 247, 246, 245, 244, 40)]
    kw = dict(variant="popc", filter_min=filter_min)
    a = Capped()
    with jsim.Context(allocator=a, **kw) as ctx:
        refs = ctx.all_pairs_batched(cols)
        rounds = ctx.stats()["batches"]
    assert rounds < 8 * len(cols)  # (8 batches of 2^29 rows each)
    Co, so, Jo = oracle.all_pairs(*cols[-1])
    assert_same(refs[-1], (Co, so, Jo))
    b = Capped(total=a.peak - 1)
    with jsim.Context(allocator=b, **kw) as ctx:
        outs = ctx.all_pairs_batched(cols)
        assert b.refused and ctx.stats()["batches"] == 8 * len(cols)
    for res, ref in zip(outs, refs):
        for x, y in zip(res, ref):
            np.testing.assert_array_equal(x.view(np.uint8), y.view(np.uint8))
    assert not b.live


def test_a_captured_call_gives_its_buffers_back(gpu):
    """The buffers kept for a replay make room when another call on the context
    needs them."""
    import torch
    cols = [spread_sets(n, 30_000, 32, seed=n) for n in (120, 200)]
    dev = [(torch.from_numpy(o.view(np.int64)).cuda(), torch.from_numpy(i.view(np.int64)).cuda()) for o, i in cols]
    off, ids = spread_sets(40, 3000, 28, seed=1)  # one batch: no narrower one to give way to
    ref = oracle.all_pairs(off, ids)
    plain = needed(lambda ctx: ctx.all_pairs(off, ids), ref)
    a = Capped()
    with jsim.Context(allocator=a) as ctx:
        outs = ctx.all_pairs_batched(dev)
        kept = a.now
        assert kept > 64 << 20
        a.total = max(a.peak, plain + kept - 4096)  # (the error word is part of both)
        assert a.total < plain + kept - 256, "the two calls fit together: nothing is tested"
        assert_same(ctx.all_pairs(off, ids), ref)
        assert a.refused
        again = ctx.all_pairs_batched(dev)
        torch.cuda.synchronize()
    for (C, s, J), (C2, s2, J2) in zip(outs, again):
        assert torch.equal(C.view(torch.int32), C2.view(torch.int32)) and torch.equal(J, J2)
    assert not a.live
