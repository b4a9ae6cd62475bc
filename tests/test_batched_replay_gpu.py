"""A batched call that replays a captured graph reads the device error word:
when a bounded wait of its product runs out, it reports JSIM_ERR_TIMEOUT and
writes no output, as the first call does.

Both calls see the same collection buffers.  The first call's values are the
same few in every sample, so its product takes a few stages; the second call's
are all distinct, so every accumulator segment of its product takes several
milliseconds and the epilogue's 1 ms wait for the first one runs out (bounded
waits: the kernel drains, returns and raises its error word)."""
import ctypes

import numpy as np
import pytest

from paper_1911_04200_gb300 import jsim

pytestmark = pytest.mark.gpu

N_SAMPLES, PER = 1000, 12_000  # 1.2e7 distinct values: 46,875 stages x 36 tiles


def call(ctx, off, ids, C, sizes, J):
    s, keep, _ = ctx._sets(off, ids)
    ptr = lambda t: (ctypes.c_void_p * 1)(t.data_ptr())
    ctx._order()
    return ctx._lib.jsim_all_pairs_batched(ctx._h, ctypes.byref(s), 1, ptr(C), ptr(sizes), ptr(J), jsim.MEM_DEVICE)


def code(name):
    return next(k for k, v in jsim.ERRORS.items() if v == name)


@pytest.mark.timeout(300)
def test_replay_reports_a_wait_that_ran_out(gpu):
    import torch
    n = N_SAMPLES
    top = n * PER  # both inputs hold 0 and `top`, so the second call replays the first one's plan
    off = torch.arange(n + 1, dtype=torch.int64, device="cuda") * PER
    same = torch.arange(PER, dtype=torch.int64, device="cuda").repeat(n)
    same[-1] = top
    spread = torch.arange(n * PER, dtype=torch.int64, device="cuda")
    spread[-1] = top
    ids = same.clone()
    C = torch.empty((n, n), dtype=torch.int32, device="cuda")
    sizes = torch.empty(n, dtype=torch.int64, device="cuda")
    J = torch.empty((n, n), dtype=torch.float64, device="cuda")
    expect = torch.full((n, n), PER, dtype=torch.int32, device="cuda")
    expect[-1, :-1] = expect[:-1, -1] = PER - 1
    with jsim.Context(variant="tc", timeout_ms=1) as ctx:
        assert call(ctx, off, ids, C, sizes, J) == 0
        assert torch.equal(C, expect)
        for t in (C, sizes):
            t.fill_(0x5A5A5A5A)
        J.fill_(-1.0)
        ids.copy_(spread)
        assert call(ctx, off, ids, C, sizes, J) == code("JSIM_ERR_TIMEOUT")
        torch.cuda.synchronize()
        assert bool((C == 0x5A5A5A5A).all()) and bool((sizes == 0x5A5A5A5A).all()) and bool((J == -1.0).all())
        # the context keeps working
        ids.copy_(same)
        assert call(ctx, off, ids, C, sizes, J) == 0
        assert torch.equal(C, expect) and bool((sizes == PER).all())
