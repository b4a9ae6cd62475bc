"""The calls that users of this library make, with inputs of the shapes they
make them on: plain all-pairs calls from the smallest collection to the full
clade recipe, on device, pageable and page-locked input, hashed and dense
values, both filters and count widths; the batched, streamed and serving
patterns; the product alone; and the sparse outputs of the J matrix.

Inputs follow the recipes of ``paper_1911_04200_gb300/synth`` (clade,
ancestral and Bernoulli collections), drawn here on the GPU so that a
collection of a billion values is made in seconds.
"""
import math

import numpy as np
import torch

from paper_1911_04200_gb300 import jsim

DEV = "cuda:0"
SIGMA = math.log(10.0) / 3.0  # set sizes within a decade of the median at 3 sigma


def listed():
    return [
        # The small plain call (64 samples of 50,000 values below 2^20, eight
        # ancestors): one batch, a few launches; latency decides.
        dict(name="small", kind="pairs", recipe="ancestral", n=64, groups=8, median=50_000, id_bits=20,
             mem="device", filter_min=1, count_bits=32, distance=False),
        # A ragged collection as a script hands it over: numpy arrays in, numpy
        # arrays out, hashed 32-bit values, sizes over two decades.
        dict(name="ragged_host", kind="pairs", recipe="clade", n=517, groups=17, median=20_000, id_bits=32,
             mem="host", filter_min=1, count_bits=32, distance=False),
        # The full clade recipe on device-resident input (1.3e9 values).
        dict(name="clade1024", kind="pairs", recipe="clade", n=1024, groups=32, median=1_000_000, id_bits=32,
             mem="device", filter_min=1, count_bits=32, distance=False),
        # The same recipe from page-locked host memory to host outputs, at a
        # seventh of its set sizes: the end-to-end call.
        dict(name="clade_pinned", kind="pairs", recipe="clade", n=1024, groups=32, median=150_000, id_bits=32,
             mem="pinned", filter_min=1, count_bits=32, distance=False),
        # The paper's synthetic indicator matrix (density 0.01) with 4000
        # samples: no structure to skip, the dense product carries it.
        dict(name="bernoulli", kind="pairs", recipe="bernoulli", n=4000, m=1 << 22, p=0.01,
             mem="device", filter_min=1, count_bits=32, distance=False),
        # A thin matrix (density 0.001) with the options: rows of two or more
        # samples only, 64-bit counts, distances instead of similarities.
        dict(name="thin_options", kind="pairs", recipe="bernoulli", n=1000, m=30_000_000, p=0.001,
             mem="device", filter_min=2, count_bits=64, distance=True),
        # Twenty independent collections of 8 to 512 samples in one call.
        dict(name="batched", kind="batched", k=20, n_lo=8, n_hi=512, median=20_000, id_bits=32),
        # Many samples from pageable host memory through the pinned staging.
        dict(name="streamed", kind="streamed", n=4096, groups=64, median=20_000, id_bits=34,
             staging=1 << 28, count_bits=64),
        # Serving, one request of one sample: the latency a lone query sees.
        dict(name="serve_one", kind="serve", n_ref=2048, ref_median=20_000, requests=1, q_lo=1, q_hi=1,
             q_median=100_000),
        # Serving, a burst of 20 requests of 1 to 64 samples: its throughput.
        dict(name="serve_burst", kind="serve", n_ref=2048, ref_median=20_000, requests=20, q_lo=1, q_hi=64,
             q_median=20_000),
        # The semiring product alone on packed words (the step-level call).
        dict(name="product", kind="product", n=1000, W=40_001, stride=40_002),
        # What users take from J: ten nearest neighbours and the pairs above a
        # threshold, up to a bound on their number.
        dict(name="sparse_outputs", kind="outputs", n=4096, k=10, tau=0.15, cap=8192),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["clade", "clade", "clade", "bernoulli", "bernoulli", "ancestral", "batched", "streamed",
                       "serve", "product", "outputs"])
    opts = dict(filter_min=rng.choice([1, 1, 2]), count_bits=rng.choice([32, 32, 64]),
                distance=rng.choice([False, False, True]))
    if kind == "clade":
        n = _log_int(rng, 16, 2048)
        # at most 5e8 values (a log-normal size averages 1.34 medians)
        median = _log_int(rng, 1000, min(1_000_000, 350_000_000 // n))
        return dict(kind="pairs", recipe="clade", n=n, groups=max(1, n // 32), median=median,
                    id_bits=rng.randint(max(22, median.bit_length() + 4), 33),
                    mem=rng.choice(["device", "device", "host", "pinned"] if n * median < 60_000_000
                                   else ["device", "device", "pinned"]), **opts)
    if kind == "ancestral":
        return dict(kind="pairs", recipe="ancestral", n=rng.randint(5, 200), groups=rng.randint(2, 16),
                    median=_log_int(rng, 500, 60_000), id_bits=rng.randint(17, 24),
                    mem=rng.choice(["device", "host"]), **opts)
    if kind == "bernoulli":
        n = _log_int(rng, 100, 4000)
        p = math.exp(rng.uniform(math.log(1e-3), math.log(5e-2)))
        m = _log_int(rng, 1 << 18, min(1 << 24, int(2e8 / (n * p))) if n * p * (1 << 18) < 2e8 else (1 << 18) + 1)
        return dict(kind="pairs", recipe="bernoulli", n=n, m=m, p=p, mem="device", **opts)
    if kind == "batched":
        lo = rng.randint(4, 100)
        return dict(kind="batched", k=rng.randint(2, 20), n_lo=lo, n_hi=lo + _log_int(rng, 10, 400),
                    median=_log_int(rng, 1000, 40_000), id_bits=rng.randint(24, 32))
    if kind == "streamed":
        n = _log_int(rng, 200, 4096)
        return dict(kind="streamed", n=n, groups=max(1, n // 64), median=_log_int(rng, 2000, 80_000_000 // n),
                    id_bits=rng.randint(26, 34), staging=rng.choice([1 << 26, 1 << 27, 1 << 28]),
                    count_bits=rng.choice([32, 64]))
    if kind == "serve":
        q_lo = rng.randint(1, 20)
        return dict(kind="serve", n_ref=rng.randint(100, 2048), ref_median=_log_int(rng, 2000, 20_000),
                    requests=rng.randint(1, 20), q_lo=q_lo, q_hi=rng.randint(q_lo, 64),
                    q_median=_log_int(rng, 2000, 50_000))
    if kind == "product":
        n, W = _log_int(rng, 30, 3000), _log_int(rng, 200, 60_000)
        return dict(kind="product", n=n, W=W, stride=W + rng.randint(0, 20))
    n = _log_int(rng, 100, 6000)
    return dict(kind="outputs", n=n, k=rng.randint(1, 32), tau=rng.uniform(0.1, 0.2), cap=rng.randint(1, 2 * n))


# --------------------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _sizes(n, median, seed):
    r = np.random.RandomState(seed % (1 << 32))
    s = median * np.exp(SIGMA * r.standard_normal(n))
    return np.clip(s, median / 10, median * 10).astype(np.int64).clip(1)


def _sorted_sets(parts, bits):
    """(offsets, ids): per sample sorted distinct values, from value tensors
    whose upper bits (above `bits`) number the sample within its part."""
    counts, ids = [], []
    for key, n in parts:
        key = torch.unique_consecutive(torch.sort(key).values)
        edge = torch.arange(n + 1, device=DEV, dtype=torch.int64) << bits
        counts.append(torch.searchsorted(key, edge).diff())
        ids.append(key & ((1 << bits) - 1))
    off = torch.zeros(sum(c.numel() for c in counts) + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(torch.cat(counts), 0)
    return off, torch.cat(ids)


def _clade(n, groups, median, id_bits, seed, first=0, stream_seed=None, sizes=None):
    """Samples of `groups` clades: 30 % of a clade's values are shared by all
    clades, and every sample replaces 0 to 40 % of its own by fresh ones."""
    g = _gen(seed)
    size = _sizes(n, median, seed) if sizes is None else sizes
    sg = _gen(seed if stream_seed is None else stream_seed)
    L = int(max(size.max(), 10 * median if stream_seed is not None else 1))
    root = torch.randint(0, 1 << id_bits, (L,), generator=sg, device=DEV)
    stream = torch.randint(0, 1 << id_bits, (groups, L), generator=sg, device=DEV)
    for c in range(groups):
        core = torch.rand(L, generator=sg, device=DEV) < 0.3
        stream[c] = torch.where(core, root, stream[c])
    sub = np.random.RandomState((seed + 1) % (1 << 32)).uniform(0, 0.4, n)
    step = max(1, min(n, int(1.2e8 // max(1, size.mean()))))

    def parts():
        for a in range(0, n, step):
            b = min(n, a + step)
            ln = torch.from_numpy(size[a:b]).to(DEV)
            who = torch.repeat_interleave(torch.arange(b - a, device=DEV), ln)
            t = torch.arange(who.numel(), device=DEV) - (torch.cumsum(ln, 0) - ln)[who]
            v = stream.view(-1)[((who + a + first) % groups) * L + t]
            fresh = torch.rand(v.numel(), generator=g, device=DEV) < torch.from_numpy(sub[a:b]).to(DEV, torch.float32)[who]
            v = torch.where(fresh, torch.randint(0, 1 << id_bits, v.shape, generator=g, device=DEV), v)
            yield (who << id_bits) | v, b - a

    return _sorted_sets(parts(), id_bits)


def _ancestral(n, groups, size, id_bits, seed):
    g = _gen(seed)
    anc = torch.randint(0, 1 << id_bits, (groups, size), generator=g, device=DEV)
    u = torch.rand(n, 1, generator=g, device=DEV) * 0.6
    v = anc[torch.arange(n, device=DEV) % groups]
    v = torch.where(torch.rand(n, size, generator=g, device=DEV) < u,
                    torch.randint(0, 1 << id_bits, (n, size), generator=g, device=DEV), v)
    key = (torch.arange(n, device=DEV)[:, None] << id_bits) | v
    return _sorted_sets([(key.reshape(-1), n)], id_bits)


def _bernoulli(n, m, p, seed):
    """Every value of [0, m) in every sample with probability p: m p values
    (plus binomial noise) drawn uniformly, repeats dropped."""
    g = _gen(seed)
    bits = max(1, (m - 1).bit_length())
    r = np.random.RandomState(seed % (1 << 32))
    size = np.maximum(1, (-m * math.log1p(-p) + math.sqrt(m * p * (1 - p)) * r.standard_normal(n))).astype(np.int64)

    def parts():
        step = max(1, int(1.2e8 // size.mean()))
        for a in range(0, n, step):
            b = min(n, a + step)
            who = torch.repeat_interleave(torch.arange(b - a, device=DEV), torch.from_numpy(size[a:b]).to(DEV))
            yield (who << bits) | torch.randint(0, m, who.shape, generator=g, device=DEV), b - a

    return _sorted_sets(parts(), bits)


def _pairs_input(case, seed):
    if case["recipe"] == "clade":
        return _clade(case["n"], case["groups"], case["median"], case["id_bits"], seed)
    if case["recipe"] == "ancestral":
        return _ancestral(case["n"], case["groups"], case["median"], case["id_bits"], seed)
    return _bernoulli(case["n"], case["m"], case["p"], seed)


def _host(off, ids):
    return off.cpu().numpy().view(np.uint64), ids.cpu().numpy().view(np.uint64)


def _pinned(off, ids):
    buf = torch.empty(ids.numel(), dtype=torch.int64, pin_memory=True)
    buf.copy_(ids)
    return off.cpu().numpy().view(np.uint64), buf.numpy().view(np.uint64), buf


def _batched_sizes(case):
    r = np.random.RandomState(case["k"] * 7919 + case["n_lo"])
    return [int(x) for x in r.randint(case["n_lo"], case["n_hi"] + 1, case["k"])]


def _request_sizes(case):
    r = np.random.RandomState(case["requests"] * 104729 + case["q_lo"])
    return [int(x) for x in r.randint(case["q_lo"], case["q_hi"] + 1, case["requests"])]


def _words(case, seed):
    g = _gen(seed)
    shape = (case["n"], case["stride"])
    w = None
    for _ in range(3):  # every bit set with probability 1/8
        r = torch.randint(-(1 << 63), (1 << 63) - 1, shape, generator=g, device=DEV)
        w = r if w is None else w & r
    return w


def _similarity(case, seed):
    """A J matrix as the all-pairs call writes it: quotients of counts, high
    within a clade of 32 samples, low between clades."""
    n, g = case["n"], _gen(seed)
    size = torch.from_numpy(_sizes(n, 100_000, seed)).to(DEV).double()
    clade = torch.arange(n, device=DEV) % max(1, n // 32)
    share = torch.rand(n, n, generator=g, device=DEV, dtype=torch.float64) * 0.3 + 0.5
    share = torch.where(clade[:, None] == clade[None, :], share, share * 0.1)
    c = torch.floor(torch.minimum(size[:, None], size[None, :]) * share)
    c = torch.triu(c, 1)
    c = c + c.T + torch.diag(size)
    return c / (size[:, None] + size[None, :] - c)


def prepare(case, seed):
    kind = case["kind"]
    state = dict(kind=kind, case=case)
    if kind == "pairs":
        off, ids = _pairs_input(case, seed)
        if case["mem"] == "host":
            off, ids = _host(off, ids)
        elif case["mem"] == "pinned":
            off, ids, state["pinned"] = _pinned(off, ids)
        state.update(off=off, ids=ids, ctx=jsim.Context(filter_min=case["filter_min"], count_bits=case["count_bits"],
                                                        distance=case["distance"]))
    elif kind == "batched":
        state["cols"] = [_clade(n, (n + 31) // 32, case["median"], case["id_bits"], seed * 64 + k)
                         for k, n in enumerate(_batched_sizes(case))]
        state["ctx"] = jsim.Context()
    elif kind == "streamed":
        state["off"], state["ids"] = _host(*_clade(case["n"], case["groups"], case["median"], case["id_bits"], seed))
        state["ctx"] = jsim.Context(count_bits=case["count_bits"])
    elif kind == "serve":
        groups = max(1, case["n_ref"] // 32)
        ref = _clade(case["n_ref"], groups, case["ref_median"], 32, seed, stream_seed=seed + 11)
        state["ctx"] = jsim.Context()
        state["index"] = jsim.Index(state["ctx"], *ref, max_batch_values=1 << 25)
        state["queries"], first = [], case["n_ref"]
        for k, q in enumerate(_request_sizes(case)):
            size = np.minimum(_sizes(q, case["q_median"], seed * 64 + k), 10 * case["ref_median"])
            state["queries"].append(_host(*_clade(q, groups, case["ref_median"], 32, seed * 64 + k, first=first,
                                                  stream_seed=seed + 11, sizes=size)))
            first += q
    elif kind == "product":
        state["words"] = _words(case, seed)
        state["C"] = torch.empty((case["n"], case["n"]), dtype=torch.uint32, device=DEV)
        state["ctx"] = jsim.Context()
    else:
        state["J"] = _similarity(case, seed)
        state["ctx"] = jsim.Context()
    return state


# --------------------------------------------------------------------------- one pass

def _signed(x):
    """Unsigned results under a signed type of the same bits (no copy): few
    torch operations take unsigned tensors, so users look at them this way."""
    if isinstance(x, (list, tuple)):
        return [_signed(v) for v in x]
    if isinstance(x, np.ndarray) and x.dtype.kind == "u":
        return x.view(np.dtype("i%d" % x.dtype.itemsize))
    if isinstance(x, torch.Tensor) and x.dtype in (torch.uint32, torch.uint64):
        return x.view(torch.int32 if x.dtype == torch.uint32 else torch.int64)
    return x


def run(state):
    return _signed(_run(state))


def _run(state):
    kind, case, ctx = state["kind"], state["case"], state["ctx"]
    if kind == "pairs":
        return ctx.all_pairs(state["off"], state["ids"])
    if kind == "batched":
        return ctx.all_pairs_batched(state["cols"])
    if kind == "streamed":
        return ctx.all_pairs_streamed(state["off"], state["ids"], staging_bytes=case["staging"])
    if kind == "serve":
        requests = [state["index"].submit(*q) for q in state["queries"]]
        out = [r.wait() for r in requests]
        for r in requests:
            r.free()
        return out
    if kind == "product":
        return ctx.product(state["words"], case["n"], case["W"], case["stride"], state["C"])
    idx, val = ctx.topk(state["J"], case["k"])
    pi, pj, pv, count = ctx.threshold(state["J"], case["tau"], cap=case["cap"])
    return idx, val, pi, pj, pv, count


# --------------------------------------------------------------------------- what a pass cannot do without

def _mean_values(case):
    if case.get("recipe") == "bernoulli":
        return case["n"] * case["m"] * case["p"]
    if case.get("recipe") == "ancestral":
        return case["n"] * case["median"]
    return 1.3 * case["n"] * case["median"]


def work(case):
    """Bytes: every value read once, every output written once.  Operations:
    an AND and an add per bit and pair of samples where the rows are dense
    (Bernoulli matrices and the product alone); for the sparse recipes, whose
    rows a few samples share, one AND and one add per pair of samples sharing a
    value (a clade's 32 samples or so)."""
    kind = case["kind"]
    if kind in ("pairs", "streamed"):
        n, N = case["n"], _mean_values(case)
        cb = case["count_bits"] // 8
        if case.get("recipe") == "bernoulli":
            flops = case["m"] * n * (n + 1.0)
        else:
            flops = N * max(1.0, n / case["groups"])
        return dict(bytes=8 * N + n * n * (cb + 8) + 8 * n, flops=flops)
    if kind == "batched":
        ns = _batched_sizes(case)
        N = 1.3 * case["median"] * sum(ns)
        return dict(bytes=8 * N + 12 * sum(n * n for n in ns) + 8 * sum(ns), flops=32 * N)
    if kind == "serve":
        q, n = sum(_request_sizes(case)), case["n_ref"]
        N = 1.3 * q * min(case["q_median"], 10 * case["ref_median"])
        # two thirds of a query's values are in the reference: one row of n bits each
        return dict(bytes=8 * N + N * 0.67 * n / 8 + 12 * q * n, flops=N * 0.67 * n)
    if kind == "product":
        n, W = case["n"], case["W"]
        return dict(bytes=8 * n * W + 4 * n * n, flops=64.0 * W * n * (n + 1))
    n = case["n"]
    return dict(bytes=2 * 8 * n * n + 16 * n * case["k"], flops=n * (n + 1.0))


# --------------------------------------------------------------------------- the same in plain torch

def _counts(rows, cols, n, m, step=1 << 21):
    """A^T A of the 0/1 matrix with ones at (rows, cols), rows ascending:
    single-precision products of at most 2^21 rows (every sum an integer below
    2^24, so exact) added up in 64 bits."""
    torch.backends.cuda.matmul.allow_tf32 = False
    step = max(1, min(step, (1 << 30) // max(1, n)))
    C = torch.zeros(n, n, dtype=torch.float64, device=DEV)
    for a in range(0, m, step):
        lo, hi = torch.searchsorted(rows, torch.tensor([a, min(m, a + step)], device=DEV)).tolist()
        if lo == hi:
            continue
        A = torch.zeros(n, min(m, a + step) - a, device=DEV)
        A[cols[lo:hi], rows[lo:hi] - a] = 1.0
        C += (A @ A.T).double()
    return C


def _exact_pairs(off, ids, distance=False):
    n = off.numel() - 1
    who = torch.repeat_interleave(torch.arange(n, device=DEV), off.diff())
    ids, order = torch.sort(ids)
    row = torch.cumsum(torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), (ids[1:] != ids[:-1]).long()]), 0)
    C = _counts(row, who[order], n, int(row[-1]) + 1)
    size = off.diff().double()
    J = C / (size[:, None] + size[None, :] - C)
    return C.long(), off.diff(), 1.0 - J if distance else J


def exact(case, seed):
    kind = case["kind"]
    if kind == "pairs":
        if _mean_values(case) * case["n"] > 2e11:
            return None
        C, s, J = _exact_pairs(*_pairs_input(case, seed), distance=case["distance"])
        return (C, s, J) if case["mem"] == "device" else (C.cpu().numpy(), s.cpu().numpy(), J.cpu().numpy())
    if kind == "product":
        n, W = case["n"], case["W"]
        if 64 * W * n * n > 1e13:
            return None
        words, C = _words(case, seed), torch.zeros(n, n, dtype=torch.float64, device=DEV)
        bit = torch.arange(64, device=DEV)
        for a in range(0, W, 2048):
            A = ((words[:, a:min(W, a + 2048), None] >> bit) & 1).reshape(n, -1).float()
            C += (A @ A.T).double()
        return C.long()
    if kind == "outputs":
        J = _similarity(case, seed)
        n = case["n"]
        P = J.clone()
        P.fill_diagonal_(-1.0)
        val, idx = torch.sort(P, dim=1, descending=True, stable=True)
        pairs = torch.nonzero(torch.triu(J >= case["tau"], 1))
        count, k = pairs.shape[0], case["k"]
        i, j = pairs[:case["cap"]].T.contiguous()
        return idx[:, :k].contiguous(), val[:, :k].contiguous(), i, j, J[i, j], count
    return None
