// Ingest kernels: per-batch plan, input validation, the zero-row filter
// f^(l) (Eq. 5), its prefix sum p^(l) as a rank directory (Eq. 6), and the
// bitmask compression of the surviving rows into 64-bit words (Sec. III-B).
#include "ingest_dev.cuh"

namespace jsim {

namespace {

// Every sample's first value at or above lo and at or above hi (hi == 0: its
// end) into the plan, and the smallest value after the batch into *s_next.
// G lanes search one sample: a step probes G places of each of its two ranges,
// and a thread has U samples under way, so the chain of dependent loads is
// short: 50,000 values take 4 steps for 64 samples (G = 16), 16 for 1024
// (G = 1), where a bisection per end takes 32.  (On unsorted values, any place
// of the range.)
template <int U>
__device__ __forceinline__ void plan_search(const u64* __restrict__ offsets, const u64* __restrict__ ids, u64 n, u64 lo,
                                            u64 hi, const Plan& plan, const u32* __restrict__ perm,
                                            const u64* __restrict__ ends, u32 G, u64* s_next, int* s_has_next)
{
    const u32 lane = threadIdx.x & 31, gl = lane & (G - 1), g0 = lane - gl;
    const u32 gmask = G == 32 ? 0xffffffffu : (1u << G) - 1u;
    const u64 groups = kPlanThreads / G, group = threadIdx.x / G;
    for (u64 j0 = 0; j0 < n; j0 += (u64)U * groups) {
        u64 end[U], a[2 * U], b[2 * U];  // a, b: what is left of each range
        #pragma unroll
        for (int u = 0; u < U; ++u) {
            const u64 j = j0 + (u64)u * groups + group;
            end[u] = a[2 * u] = 0;
            if (j < n) {
                const u64 sj = perm ? (u64)perm[j] : j;
                a[2 * u] = offsets[sj];
                end[u] = ends ? ends[sj] : offsets[sj + 1];
            }
            a[2 * u + 1] = hi ? a[2 * u] : end[u];
            b[2 * u] = b[2 * u + 1] = end[u];
        }
        // (every step at least halves what is left of a range)
        for (int round = 0; round < 65; ++round) {
            bool left = false;
            #pragma unroll
            for (int k = 0; k < 2 * U; ++k) left = left || a[k] < b[k];
            if (!__any_sync(0xffffffffu, left)) break;
            u64 x[2 * U], step[2 * U];
            bool in[2 * U];
            #pragma unroll
            for (int k = 0; k < 2 * U; ++k) {
                const u64 len = b[k] - a[k];
                step[k] = len <= G ? 1 : (len >> 32) ? len / (G + 1) + 1 : (u64)((u32)len / (G + 1)) + 1;
                const u64 p = a[k] + (gl + 1) * step[k] - 1;
                in[k] = p < b[k];
                x[k] = in[k] ? ids[p] : 0ull;
            }
            #pragma unroll
            for (int k = 0; k < 2 * U; ++k) {
                const u32 m = __ballot_sync(0xffffffffu, in[k] && x[k] < ((k & 1) ? hi : lo));
                const u32 below = (u32)__popc((m >> g0) & gmask);
                a[k] += below * step[k];
                const u64 top = a[k] + step[k] - 1;  // the first probe not below
                if (below < G && top < b[k]) b[k] = top;
            }
        }
        #pragma unroll
        for (int u = 0; u < U; ++u) {
            const u64 j = j0 + (u64)u * groups + group;
            if (j >= n || gl != 0) continue;
            const u64 q = max(a[2 * u], a[2 * u + 1]);
            plan.beg[j] = a[2 * u];
            plan.len[j] = q - a[2 * u];
            if (q < end[u]) {
                atomicMin((unsigned long long*)s_next, (unsigned long long)ids[q]);
                *s_has_next = 1;
            }
        }
    }
}

// kProbes values (null: none).
__device__ __forceinline__ void take_probes(const u64* __restrict__ ids, u64 N, u64* probes)
{
    static_assert(kProbes <= kPlanThreads, "a probe a thread");
    if (probes && threadIdx.x < kProbes) probes[threadIdx.x] = ids[probe_place(threadIdx.x, N)];
}

// One CTA: per-sample [beg, beg+len) of values in [lo, hi) and chunk prefix.
// With perm, entry i of the plan is sample perm[i] (the ingest kernels then
// walk the samples in that order).  With ends, sample i is searched in
// [offsets[i], ends[i]) only.  Bound by the searches' dependent loads: 64
// samples of 50,000 values 24.6 us by bisection, 9 us here.
__global__ void __launch_bounds__(kPlanThreads)
k_plan(const u64* __restrict__ offsets, const u64* __restrict__ ids, u64 n, u64 lo, u64 hi,
       int full, Plan plan, const u32* __restrict__ perm, const u64* __restrict__ ends, u64* probes, u64 N)
{
    take_probes(ids, N, probes);
    __shared__ u64 sm[kPlanThreads / 32];
    __shared__ u64 s_next;
    __shared__ int s_has_next;
    if (threadIdx.x == 0) { s_next = ~0ull; s_has_next = 0; }
    __syncthreads();
    if (!full) {
        u32 G = 1;
        while (G < 32 && 2 * (u64)G * n <= kPlanThreads) G *= 2;
        if (n <= kPlanThreads)
            plan_search<1>(offsets, ids, n, lo, hi, plan, perm, ends, G, &s_next, &s_has_next);
        else
            plan_search<2>(offsets, ids, n, lo, hi, plan, perm, ends, G, &s_next, &s_has_next);
        __syncthreads();
    }
    u64 carry = 0, total_len = 0;
    for (u64 base = 0; base < n; base += kPlanThreads) {
        const u64 i = base + threadIdx.x;
        u64 l = 0;
        if (i < n) {
            if (full) {
                const u64 si = perm ? (u64)perm[i] : i;
                const u64 s = offsets[si];
                l = (ends ? ends[si] : offsets[si + 1]) - s;
                plan.beg[i] = s;
                plan.len[i] = l;
            } else {
                l = plan.len[i];
            }
        }
        const u64 nch = (l + kChunk - 1) / kChunk;
        u64 ex;
        u64 tot = block_exclusive_scan<kPlanThreads>(nch, ex, sm);
        if (i < n) plan.cofs[i] = carry + ex;
        carry += tot;
        u64 ex2;
        total_len += block_exclusive_scan<kPlanThreads>(l, ex2, sm);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        plan.cofs[n] = carry;
        plan.totals[0] = total_len;
        plan.totals[1] = carry;
        plan.totals[2] = s_next;
        plan.totals[3] = (u64)s_has_next;
        for (u64 k = 4; k < kPlanTotals; ++k) plan.totals[k] = 0;  // chunk tickets
    }
}

constexpr int kValidateDepth = 4;  // values a thread loads per step

__global__ void __launch_bounds__(kIngestThreads)
k_validate(const u64* __restrict__ offsets, const u64* __restrict__ ids, u64 n, Plan plan,
           int id_bits, u64* sizes, u32* err, u64* maxid, u64* minid, u64 err_stride)
{
    __shared__ ChunkDesc s_d[2];
    __shared__ u32 s_cnt[kIngestThreads / 32];
    const u64 nch = plan.totals[1];
    if (threadIdx.x == 0) fetch_chunk(plan, n, nch, kTicketValidate, s_d[0]);
    __syncthreads();
    for (int db = 0;; db ^= 1) {
        const ChunkDesc d = s_d[db];
        if (d.c >= nch) break;
        if (threadIdx.x == 0) fetch_chunk(plan, n, nch, kTicketValidate, s_d[db ^ 1]);
        const u64 i = d.i, p0 = d.p0, p1 = d.p1;
        const u64 sb = offsets[i], se = offsets[i + 1];
        u32 cnt = 0, flags = 0;
        // kValidateDepth coalesced loads a thread in flight per step; a
        // value's predecessor comes from the lane before it (lane 0 loads
        // its own, ahead, with the values)
        const int lane = threadIdx.x & 31;
        for (u64 base = p0; base < p1; base += kValidateDepth * kIngestThreads) {
            u64 x[kValidateDepth], pv[kValidateDepth];
            #pragma unroll
            for (int k = 0; k < kValidateDepth; ++k) {
                const u64 pos = base + (u64)(k * kIngestThreads) + threadIdx.x;
                x[k] = pos < p1 ? ids[pos] : 0ull;
                pv[k] = (lane == 0 && pos < p1 && pos > sb) ? ids[pos - 1] : 0ull;
            }
            #pragma unroll
            for (int k = 0; k < kValidateDepth; ++k) {
                const u64 pos = base + (u64)(k * kIngestThreads) + threadIdx.x;
                const u64 up = __shfl_up_sync(0xffffffffu, x[k], 1);
                if (pos >= p1) continue;
                const u64 v = x[k];
                if (pos > sb) {
                    const u64 prev = lane ? up : pv[k];
                    if (v < prev) flags |= kFlagUnsorted;
                    cnt += (v != prev);
                } else {
                    cnt += 1;
                    atomicMin(minid, v);
                }
                if (id_bits < 64 && (v >> id_bits) != 0) flags |= kFlagIdRange;
                if (pos + 1 == se) atomicMax(maxid, v);
            }
        }
        #pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
            flags |= __shfl_xor_sync(0xffffffffu, flags, o);
        }
        if ((threadIdx.x & 31) == 0) {
            s_cnt[threadIdx.x >> 5] = cnt;
            if (flags) atomicOr(err + i * err_stride, flags);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            u32 t = 0;
            for (int w = 0; w < kIngestThreads / 32; ++w) t += s_cnt[w];
            atomicAdd(sizes + i, (u64)t);
        }
        __syncthreads();
    }
}

// f^(l): set bit (x - lo) for every value x of the batch (Eq. 5).  With
// `twice`, also set it there for rows held by two or more samples: the
// atomic OR returns the bits other samples had already set.  A sample's
// repeated value is skipped for `twice` (a set holds it once).
__global__ void __launch_bounds__(kIngestThreads)
k_filter(const u64* __restrict__ ids, u64 n, Plan plan, u64 lo, u64 width, u32* bitmap_all, u32* twice_all,
         const u32* __restrict__ tile_of, u64 tile_words)
{
    __shared__ ChunkDesc s_d[2];
    const u64 nch = plan.totals[1];
    if (threadIdx.x == 0) fetch_chunk(plan, n, nch, kTicketFilter, s_d[0]);
    __syncthreads();
    for (int db = 0;; db ^= 1) {
        const ChunkDesc d = s_d[db];
        if (d.c >= nch) break;
        if (threadIdx.x == 0) fetch_chunk(plan, n, nch, kTicketFilter, s_d[db ^ 1]);
        const u64 p0 = d.p0, p1 = d.p1, bb = d.b;
        // the sample's own bitmap (one per sample tile when tile_of is given)
        const u64 toff = tile_of ? (u64)tile_of[d.i] * tile_words : 0ull;
        u32* bitmap = bitmap_all + toff;
        u32* twice = twice_all ? twice_all + toff : nullptr;
        // every warp walks whole 32-position groups so shuffles see full warps
        for (u64 base = p0 + (threadIdx.x & ~31u); base < p1; base += kIngestThreads) {
            u64 pos = base + (threadIdx.x & 31);
            u64 q = ~0ull;
            u32 bit = 0;
            if (pos < p1) {
                const u64 x = __ldcs(ids + pos);  // read once: evict first
                u64 d = x - lo;
                if (d < width && !(twice && pos > bb && ids[pos - 1] == x)) { q = d >> 5; bit = 1u << (d & 31); }
            }
            bool lead = segmented_or<u32>(q, bit);
            if (lead && bit) {
                const u32 old = atomicOr(bitmap + q, bit);
                if (twice && (old & bit)) atomicOr(twice + q, old & bit);
            }
        }
        __syncthreads();
    }
}

// Directory pass 1: per 4096-word block, block-relative exclusive popcounts.
// Rounds of 512 consecutive words, two per thread, so every load and store
// of a warp is one contiguous 256-byte (load) or 128-byte (store) run.
__global__ void __launch_bounds__(kScanThreads)
k_scan_blocks(const u64* __restrict__ bitmap, u64 nwords, u32* __restrict__ dir, u64* __restrict__ bsum)
{
    constexpr int kRound = 2 * kScanThreads;
    static_assert(kScanBlockWords % kRound == 0, "whole rounds per block");
    __shared__ u32 wsum[kScanThreads / 32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const bool vec = ((uintptr_t)bitmap & 15u) == 0 && ((uintptr_t)dir & 7u) == 0;
    const u64 b0 = (u64)blockIdx.x * kScanBlockWords;
    u32 run = 0;
    for (int it = 0; it < (int)(kScanBlockWords / kRound); ++it) {
        const u64 w = b0 + (u64)it * kRound + 2 * (u64)t;
        u64 a = 0, b = 0;
        if (vec && w + 1 < nwords) {
            const ulonglong2 v = __ldg((const ulonglong2*)(bitmap + w));
            a = v.x;
            b = v.y;
        } else {
            if (w < nwords) a = bitmap[w];
            if (w + 1 < nwords) b = bitmap[w + 1];
        }
        const u32 pa = (u32)__popcll(a), pc = pa + (u32)__popcll(b);
        u32 x = pc;
        #pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const u32 y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[warp] = x;
        __syncthreads();
        u32 woff = 0, tot = 0;
        #pragma unroll
        for (int k = 0; k < kScanThreads / 32; ++k) {
            const u32 v = wsum[k];
            if (k < warp) woff += v;
            tot += v;
        }
        const u32 ex = run + woff + x - pc;
        if (vec && w + 1 < nwords) {
            *(uint2*)(dir + w) = make_uint2(ex, ex + pa);
        } else {
            if (w < nwords) dir[w] = ex;
            if (w + 1 < nwords) dir[w + 1] = ex + pa;
        }
        run += tot;
        __syncthreads();  // wsum is rewritten next round
    }
    if (t == 0) bsum[blockIdx.x] = run;
}

// Directory pass 2 (one CTA): exclusive prefix of block sums; R = total.
__global__ void __launch_bounds__(1024)
k_scan_top(const u64* __restrict__ bsum, u64 nb, u64* __restrict__ boff, u64* R, u64* ktotal, u64* kbase)
{
    __shared__ u64 sm[32];
    u64 carry = 0;
    for (u64 base = 0; base < nb; base += 1024) {
        u64 b = base + threadIdx.x;
        u64 v = b < nb ? bsum[b] : 0, ex;
        u64 tot = block_exclusive_scan<1024>(v, ex, sm);
        if (b < nb) boff[b] = carry + ex;
        carry += tot;
    }
    if (threadIdx.x == 0) {
        *R = carry;
        // batches appended along the word axis: this batch's words start at
        // the running total, which then grows by ceil(R / 64)
        if (ktotal) {
            *kbase = *ktotal;
            *ktotal += (carry + 63) / 64;
        }
    }
}

__global__ void k_zero_rows(u64* X, u64 rows, u64 stride, u64 words)
{
    const u64 per_row = words;
    const u64 total = rows * per_row;
    for (u64 t = (u64)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (u64)gridDim.x * blockDim.x) {
        u64 r = t / per_row, w = t - r * per_row;
        X[r * stride + w] = 0ull;
    }
}

// Bitmask compression: value x of sample i -> rank r = p^(l)_{x-lo}; word
// r/64, bit r%64 of row i (Eq. 6 and the b-bit masks before Eq. 7).
__global__ void __launch_bounds__(kIngestThreads)
k_pack(const u64* __restrict__ ids, u64 n, Plan plan, u64 lo, u64 width,
       const u64* __restrict__ bitmap, const u32* __restrict__ dir, const u64* __restrict__ boff,
       u64* X, u64 stride, u64* batch_sizes, const u64* kbase, u64 wstride)
{
    __shared__ u64 s_i, s_p0, s_p1, s_b, s_c;
    __shared__ u32 s_cnt[kIngestThreads / 32];
    const u64 nch = plan.totals[1];
    for (;;) {
        if (threadIdx.x == 0) {
            const u64 c = next_chunk(plan, kTicketPack);
            s_c = c;
            if (c < nch) {
                u64 i = chunk_sample(plan.cofs, n, c);
                u64 p0 = plan.beg[i] + (c - plan.cofs[i]) * kChunk;
                s_i = i; s_p0 = p0; s_b = plan.beg[i];
                s_p1 = min(p0 + kChunk, plan.beg[i] + plan.len[i]);
            }
        }
        __syncthreads();
        if (s_c >= nch) break;
        const u64 i = s_i, p0 = s_p0, p1 = s_p1, bb = s_b;
        u64* row = X + i * stride + (kbase ? *kbase : 0ull) * wstride;
        u32 cnt = 0;
        for (u64 base = p0 + (threadIdx.x & ~31u); base < p1; base += kIngestThreads) {
            u64 pos = base + (threadIdx.x & 31);
            u64 q = ~0ull, bit = 0;
            if (pos < p1) {
                u64 x = ids[pos];
                u64 d = x - lo;
                if (d < width) {
                    const u64 w = d >> 6, word = bitmap[w];
                    // rows the bitmap leaves out (held by one sample, when it
                    // is the two-or-more filter) are not packed
                    if ((word >> (d & 63)) & 1ull) {
                        u64 r = boff[w / kScanBlockWords] + (u64)dir[w] +
                                (u64)__popcll(word & ((1ull << (d & 63)) - 1ull));
                        q = r >> 6;
                        bit = 1ull << (r & 63);
                    }
                }
                if (batch_sizes) cnt += (pos == bb) || (ids[pos - 1] != x);
            }
            bool lead = segmented_or<u64>(q, bit);
            if (lead && bit) atomicOr(row + q * wstride, bit);
        }
        if (batch_sizes) {
            #pragma unroll
            for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
            if ((threadIdx.x & 31) == 0) s_cnt[threadIdx.x >> 5] = cnt;
            __syncthreads();
            if (threadIdx.x == 0) {
                u32 t = 0;
                for (int w = 0; w < kIngestThreads / 32; ++w) t += s_cnt[w];
                atomicAdd(batch_sizes + i, (u64)t);
            }
        }
        __syncthreads();
    }
}

// Packing of whole rows into the zeroed packed matrix.  Rank r' (the number of
// kept rows below a value) is non-decreasing along a sample's sorted values,
// and so is its word q = r'/64 (a value whose row is not kept still has an
// insertion word), so of a warp's 32 neighbouring values those of one word
// are a run of lanes.  A run inside the group is all there is of its word and
// is stored; the first and the last run may go on in the neighbouring groups
// and are OR-ed in.
//
// Bound by instruction issue: words as 32-bit numbers (ranks are below 2^38:
// every kept row takes 8 bytes of input), no state from group to group.  Pack
// of 1.7e8 values (4000 samples), with open words carried from group to group
// and completed across segments: 1.10 ms, this 1.01.
__global__ void __launch_bounds__(kIngestThreads)
k_pack_full(const u64* __restrict__ ids, u64 n, Plan plan, u64 lo, u64 width, const u64* __restrict__ bitmap,
            const u32* __restrict__ dir, const u64* __restrict__ boff, u64* X, u64 stride,
            const u64* kbase, const u64* __restrict__ Rdev)
{
    __shared__ ChunkDesc s_d[2];
    const u64 nch = plan.totals[1];
    const u32 lane = threadIdx.x & 31;
    const u32 Wl = (u32)((*Rdev + 63) / 64);
    if (threadIdx.x == 0) fetch_chunk(plan, n, nch, kTicketPack, s_d[0]);
    __syncthreads();
    for (int db = 0;; db ^= 1) {
        const ChunkDesc d = s_d[db];
        if (d.c >= nch) break;
        if (threadIdx.x == 0) fetch_chunk(plan, n, nch, kTicketPack, s_d[db ^ 1]);
        const u64 p1 = d.p1;
        u64* row = X + d.i * stride + (kbase ? *kbase : 0ull);
        for (u64 base = d.p0 + (threadIdx.x & ~31u); base < p1; base += kIngestThreads) {
            const u64 pos = base + lane;
            u32 key = ~0u;  // past the end, or outside the batch (unsorted input only): no word
            u64 bit = 0ull;
            if (pos < p1) {
                const u64 x = ids[pos] - lo;
                if (x < width) {
                    const u64 w = x >> 6, word = bitmap[w];
                    const u64 r = boff[w / kScanBlockWords] + dir[w] +
                                  (u64)__popcll(word & ((1ull << (x & 63)) - 1ull));
                    key = (u32)(r >> 6);
                    bit = ((word >> (x & 63)) & 1ull) << (r & 63);
                }
            }
            const bool lead = segmented_or<u64>(key, bit);
            const u32 leads = __ballot_sync(0xffffffffu, lead && pos < p1);  // (the last value's run is an edge)
            if (lead && bit && key < Wl) {
                const bool inside = lane != 0 && (leads >> lane) != 1u;
                if (inside) row[key] = bit;
                else atomicOr((unsigned long long*)(row + key), (unsigned long long)bit);
            }
        }
        __syncthreads();
    }
}

// The class-major layout of the block-sparse product: the rows of a batch
// are split into classes, each with its own bitmap (class c's words at cls +
// c * nwords), rank-scanned together (one directory over all classes; nwords
// is a multiple of kScanBlockWords, so class c's first block is c * nwords /
// kScanBlockWords and its ranks are the directory's minus that block's
// offset).
struct ClassView {
    const u64* cls;      // class bitmaps, class-major
    const u32* dir;      // rank directory of all classes (one entry per word)
    const u64* boff;     // block offsets of all classes
    const u64* kbase;    // first word of each class in X (device)
    u64 nwords;          // bitmap words per class
    const u32* cls_of;   // class of each sample, or null for class 0
    const u32* row_of;   // row of X of each sample
};

// The values' row numbers among the batch's kept rows (bitmap, with its rank
// directory), one u32 per value at the value's own position of `ranks` (~0: a
// row that is not kept), and every tile's bitmap over those rows (tile t's at
// tiles + t * tile_words).
//
// Bound by the latency of three dependent loads (value, bitmap word,
// directory entry); kRankDepth groups of a warp are in flight together, and
// the rank is kept so that the pack reads it in order instead of searching
// the bitmap of the whole value range again.  Whole calls before (tile bitmaps
// and classes over the value range, one copy a tile) and after, clade samples
// over [0, 2^32): 517 x 20,000 values 7.9 -> 2.0 ms, 1024 x 30,000 10.2 -> 4.1,
// 1024 x 100,000 11.4 -> 7.5, 2048 x 20,000 22.5 -> 7.7.
constexpr int kRankDepth = 4;
__global__ void __launch_bounds__(kIngestThreads)
k_rank_tiles(const u64* __restrict__ ids, u64 n, Plan plan, u64 lo, u64 width, const u64* __restrict__ bitmap,
             const u32* __restrict__ dir, const u64* __restrict__ boff, u32* __restrict__ ranks, u32* tiles,
             const u32* __restrict__ tile_of, u64 tile_words)
{
    __shared__ ChunkDesc s_d[2];
    const u64 nch = plan.totals[1];
    if (threadIdx.x == 0) fetch_chunk(plan, n, nch, kTicketRank, s_d[0]);
    __syncthreads();
    for (int db = 0;; db ^= 1) {
        const ChunkDesc d = s_d[db];
        if (d.c >= nch) break;
        if (threadIdx.x == 0) fetch_chunk(plan, n, nch, kTicketRank, s_d[db ^ 1]);
        const u64 p0 = d.p0, p1 = d.p1;
        u32* own = tiles + (u64)tile_of[d.i] * tile_words;
        // every warp walks whole 32-position groups so shuffles see full warps
        for (u64 base = p0 + (threadIdx.x & ~31u); base < p1; base += kRankDepth * kIngestThreads) {
            u64 x[kRankDepth], word[kRankDepth];
            u32 r[kRankDepth];
            #pragma unroll
            for (int k = 0; k < kRankDepth; ++k) {
                const u64 pos = base + (u64)(k * kIngestThreads) + (threadIdx.x & 31);
                x[k] = pos < p1 ? __ldcs(ids + pos) - lo : ~0ull;
            }
            #pragma unroll
            for (int k = 0; k < kRankDepth; ++k) word[k] = x[k] < width ? bitmap[x[k] >> 6] : 0ull;
            #pragma unroll
            for (int k = 0; k < kRankDepth; ++k) {
                r[k] = ~0u;
                if ((word[k] >> (x[k] & 63)) & 1ull) {
                    const u64 w = x[k] >> 6;
                    r[k] = (u32)boff[w / kScanBlockWords] + dir[w] +
                           (u32)__popcll(word[k] & ((1ull << (x[k] & 63)) - 1ull));
                }
            }
            #pragma unroll
            for (int k = 0; k < kRankDepth; ++k) {
                const u64 pos = base + (u64)(k * kIngestThreads) + (threadIdx.x & 31);
                if (pos < p1) __stcs(ranks + pos, r[k]);
                u32 bit = r[k] != ~0u ? 1u << (r[k] & 31) : 0u;
                const u64 q = r[k] != ~0u ? (u64)(r[k] >> 5) : ~0ull;
                const bool lead = segmented_or<u32>(q, bit);
                if (lead && bit) atomicOr(own + q, bit);
            }
        }
        __syncthreads();
    }
}

// Single-pass packing into both class matrices of the block-sparse product:
// a value of sample i whose row is of class 0 goes to XM, one of class
// cls_of[i] (the sample's tile) to XS, at word kbase[c] + (rank within the
// class) / 64 of row row_of[i]; other rows are not packed.  Classes
// interleave along a sample's values, so the words are OR-ed in with atomics
// (lanes of a warp holding the same word combine first).  RANKS: the rows are
// k_rank_tiles' (one u32 per value; `width` of them, values not kept above).
template <bool RANKS>
__global__ void __launch_bounds__(kIngestThreads)
k_pack_classes(const u64* __restrict__ ids, const u32* __restrict__ ranks, u64 n, Plan plan, u64 lo, u64 width,
               ClassView v, u64* XM, u64 stride_m, u64* XS, u64 stride_s)
{
    // 32-value groups of a warp in flight: their values and class-0 words are
    // loaded before any is used (ranks leave registers for more)
    constexpr int kDepth = RANKS ? 4 : 2;
    __shared__ ChunkDesc s_d[2];
    const u64 nch = plan.totals[1];
    const u64 blk0 = 0;
    if (threadIdx.x == 0) fetch_chunk(plan, n, nch, kTicketPack, s_d[0]);
    __syncthreads();
    for (int db = 0;; db ^= 1) {
        const ChunkDesc d = s_d[db];
        if (d.c >= nch) break;
        if (threadIdx.x == 0) fetch_chunk(plan, n, nch, kTicketPack, s_d[db ^ 1]);
        const u64 i = d.i, p0 = d.p0, p1 = d.p1;
        const u64 cs = v.cls_of[i];
        const u64 row = v.row_of[i];
        u64* rowm = XM ? XM + row * stride_m + v.kbase[0] : nullptr;
        u64* rows = XS + row * stride_s + v.kbase[cs];
        const u64 bm0 = blk0, bms = cs * v.nwords / kScanBlockWords;
        for (u64 base = p0 + (threadIdx.x & ~31u); base < p1; base += kDepth * kIngestThreads) {
            u64 d[kDepth], m0[kDepth];
            #pragma unroll
            for (int g = 0; g < kDepth; ++g) {
                const u64 pos = base + (u64)(g * kIngestThreads) + (threadIdx.x & 31);
                d[g] = ~0ull;
                if (pos < p1) d[g] = RANKS ? (u64)__ldcs(ranks + pos) : __ldcs(ids + pos) - lo;
            }
            #pragma unroll
            for (int g = 0; g < kDepth; ++g) m0[g] = d[g] < width ? v.cls[d[g] >> 6] : 0ull;
            #pragma unroll
            for (int g = 0; g < kDepth; ++g) {
                u64 key = ~0ull, bit = 0ull;
                if (d[g] < width) {
                    const u64 w0 = d[g] >> 6, sh = d[g] & 63, low = (1ull << sh) - 1ull;
                    if ((m0[g] >> sh) & 1ull) {
                        const u64 r = v.boff[w0 / kScanBlockWords] - v.boff[bm0] + (u64)v.dir[w0] +
                                      (u64)__popcll(m0[g] & low);
                        key = r >> 6;  // class 0: keys below 2^62
                        bit = 1ull << (r & 63);
                    } else {
                        const u64 ws = cs * v.nwords + w0, ms = v.cls[ws];
                        if ((ms >> sh) & 1ull) {
                            const u64 r = v.boff[ws / kScanBlockWords] - v.boff[bms] + (u64)v.dir[ws] +
                                          (u64)__popcll(ms & low);
                            key = (1ull << 62) | (r >> 6);
                            bit = 1ull << (r & 63);
                        }
                    }
                }
                const bool lead = segmented_or<u64>(key, bit);
                if (lead && bit) {
                    if (key >> 62) atomicOr((unsigned long long*)(rows + (key & ((1ull << 62) - 1))), bit);
                    else atomicOr((unsigned long long*)(rowm + key), bit);
                }
            }
        }
        __syncthreads();
    }
}

// The smallest first value and the largest last value over the non-empty
// samples (for sorted samples: the collection's minimum and maximum); out
// must hold {~0, 0} before.  One CTA.
__global__ void __launch_bounds__(kPlanThreads)
k_first_last(const u64* __restrict__ offsets, const u64* __restrict__ ids, u64 n, u64* out, u64* probes, u64 N)
{
    take_probes(ids, N, probes);
    __shared__ unsigned long long s_min, s_max;
    if (threadIdx.x == 0) { s_min = ~0ull; s_max = 0ull; }
    __syncthreads();
    unsigned long long mn = ~0ull, mx = 0ull;
    for (u64 i = threadIdx.x; i < n; i += blockDim.x) {
        const u64 a = offsets[i], e = offsets[i + 1];
        if (e > a) {
            mn = min(mn, (unsigned long long)ids[a]);
            mx = max(mx, (unsigned long long)ids[e - 1]);
        }
    }
    atomicMin(&s_min, mn);
    atomicMax(&s_max, mx);
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicMin((unsigned long long*)out, s_min);
        atomicMax((unsigned long long*)out + 1, s_max);
    }
}

inline unsigned grid_for_chunks(u64 max_chunks, int sms)
{
    u64 g = (u64)sms * 8;
    if (max_chunks < g) g = max_chunks;
    return (unsigned)(g ? g : 1);
}

}  // namespace

cudaError_t launch_plan(const u64* offsets, const u64* ids, u64 n, u64 lo, u64 hi, bool full,
                        Plan plan, cudaStream_t st, const u32* perm, const u64* ends, u64* probes, u64 N)
{
    k_plan<<<1, kPlanThreads, 0, st>>>(offsets, ids, n, lo, hi, full ? 1 : 0, plan, perm, ends, probes, N);
    return cudaGetLastError();
}

cudaError_t launch_validate(const u64* offsets, const u64* ids, u64 n, Plan plan, u64 max_chunks,
                            int id_bits, u64* sizes, u32* err, u64* maxid, u64* minid, int sms,
                            cudaStream_t st, u64 err_stride)
{
    k_validate<<<grid_for_chunks(max_chunks, sms), kIngestThreads, 0, st>>>(offsets, ids, n, plan, id_bits,
                                                                            sizes, err, maxid, minid, err_stride);
    return cudaGetLastError();
}

cudaError_t launch_filter_tiles(const u64* ids, u64 n, Plan plan, u64 max_chunks, u64 lo, u64 width,
                               u32* bitmaps, u32* twice, const u32* tile_of, int sms, cudaStream_t st)
{
    k_filter<<<grid_for_chunks(max_chunks, sms), kIngestThreads, 0, st>>>(ids, n, plan, lo, width, bitmaps, twice,
                                                                          tile_of, width / 32);
    return cudaGetLastError();
}

cudaError_t launch_filter(const u64* ids, u64 n, Plan plan, u64 max_chunks, u64 lo, u64 width,
                          u32* bitmap, int sms, cudaStream_t st, u32* twice)
{
    k_filter<<<grid_for_chunks(max_chunks, sms), kIngestThreads, 0, st>>>(ids, n, plan, lo, width, bitmap, twice,
                                                                          nullptr, 0);
    return cudaGetLastError();
}

cudaError_t launch_scan(const u64* bitmap, u64 nwords, u32* dir, u64* bsum, u64* boff, u64* R,
                        cudaStream_t st, u64* ktotal, u64* kbase)
{
    u64 nb = (nwords + kScanBlockWords - 1) / kScanBlockWords;
    if (nb == 0) nb = 1;
    k_scan_blocks<<<(unsigned)nb, kScanThreads, 0, st>>>(bitmap, nwords, dir, bsum);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_scan_top<<<1, 1024, 0, st>>>(bsum, nb, boff, R, ktotal, kbase);
    return cudaGetLastError();
}

cudaError_t launch_scan_top(const u64* bsum, u64 nb, u64* boff, u64* R, cudaStream_t st)
{
    k_scan_top<<<1, 1024, 0, st>>>(bsum, nb, boff, R, nullptr, nullptr);
    return cudaGetLastError();
}

cudaError_t launch_pack_full(const u64* ids, u64 n, Plan plan, u64 max_chunks, u64 lo, u64 width,
                             const u64* bitmap, const u32* dir, const u64* boff, u64* X, u64 stride,
                             const u64* Rdev, int sms, cudaStream_t st, const u64* kbase)
{
    k_pack_full<<<grid_for_chunks(max_chunks, sms), kIngestThreads, 0, st>>>(ids, n, plan, lo, width, bitmap, dir,
                                                                            boff, X, stride, kbase, Rdev);
    return cudaGetLastError();
}

cudaError_t launch_rank_tiles(const u64* ids, u64 n, Plan plan, u64 max_chunks, u64 lo, u64 width, const u64* bitmap,
                              const u32* dir, const u64* boff, u32* ranks, u32* tiles, const u32* tile_of,
                              u64 tile_words, int sms, cudaStream_t st)
{
    k_rank_tiles<<<grid_for_chunks(max_chunks, sms), kIngestThreads, 0, st>>>(ids, n, plan, lo, width, bitmap, dir, boff,
                                                                              ranks, tiles, tile_of, tile_words);
    return cudaGetLastError();
}

cudaError_t launch_pack_classes(const u64* ids, const u32* ranks, u64 n, Plan plan, u64 max_chunks, u64 lo, u64 width,
                                const u64* cls, const u32* dir, const u64* boff, u64 nwords, const u64* kbase,
                                const u32* cls_of, const u32* row_of, u64* XM, u64 stride_m, u64* XS, u64 stride_s,
                                int sms, cudaStream_t st)
{
    ClassView v{cls, dir, boff, kbase, nwords, cls_of, row_of};
    const unsigned g = grid_for_chunks(max_chunks, sms);
    if (ranks)
        k_pack_classes<true><<<g, kIngestThreads, 0, st>>>(ids, ranks, n, plan, lo, width, v, XM, stride_m, XS, stride_s);
    else
        k_pack_classes<false><<<g, kIngestThreads, 0, st>>>(ids, ranks, n, plan, lo, width, v, XM, stride_m, XS,
                                                            stride_s);
    return cudaGetLastError();
}

cudaError_t launch_first_last(const u64* offsets, const u64* ids, u64 n, u64* out, cudaStream_t st, u64* probes, u64 N)
{
    k_first_last<<<1, kPlanThreads, 0, st>>>(offsets, ids, n, out, probes, N);
    return cudaGetLastError();
}

cudaError_t launch_zero_rows(u64* X, u64 rows, u64 stride, u64 words, int sms, cudaStream_t st)
{
    if (rows == 0 || words == 0) return cudaSuccess;
    u64 total = rows * words;
    u64 g = (total + 255) / 256;
    u64 cap = (u64)sms * 16;
    if (g > cap) g = cap;
    k_zero_rows<<<(unsigned)g, 256, 0, st>>>(X, rows, stride, words);
    return cudaGetLastError();
}

cudaError_t launch_pack(const u64* ids, u64 n, Plan plan, u64 max_chunks, u64 lo, u64 width,
                        const u64* bitmap, const u32* dir, const u64* boff, u64* X, u64 stride,
                        u64* batch_sizes, int sms, cudaStream_t st, const u64* kbase, u64 wstride)
{
    k_pack<<<grid_for_chunks(max_chunks, sms), kIngestThreads, 0, st>>>(ids, n, plan, lo, width, bitmap, dir,
                                                                        boff, X, stride, batch_sizes, kbase,
                                                                        wstride);
    return cudaGetLastError();
}

}  // namespace jsim
