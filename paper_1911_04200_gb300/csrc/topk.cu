// Nearest neighbours from a similarity matrix: for every sample the k others
// with the largest J (the sparsified output that large collections need in
// place of an n x n matrix).  Ties in J go to the smaller index, so the
// result is unique.
//
// A CTA per row.  Candidates are ordered by (bits of J descending, index
// ascending) - non-negative doubles order like their bit patterns, and the
// index makes every candidate distinct.  The row is read once: every thread
// takes the largest of its share, and the k-th largest of those maxima bounds
// the k-th best from below (k <= 64 of 256 threads), so the few candidates at
// or above it hold the answer; they are collected and each one's rank counted
// among them.  Should more than kTkCand pass (many equal values), pass t over
// the row takes the best candidate strictly after the pick of pass t-1.
//
// Bound by reading J.  n = 4096, k = 10 (134 MB): k passes over the staged
// row 262 us, this 56.  Pairs above a threshold of the same matrix: binary64
// compares 42 us, integer ones 19 (threshold.cu).
#include <algorithm>
#include "ctx.cuh"

namespace {

constexpr int kTkThreads = 256;
constexpr int kTkDepth = 8;         // loads of a thread in flight
constexpr u32 kTkCand = 512;        // candidates ranked in shared memory
constexpr u64 kTkSmemRows = 16384;  // rows up to this length are staged in shared memory

__global__ void __launch_bounds__(kTkThreads)
k_topk(const double* __restrict__ J, u64 n, u32 k, u64* __restrict__ idx, double* __restrict__ val)
{
    extern __shared__ double row_s[];
    __shared__ u64 red_b[kTkThreads / 32];
    __shared__ u64 red_j[kTkThreads / 32];
    __shared__ u64 cand_b[kTkCand];
    __shared__ u32 cand_j[kTkCand];
    __shared__ u32 maxima[kTkThreads];
    __shared__ u32 s_cut, s_count;
    const u64 i = blockIdx.x;
    const double* row = J + i * n;
    const bool staged = n <= kTkSmemRows;
    const u32 t = threadIdx.x;
    const int lane = t & 31, warp = t >> 5;
    const u32 m32 = (u32)n, i32 = (u32)i;  // (n x n binary64 fit no device above 2^31)
    // the largest upper half among this thread's values
    u32 mx = 0;
    for (u32 c0 = 0; c0 < m32; c0 += kTkDepth * kTkThreads) {
        const bool whole = m32 - c0 >= kTkDepth * kTkThreads;
        double v[kTkDepth];
        #pragma unroll
        for (u32 q = 0; q < kTkDepth; ++q) {
            const u32 j = c0 + q * kTkThreads + t;
            v[q] = whole || j < m32 ? row[j] : 0.0;
        }
        #pragma unroll
        for (u32 q = 0; q < kTkDepth; ++q) {
            const u32 j = c0 + q * kTkThreads + t;
            if (!whole && j >= m32) break;
            if (staged) row_s[j] = v[q];
            if (j != i32) mx = max(mx, (u32)__double2hiint(v[q]));
        }
    }
    maxima[t] = mx;
    if (t == 0) s_count = 0;
    __syncthreads();
    if (warp == 0) {
        // the largest cut that k of the maxima reach, bit by bit
        u32 m[kTkThreads / 32];
        #pragma unroll
        for (int q = 0; q < kTkThreads / 32; ++q) m[q] = maxima[32 * q + lane];
        u32 hi = 0, lo = ~0u;
        #pragma unroll
        for (int q = 0; q < kTkThreads / 32; ++q) { hi = max(hi, m[q]); lo = min(lo, m[q]); }
        hi = __reduce_max_sync(0xffffffffu, hi);
        lo = __reduce_min_sync(0xffffffffu, lo);
        // (all of them reach lo: the search begins below their common bits)
        const int top = hi == lo ? -1 : 31 - __clz((int)(hi ^ lo));
        u32 cut = hi == lo ? lo : hi & ~((2u << top) - 1u);
        for (int bit = top; bit >= 0; --bit) {
            const u32 c = cut | (1u << bit);
            u32 have = 0;
            #pragma unroll
            for (int q = 0; q < kTkThreads / 32; ++q) have += m[q] >= c ? 1u : 0u;
            have = __reduce_add_sync(0xffffffffu, have);
            if (have >= k) cut = c;
            if (have == k) break;
        }
        if (lane == 0) s_cut = cut;
    }
    __syncthreads();
    const u32 cut = s_cut;
    for (u32 c0 = 0; c0 < m32; c0 += kTkDepth * kTkThreads) {
        const bool whole = m32 - c0 >= kTkDepth * kTkThreads;
        double v[kTkDepth];
        #pragma unroll
        for (u32 q = 0; q < kTkDepth; ++q) {
            const u32 j = c0 + q * kTkThreads + t;
            v[q] = whole || j < m32 ? (staged ? row_s[j] : row[j]) : 0.0;
        }
        #pragma unroll
        for (u32 q = 0; q < kTkDepth; ++q) {
            const u32 j = c0 + q * kTkThreads + t;
            if ((u32)__double2hiint(v[q]) >= cut && j != i32 && (whole || j < m32)) {
                const u32 at = atomicAdd(&s_count, 1u);
                if (at < kTkCand) {
                    cand_b[at] = (u64)__double_as_longlong(v[q]);
                    cand_j[at] = j;
                }
            }
        }
    }
    __syncthreads();
    const u32 count = s_count;
    if (count <= kTkCand) {
        for (u32 c = t; c < count; c += kTkThreads) {
            const u64 b = cand_b[c];
            const u32 j = cand_j[c];
            u32 rank = 0;
            for (u32 o = 0; o < count; ++o) rank += cand_b[o] > b || (cand_b[o] == b && cand_j[o] < j) ? 1u : 0u;
            if (rank < k) {
                idx[i * k + rank] = j;
                if (val) val[i * k + rank] = __longlong_as_double((long long)b);
            }
        }
        return;
    }
    // previous pick (bits of J, index): the next pick is the best strictly after it
    u64 pb = ~0ull, pj = 0;
    bool first = true;
    for (u32 p = 0; p < k; ++p) {
        u64 bb = 0, bj = ~0ull;
        bool have = false;
        for (u64 j = t; j < n; j += kTkThreads) {
            if (j == i) continue;
            const u64 b = (u64)__double_as_longlong(staged ? row_s[j] : row[j]);
            // strictly after (pb, pj) in (bits desc, index asc)
            const bool after = first || b < pb || (b == pb && j > pj);
            if (!after) continue;
            // better than the current best (bb, bj)?
            if (!have || b > bb || (b == bb && j < bj)) { bb = b; bj = j; have = true; }
        }
        if (!have) { bb = 0; bj = ~0ull; }
        // block-wide best: larger bits, then smaller index; "none" is (0, ~0)
        #pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const u64 ob = __shfl_xor_sync(0xffffffffu, bb, o), oj = __shfl_xor_sync(0xffffffffu, bj, o);
            if (ob > bb || (ob == bb && oj < bj)) { bb = ob; bj = oj; }
        }
        if (lane == 0) { red_b[warp] = bb; red_j[warp] = bj; }
        __syncthreads();
        if (warp == 0) {
            bb = lane < kTkThreads / 32 ? red_b[lane] : 0ull;
            bj = lane < kTkThreads / 32 ? red_j[lane] : ~0ull;
            #pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const u64 ob = __shfl_xor_sync(0xffffffffu, bb, o), oj = __shfl_xor_sync(0xffffffffu, bj, o);
                if (ob > bb || (ob == bb && oj < bj)) { bb = ob; bj = oj; }
            }
            if (lane == 0) { red_b[0] = bb; red_j[0] = bj; }
        }
        __syncthreads();
        pb = red_b[0];
        pj = red_j[0];
        first = false;
        if (t == 0) {
            idx[i * k + p] = pj;
            if (val) val[i * k + p] = __longlong_as_double((long long)pb);
        }
        __syncthreads();
    }
}

}  // namespace

extern "C" int jsim_topk(jsim_ctx* ctx, const double* J, uint64_t n, uint32_t k, uint64_t* idx, double* val, int mem)
{
    if (!ctx || !J || !idx) return JSIM_ERR_ARG;
    if (mem != JSIM_MEM_HOST && mem != JSIM_MEM_DEVICE) return JSIM_ERR_ARG;
    if (k == 0 || k > 64 || n < 2 || k > n - 1 || n > 0xffffffffull) return JSIM_ERR_ARG;
    CK(cudaSetDevice(ctx->opt.device));
    CallScope scope(ctx);
    StageTimer total(ctx, &ctx->stats.ms_total);
    cudaStream_t st = ctx->stream;
    DevBuf Jd, id, vd;
    const double* Jp = J;
    u64* ip = (u64*)idx;
    double* vp = val;
    if (mem == JSIM_MEM_HOST) {
        ALLOC(Jd, n * n * sizeof(double));
        CK(cudaMemcpyAsync(Jd.p, J, n * n * sizeof(double), cudaMemcpyHostToDevice, st));
        Jp = Jd.as<double>();
        ALLOC(id, n * k * sizeof(u64));
        ip = id.as<u64>();
        if (val) {
            ALLOC(vd, n * k * sizeof(double));
            vp = vd.as<double>();
        }
    }
    const size_t smem = n <= kTkSmemRows ? n * sizeof(double) : 0;
    CK(cudaFuncSetAttribute(k_topk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kTkSmemRows * 8)));
    {
        StageTimer t(ctx, &ctx->stats.ms_epilogue);
        k_topk<<<(unsigned)n, kTkThreads, smem, st>>>(Jp, n, k, ip, vp);
        CK(cudaGetLastError());
        ctx->stats.launches += 1;
    }
    if (mem == JSIM_MEM_HOST) {
        CK(cudaMemcpyAsync(idx, ip, n * k * sizeof(u64), cudaMemcpyDeviceToHost, st));
        if (val) CK(cudaMemcpyAsync(val, vp, n * k * sizeof(double), cudaMemcpyDeviceToHost, st));
    }
    CK(cudaStreamSynchronize(st));
    return JSIM_OK;
}
