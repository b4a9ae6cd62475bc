// Diagonal tiles of the block-sparse path on the tensor cores (tcgen05,
// sm_103a): for up to 16 tiles of at most 128 samples each, C_t += X_t X_t^T
// over (AND, popcount, +) (Eq. 7), one 128 x 128 block per tile, all tiles in
// one persistent launch.
//
// The operands are 4-bit (kind::mxf4) with the encoding of the SM-pair
// product (product_tc2.cu): 128 bits of a row become four 16-byte blocks, the
// words masked to every nibble's bit 0, 1 and 2, and bit 3 shifted into bit
// 2, and the block scales 2, 1, 1/2, 1/2 make every set bit 1.  Rows and
// columns are the same samples, so a stage is unpacked once and the MMA reads
// the same shared memory for both operands.
//
// What bounds it: shared memory.  512 bit-rows take 32 KiB of writes and 64
// KiB of operand reads (768 cycles at 128 bytes a cycle) and 512 cycles of
// MMA.  The words come by TMA (64 bytes of every row), so the unpacking warps
// compute no addresses; waits suspend in hardware.  Measured on 1024 clade
// samples (8 tiles, 6.6e5 words each): FP8 operands, row-wise 16-byte loads
// 5.1 ms; this kernel 2.4 ms.
//
// Work: the (tile, 512-bit stage) units of all tiles are laid out tile-major
// and one CTA per SM takes an equal contiguous share, split into segments at
// tile boundaries and at the exactness cap of 2^22 bit-rows
// (product_tc_sched.cuh).  Roles (14 warps): warps 0-7 unpack (16 rows each),
// warp 8 issues the MMAs, warps 9-12 add finished accumulators into C while
// the next runs (two accumulators in turn), warp 13 loads.  Every wait is
// bounded (clock64 budget, plus a CTA-wide abort flag); on time-out the CTA
// raises the error word, waits (bounded) for its issued MMAs and copies,
// frees its TMEM and leaves.
#include <algorithm>
#include <vector>
#include "tensor_map.cuh"
#include "product_tc_sched.cuh"

namespace jsim {

namespace {

using tcs::JobInfo;
using tcs::Seg;
using tcs::Slots;
using tcs::WorkIter;

constexpr int kMaxDiag = 16;
constexpr int kRows = 128;
constexpr int kStageBits = 512;
constexpr int kStageWords = kStageBits / 64;
constexpr int kSteps = kStageBits / 64;           // MMAs (K = 64) of a stage
constexpr int kAtom = kRows * 128;                // a 128-byte swizzle atom column: 256 bit-rows
constexpr int kStageBytes = kStageBits / 256 * kAtom;  // 32 KiB
constexpr int kBufs = 4;
constexpr int kSlotBytes = kRows * kStageWords * 8;    // packed words of a stage: 8 KiB
constexpr int kSlots = 6;
constexpr int kSmemBytes = kBufs * kStageBytes + kSlots * kSlotBytes + 1024;  // + alignment slack
static_assert(kSmemBytes + 4096 <= 232448, "fits the per-CTA shared-memory limit");
constexpr int kUnpackWarps = 8;
constexpr int kMmaWarp = kUnpackWarps;
constexpr int kEpiWarp0 = kUnpackWarps + 1;
constexpr int kLoadWarp = kUnpackWarps + 5;
constexpr int kThreads = (kLoadWarp + 1) * 32;
static_assert(kEpiWarp0 % 4 == 1, "epilogue warp e reads TMEM lanes of warp rank (kEpiWarp0 + e) % 4");
constexpr int kTmemCols = 512;                    // two 128-column accumulators, 8 columns of scales
constexpr u32 kScaleCol = 2 * kRows;
constexpr u32 kScales = 0x7e7e7f80u;              // ue8m0 2, 1, 1/2, 1/2: blocks 0-3 of 128 bits
constexpr u64 kMaxSeg = (1ull << 22) / kStageBits;
constexpr u32 kErrTimeout = 4u;
constexpr u32 kSuspendNs = 20000;

// instruction descriptor: kind::mxf4, A = B = E2M1, both K-major, N = 128
// (bits 17..22 hold N/8), ue8m0 scales (bit 23), M = 128 (bits 24..28 hold
// M/16); kScaleHigh: scale bytes 2-3 of both operands
constexpr u32 kIdesc =
    (1u << 7) | (1u << 10) | ((u32)(kRows >> 3) << 17) | (1u << 23) | ((u32)(kRows >> 4) << 24);
constexpr u32 kScaleHigh = (2u << 4) | (2u << 29);

struct DiagParams {
    CUtensorMap map[kMaxDiag];
    void* C[kMaxDiag];
    u64 n[kMaxDiag], W[kMaxDiag], ldc[kMaxDiag];
    const u64* Wdev[kMaxDiag];  // optional: the words of the job, W their bound (zeros between)
    u32 njobs;
};

__device__ __forceinline__ u32 smem_u32(const void* p) { return (u32)__cvta_generic_to_shared(p); }

__device__ __forceinline__ u64 sw128_desc(u32 saddr)
{
    return (u64)((saddr & 0x3FFFFu) >> 4) | ((u64)1 << 16) | ((u64)(1024 >> 4) << 32) | ((u64)1 << 46) |
           ((u64)2 << 61);
}

__device__ __forceinline__ void mbar_init(u64* bar, u32 count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" :: "r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(u64* bar)
{
    asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" :: "r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(u64* bar, u32 parity)
{
    u32 ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2, %3;\n"
                 " selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity), "r"(kSuspendNs) : "memory");
    return ok != 0;
}

// Bounded wait; false on time-out or when another role has aborted the CTA.
__device__ __forceinline__ bool mbar_wait(u64* bar, u32 parity, long long budget, volatile int* abort_flag)
{
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (*abort_flag) return false;
        if (clock64() - t0 > budget) {
            *abort_flag = 1;
            return false;
        }
    }
    return true;
}

__device__ __forceinline__ void commit(u64* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
                 :: "r"(smem_u32(bar)) : "memory");
}

// 128 bits of a row -> its four 16-byte blocks, block m at chunk m ^ c of the
// row's 128 bytes at rowp
__device__ __forceinline__ void store_blocks(unsigned char* rowp, u32 c, ulonglong2 w)
{
    const u32 x0 = (u32)w.x, x1 = (u32)(w.x >> 32), x2 = (u32)w.y, x3 = (u32)(w.y >> 32);
    const u32 m0 = 0x11111111u, m1 = 0x22222222u, m2 = 0x44444444u;
    *(uint4*)(rowp + ((0 ^ c) << 4)) = make_uint4(x0 & m0, x1 & m0, x2 & m0, x3 & m0);
    *(uint4*)(rowp + ((1 ^ c) << 4)) = make_uint4(x0 & m1, x1 & m1, x2 & m1, x3 & m1);
    *(uint4*)(rowp + ((2 ^ c) << 4)) = make_uint4(x0 & m2, x1 & m2, x2 & m2, x3 & m2);
    *(uint4*)(rowp + ((3 ^ c) << 4)) = make_uint4((x0 >> 1) & m2, (x1 >> 1) & m2, (x2 >> 1) & m2, (x3 >> 1) & m2);
}

__device__ __forceinline__ void tmem_ld32(u32 taddr, u32 (&r)[32])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                   "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
                   "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
                   "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}

template <typename CT>
__global__ void __launch_bounds__(kThreads, 1)
k_prod_diag(const __grid_constant__ DiagParams P, u32* err, long long budget)
{
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) u64 full_bar[kBufs], empty_bar[kBufs], ldf_bar[kSlots], lde_bar[kSlots], accf_bar[2],
        acce_bar[2], done_bar;
    __shared__ u32 tmem_slot;
    __shared__ int abort_flag;
    __shared__ JobInfo ji[kMaxDiag];
    __shared__ u64 s_T;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const u32 njobs = P.njobs;
    if (tid == 0) {
        u64 U = 0;
        for (u32 j = 0; j < njobs; ++j) {
            const u64 W = P.Wdev[j] ? min(P.W[j], *P.Wdev[j]) : P.W[j];
            ji[j] = tcs::job_info(P.n[j], W, U, kRows, kStageWords);
            U += ji[j].tiles * ji[j].nst;
        }
        s_T = tcs::cta_stages(U, gridDim.x, blockIdx.x);
    }
    __syncthreads();
    const u64 T = s_T;
    if (T == 0) return;  // uniform per CTA, before any TMEM or barrier use

    const u32 raw = smem_u32(smem_raw);
    const u32 base = (raw + 1023u) & ~1023u;
    unsigned char* sm = smem_raw + (base - raw);

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n"
                     :: "r"(smem_u32(&tmem_slot)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 32) {
        for (int b = 0; b < kBufs; ++b) {
            mbar_init(&full_bar[b], kUnpackWarps);
            mbar_init(&empty_bar[b], 1);
        }
        for (int y = 0; y < kSlots; ++y) {
            mbar_init(&ldf_bar[y], 1);
            mbar_init(&lde_bar[y], kUnpackWarps);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&accf_bar[a], 1);
            mbar_init(&acce_bar[a], 4);
        }
        mbar_init(&done_bar, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const u32 tmem = tmem_slot;
    if (warp >= kEpiWarp0 && warp < kLoadWarp) {
        // the block scales, in every lane of 8 columns
        const u32 at = tmem + ((((u32)(warp - kEpiWarp0 + 1) & 3u) * 32u) << 16) + kScaleCol;
        asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1};\n"
                     "tcgen05.wait::st.sync.aligned;\n" :: "r"(at), "r"(kScales) : "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    volatile int* abort_v = &abort_flag;
    unsigned char* slots = sm + kBufs * kStageBytes;

    if (warp < kUnpackWarps) {
        // ---------------- unpack ----------------
        // Lane l takes 16-byte piece l % 4 of row l / 4 of two groups of 8 rows
        // (rows of a slot are 64 bytes: the lanes read contiguously).  Piece h
        // is half h % 2 of atom column h / 2; block m of it goes to chunk
        // (4 (h % 2) + m) ^ (2 (h / 2)), stored at ^ (row % 8): the 8 lanes that
        // store together (two rows, four pieces) hit 8 chunk columns, and atom
        // column 1 holds blocks 2-3 before blocks 0-1.
        const int lr = lane >> 2, h = lane & 3;
        const u32 chunk = (u32)((4 * (h & 1)) ^ (2 * (h >> 1)) ^ lr);
        const u32 src = (u32)(warp * 16 * 64 + lane * 16);
        const u32 dst = (u32)((h >> 1) * kAtom + (warp * 16 + lr) * 128);
        int b = 0, y = 0;
        u32 par = 1, lpar = 0;
        for (u64 t = 0; t < T; ++t) {
            bool ok = mbar_wait(&ldf_bar[y], lpar, budget, abort_v);
            const ulonglong2 w0 = *(const ulonglong2*)(slots + y * kSlotBytes + src);
            const ulonglong2 w1 = *(const ulonglong2*)(slots + y * kSlotBytes + src + 8 * 64);
            // The slot has been read: the fence orders these reads before the
            // async proxy's next write to it.  Without it the release overtook
            // reads still in flight, and stages mixed old and new words when
            // copy CTAs shared the SM.
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&lde_bar[y]);
            ok = ok && (t < kBufs || mbar_wait(&empty_bar[b], par, budget, abort_v));
            if (!__all_sync(0xffffffffu, ok)) break;
            unsigned char* st = sm + b * kStageBytes + dst;
            store_blocks(st, chunk, w0);
            store_blocks(st + 8 * 128, chunk, w1);
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&full_bar[b]);
            if (++b == kBufs) { b = 0; par ^= 1u; }
            if (++y == kSlots) { y = 0; lpar ^= 1u; }
        }
    } else if (warp == kMmaWarp) {
        // ---------------- MMA issuer ----------------
        if (lane == 0) {
            WorkIter it;
            it.init(ji, njobs, gridDim.x, blockIdx.x);
            it.max_seg = kMaxSeg;
            Slots sl;
            sl.init();
            sl.max_seg = kMaxSeg;
            Seg sg;
            int b = 0;
            u32 par = 0;
            bool ok = true;
            while (ok && it.next(sg)) {
                const u64 tile = ((u64)sg.job << 40) | sg.tile, len = sg.len;
                const int sidx = sl.pick(tile);
                if (sl.needs_flush(sidx, tile, len)) {
                    commit(&accf_bar[sidx]);
                    sl.flushes[sidx] += 1;
                    sl.tile[sidx] = ~0ull;
                }
                bool fresh = false;
                if (sl.tile[sidx] == ~0ull) {
                    // reuse of a flushed slot waits until the epilogue has read it
                    if (sl.flushes[sidx] > 0 &&
                        !mbar_wait(&acce_bar[sidx], (sl.flushes[sidx] - 1) & 1u, budget, abort_v)) {
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    sl.tile[sidx] = tile;
                    sl.fill[sidx] = 0;
                    fresh = true;
                }
                const u32 dt = tmem + (u32)sidx * (u32)kRows;
                for (u64 q = 0; q < len; ++q) {
                    if (!mbar_wait(&full_bar[b], par, budget, abort_v)) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    const u32 abase = base + b * kStageBytes;
                    #pragma unroll
                    for (int k = 0; k < kSteps; ++k) {
                        // K step k: atom column k / 4, 32-byte slice k % 4: blocks 0-1
                        // or 2-3 of 128 bits, the other way round in atom column 1
                        const u64 d = sw128_desc(abase + (k >> 2) * kAtom + (k & 3) * 32);
                        const u32 accum = (fresh && q == 0 && k == 0) ? 0u : 1u;
                        asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                                     " tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X"
                                     " [%0], %1, %1, %2, [%3], [%3], p;\n}\n"
                                     :: "r"(dt), "l"(d), "r"(((k ^ (k >> 2)) & 1) ? kIdesc | kScaleHigh : kIdesc),
                                        "r"(tmem + kScaleCol), "r"(accum) : "memory");
                    }
                    commit(&empty_bar[b]);
                    if (++b == kBufs) { b = 0; par ^= 1u; }
                }
                sl.fill[sidx] += len;
                sl.last = sidx;
            }
            if (ok)
                for (int sidx = 0; sidx < 2; ++sidx)
                    if (sl.tile[sidx] != ~0ull) commit(&accf_bar[sidx]);
            commit(&done_bar);  // every MMA this thread issued completes before this arrival
        }
        __syncwarp();
    } else if (warp == kLoadWarp) {
        // ---------------- packed words ----------------
        if (lane == 0) {
            WorkIter it;
            it.init(ji, njobs, gridDim.x, blockIdx.x);
            it.max_seg = kMaxSeg;
            Seg sg;
            u64 t = 0;
            bool ok = true;
            while (ok && it.next(sg)) {
                for (u64 q = 0; q < sg.len; ++q, ++t) {
                    const int y = (int)(t % kSlots);
                    if (t >= kSlots && !mbar_wait(&lde_bar[y], (u32)((t / kSlots - 1) & 1), budget, abort_v)) {
                        ok = false;
                        break;
                    }
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n"
                                 :: "r"(smem_u32(&ldf_bar[y])), "r"(kSlotBytes) : "memory");
                    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
                                 " [%0], [%1, {%2, %3}], [%4];\n"
                                 :: "r"(base + kBufs * kStageBytes + y * kSlotBytes), "l"(&P.map[sg.job]),
                                    "r"((int)((sg.kst + q) * kStageWords)), "r"(0), "r"(smem_u32(&ldf_bar[y]))
                                 : "memory");
                }
            }
            // no copy of this CTA is in flight when it ends (bounded)
            for (u64 q = t > kSlots ? t - kSlots : 0; q < t; ++q) {
                const long long t0 = clock64();
                while (!mbar_try_wait(&ldf_bar[q % kSlots], (u32)((q / kSlots) & 1)))
                    if (clock64() - t0 > budget) { *abort_v = 1; break; }
            }
        }
        __syncwarp();
    } else {
        // ---------------- epilogue ----------------
        const int e = (warp - kEpiWarp0 + 1) & 3;  // TMEM lane quarter of this warp (warp % 4)
        auto drain = [&](int sidx, u64 key, u32 nth) -> bool {
            int got = 0;
            if (lane == 0) got = mbar_wait(&accf_bar[sidx], nth & 1u, budget, abort_v) ? 1 : 0;
            got = __shfl_sync(0xffffffffu, got, 0);  // the warp follows one verdict
            if (!got) return false;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const u32 jb = (u32)(key >> 40);
            CT* C = (CT*)P.C[jb];
            const u64 n = P.n[jb], ldc = P.ldc[jb], i = (u64)(e * 32 + lane);
            #pragma unroll 1
            for (int cb = 0; cb < kRows / 32; ++cb) {
                u32 r[32];
                tmem_ld32(tmem + ((u32)(e * 32) << 16) + (u32)(sidx * kRows + cb * 32), r);
                if (i < n) {
                    #pragma unroll
                    for (int x = 0; x < 32; ++x) {
                        const u64 j = (u64)(cb * 32 + x);
                        const u32 v = (u32)__uint_as_float(r[x]);
                        if (j < n && i <= j && v) atomicAdd(C + i * ldc + j, (CT)v);
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&acce_bar[sidx]);
            return true;
        };
        WorkIter it;
        it.init(ji, njobs, gridDim.x, blockIdx.x);
        it.max_seg = kMaxSeg;
        Slots sl;
        sl.init();
        sl.max_seg = kMaxSeg;
        Seg sg;
        bool ok = true;
        while (ok && it.next(sg)) {
            const u64 tile = ((u64)sg.job << 40) | sg.tile, len = sg.len;
            const int sidx = sl.pick(tile);
            if (sl.needs_flush(sidx, tile, len)) {
                ok = drain(sidx, sl.tile[sidx], sl.flushes[sidx]);
                sl.flushes[sidx] += 1;
                sl.tile[sidx] = ~0ull;
            }
            if (sl.tile[sidx] == ~0ull) {
                sl.tile[sidx] = tile;
                sl.fill[sidx] = 0;
            }
            sl.fill[sidx] += len;
            sl.last = sidx;
        }
        for (int sidx = 0; ok && sidx < 2; ++sidx) {
            if (sl.tile[sidx] == ~0ull) continue;
            ok = drain(sidx, sl.tile[sidx], sl.flushes[sidx]);
            sl.flushes[sidx] += 1;
        }
    }

    // wait (bounded) until every issued MMA has completed, then free TMEM
    if (warp == 0) {
        const long long t0 = clock64();
        while (!mbar_try_wait(&done_bar, 0u))
            if (clock64() - t0 > budget) { *abort_v = 1; break; }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (tid == 0 && *abort_v) atomicOr(err, kErrTimeout);
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" :: "r"(tmem), "r"(kTmemCols)
                     : "memory");
    }
}

template <typename CT>
cudaError_t run(const DiagParams& P, int sms, u32* err, int timeout_ms, cudaStream_t st)
{
    cudaError_t e = cudaFuncSetAttribute(k_prod_diag<CT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (e != cudaSuccess) return e;
    k_prod_diag<CT><<<(unsigned)sms, kThreads, kSmemBytes, st>>>(P, err, wait_budget(timeout_ms));
    return cudaGetLastError();
}

}  // namespace

cudaError_t product_tc_diag(const TcJobDesc* jobs, int njobs, int count_bits, int sms, u32* err, int timeout_ms,
                            cudaStream_t st, int* launches, bool* taken)
{
    *taken = false;
    // every job's map before the first launch: all jobs or none
    std::vector<DiagParams> groups((size_t)((njobs + kMaxDiag - 1) / kMaxDiag));
    for (int q = 0; q < njobs; ++q) {
        DiagParams& P = groups[(size_t)(q / kMaxDiag)];
        const int j = q % kMaxDiag;
        const TcJobDesc& d = jobs[q];
        if (d.n > (u64)kRows) return cudaErrorInvalidValue;
        P.njobs = (u32)j + 1;
        P.C[j] = d.C;
        P.n[j] = d.n;
        P.W[j] = d.W;
        P.Wdev[j] = d.Wdev;
        P.ldc[j] = d.ldc;
        if (d.n && d.W && !packed_map(&P.map[j], d.X, d.n, d.W, d.stride, kStageWords, CU_TENSOR_MAP_SWIZZLE_NONE))
            return cudaSuccess;
    }
    *taken = true;
    for (const DiagParams& P : groups) {
        const cudaError_t e = count_bits == 64 ? run<u64>(P, sms, err, timeout_ms, st)
                                               : run<u32>(P, sms, err, timeout_ms, st);
        if (e != cudaSuccess) return e;
        if (launches) *launches += 1;
    }
    return cudaSuccess;
}

}  // namespace jsim
