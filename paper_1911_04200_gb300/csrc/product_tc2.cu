// Semiring product on pairs of SMs (tcgen05 with cta_group::2, sm_103a):
// C += X X^T over (AND, popcount, +) (Eq. 7), computed exactly as a 4-bit
// floating-point product (kind::mxf4: e2m1 operands, a power-of-two scale per
// 32 elements).
//
// Encoding.  A 32-bit word of a packed row becomes four words of eight 4-bit
// elements: the word masked to every nibble's bit 0, bit 1 and bit 2, and bit
// 3 shifted into bit 2.  A set bit is then the e2m1 value 0.5, 1, 2 or 2, and
// the block scales 2, 1, 1/2 and 1/2 make each of them exactly 1: an element
// word costs one AND (and one shift for the last mask), where a byte format
// spreads bits with a multiply per four of them.  The same bit goes to the
// same element in A and B, so the order of the contraction index does not
// matter.  Products are 0 or 1; an accumulation takes at most 2^22 bit-rows,
// so every FP32 accumulator is a count below 2^24, held exactly.  The scales
// are the same for every row: two 32-bit patterns of ue8m0 bytes, written once
// to 8 TMEM columns each that both operands' scale addresses name.
//
// What bounds it: the unpacking.  With both operands in shared memory an SM
// writes, and the tensor core reads, 64 KiB per 512 bit-rows of a 128 x 256
// block - all of the 128 bytes a cycle that shared memory moves in the 1024
// cycles those MMAs take - and the words' loads pass through the same pipe;
// and every instruction of the unpacking warps counts.  So (1) pairs: a 2-SM
// MMA of M = 256, N = 256 reads its B operand as 128 rows from each SM; (2)
// the A operand lives in TMEM, written with tcgen05.st, which halves the
// traffic; (3) the packed words come by TMA, a 128-byte line of every row at
// a time, so the unpacking warps spend nothing on addresses and bounds; (4)
// waits suspend in hardware instead of polling.  Measured (4096 samples,
// 65,536 words; ms): FP8 operands in shared memory, 32-byte loads per row
// 25.5; MXF4, same structure 15.5; whole-line loads 12.7; A in TMEM with
// loads through registers 12.4, with cp.async 11.4; TMA 9.6 (7.8e15
// multiply-adds x 2 per second, of 10.3e15 for K = 64 MMAs at 2070 MHz; the
// MMAs alone, with nothing unpacked, take 8.3 to 8.7, so most of what is left
// is the MMAs' own).  n = 1024 and 65,536 words: 1.6 -> 0.73 ms.  Tried: six stages of 256 bit-rows 15.2 (the
// handshake between the CTAs is paid per stage); 16 unpacking warps 11.9 to
// 12.4.
//
// A cluster of two CTAs (ranks 0 and 1) works on 256 x 256 tiles of C on or
// above the diagonal (tile rows [256 ti, +256), columns [256 tj, +256),
// ti <= tj).  Words are loaded in units of 1024 bit-rows (one line of a row)
// and unpacked in two stages of 512: CTA r unpacks A rows 256 ti + 128 r +
// [0, 128) into its TMEM and B rows 256 tj + 128 r + [0, 128) into its shared
// memory (same offsets in both CTAs).  Roles (14 warps per CTA):
//   warps 0-3   unpack A (warp w: rows 32 w .., the TMEM lanes it may write);
//   warps 4-7   unpack B; after writing a stage (and, for B, fencing for the
//               async proxy) one lane per warp arrives on `full` (rank 0) or
//               on the local `ready` (rank 1), whose completion the rank-1
//               signal thread forwards to the rank-0 `full` (one cluster-scope
//               release per stage, 9 arrivals);
//   warp 8      rank 1: the signal thread; rank 0: one lane issues 8 tcgen05.mma
//               (cta_group::2, M = 256, N = 256, K = 64) per stage into the
//               TMEM accumulator and commits them, multicast to both CTAs, to
//               `empty` (stage reusable) and, per finished accumulation, to
//               `acc_full`;
//   warps 9-12  epilogue in both CTAs: copy this CTA's 128 accumulator rows
//               to shared memory, arrive (a lane per warp) on the rank-0
//               CTA's `acc_empty` (8 arrivals), and add the counts into C
//               row by row (32 consecutive counts per atomic instruction)
//               while the next accumulation runs;
//   warp 13     loads the units into two slots of shared memory (one thread,
//               TMA, the next unit in flight while one is unpacked).
// Rows that are not 16-byte aligned (a caller's own matrix) take the same
// path with the words copied by the unpacking warps, 8 bytes at a time.
// Every wait is bounded (clock64 budget, plus a CTA-wide abort flag); on
// time-out the CTA raises the error word, waits (bounded) for the MMAs and
// copies already issued, and both CTAs meet at a cluster barrier before TMEM
// is freed and the CTAs exit.
#include <algorithm>
#include <atomic>
#include "tensor_map.cuh"

namespace jsim {

namespace {

// L2 window shared by all clusters: kWindowMiB of packed words of all rows,
// but at least kMinUnits units per chunk.  Every tile switch drains an
// accumulator, so for many rows a window that fits L2 is too short; for few
// rows a window beyond L2 re-reads the panels from DRAM.  n = 1024 and 2^20
// words, ms: 48 MiB 13.5, 64 MiB 13.0, 64 MiB but 768 units (96 MiB) 12.8.
constexpr u64 kWindowMiB = 64;
constexpr u64 kMinUnits = 768;
constexpr int kProducerWarps = 8;                 // four unpack A, four B
constexpr int kMmaWarp = kProducerWarps;
constexpr int kEpiWarp0 = kProducerWarps + 1;
constexpr int kLoadWarp = kProducerWarps + 5;     // after the MMA warp and four epilogue warps
constexpr int kWarps = kLoadWarp + 1;
constexpr int kThreads = kWarps * 32;             // 448
constexpr int kHalf = 128;                        // A rows and B rows per CTA per tile
constexpr int kTile = 256;                        // tile side (rows and columns of C)
static_assert(kEpiWarp0 % 4 == 1, "epilogue warp e reads TMEM lanes of warp rank (kEpiWarp0 + e) % 4");
constexpr int kStageBits = 512;                   // bit-rows of a stage
constexpr int kSteps = kStageBits / 64;           // MMAs (K = 64) of a stage
constexpr int kUnitStages = 2;                    // stages unpacked from one unit of loaded words
constexpr int kUnitBits = kUnitStages * kStageBits;
constexpr int kUnitWords = kUnitBits / 64;        // 16: one 128-byte line of a row
constexpr int kWarpGroups = 4;                    // groups of 8 rows a producer warp unpacks
static_assert(kWarpGroups * 8 * (kProducerWarps / 2) == kHalf, "rows of an operand");
constexpr int kAtom = kHalf * 128;                // one 128-byte swizzle atom column (256 bit-rows) of B: 16 KiB
constexpr int kStageBytes = kStageBits / 256 * kAtom;  // 32 KiB
constexpr int kBufs = 3;
constexpr int kSlots = 2;                         // units of packed words in shared memory
constexpr int kHalfSlot = kHalf * 128;            // A rows (then B rows) of a unit: 16 KiB
constexpr int kSlotBytes = 2 * kHalfSlot;
constexpr int kRingBytes = kSlots * kSlotBytes;   // 64 KiB
constexpr int kDrainCols = kTile / 2;             // columns the epilogue copies at a time
constexpr int kDrainBytes = kHalf * kDrainCols * 4;  // 64 KiB
constexpr int kSmemBytes = kBufs * kStageBytes + kRingBytes + kDrainBytes + 1024;  // + alignment slack
static_assert(kSmemBytes + 512 <= 232448, "fits the per-CTA shared-memory limit");
// TMEM columns: the accumulator, two patterns of block scales, the A stages
constexpr int kTmemCols = 512;
constexpr u32 kScaleCol = kTile;
constexpr u32 kScaleCols = 8;                     // columns a pattern fills (B's 256 rows take 8)
constexpr u32 kACol = kScaleCol + 2 * kScaleCols;
constexpr u32 kACols = kStageBits / 8;            // columns of an A stage: 8 elements each
static_assert(kACol + kBufs * kACols <= kTmemCols, "TMEM columns");
// ue8m0 bytes: masks 0 and 1 (2, 2, 1, 1: bytes 0-1 or 2-3 by the MMA's scale
// id), masks 2 and 3 (1/2)
constexpr u32 kScales0 = 0x7f7f8080u, kScales1 = 0x7e7e7e7eu;
constexpr u64 kMaxSegUnits = (1ull << 22) / kUnitBits;
constexpr u32 kErrTimeout = 4u;

// instruction descriptor: kind::mxf4, A = B = E2M1 (1 at bits 7.. and 10..),
// both K-major, N = 256 (bits 17..22 hold N/8), ue8m0 scales (bit 23), M =
// 256 across the pair (bits 24..28 hold M/16); kScaleHigh: scale bytes 2-3 of
// both operands (id 2 at bits 4.. and 29..)
constexpr u32 kIdesc =
    (1u << 7) | (1u << 10) | ((u32)(kTile >> 3) << 17) | (1u << 23) | ((u32)(kTile >> 4) << 24);
constexpr u32 kScaleHigh = (2u << 4) | (2u << 29);

__device__ __forceinline__ u32 smem_u32(const void* p) { return (u32)__cvta_generic_to_shared(p); }

__device__ __forceinline__ u32 cta_rank()
{
    u32 r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
    return r;
}

// the same shared-memory variable in CTA `rank` of the cluster
__device__ __forceinline__ u32 peer_addr(const void* p, u32 rank)
{
    u32 r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
    return r;
}

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;\n" ::: "memory");
}

__device__ __forceinline__ u64 sw128_desc(u32 saddr)
{
    return (u64)((saddr & 0x3FFFFu) >> 4) | ((u64)1 << 16) | ((u64)(1024 >> 4) << 32) | ((u64)1 << 46) |
           ((u64)2 << 61);
}

__device__ __forceinline__ void mbar_init(u64* bar, u32 count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" :: "r"(smem_u32(bar)), "r"(count) : "memory");
}

// arrive on the barrier at cluster address `caddr` (this CTA's or the peer's)
__device__ __forceinline__ void mbar_arrive_cluster(u32 caddr)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];\n" :: "r"(caddr) : "memory");
}

__device__ __forceinline__ void mbar_arrive(u64* bar)
{
    asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" :: "r"(smem_u32(bar))
                 : "memory");
}

// Waits in hardware for the phase of `parity`, up to about kSuspendNs (no
// polling loop takes issue slots from the unpacking warps).  CLUSTER: arrivals
// come from the other CTA's threads too.
constexpr u32 kSuspendNs = 20000;
template <bool CLUSTER>
__device__ __forceinline__ bool mbar_try_wait(u64* bar, u32 parity)
{
    u32 ok;
    if (CLUSTER)
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n"
                     " selp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity), "r"(kSuspendNs) : "memory");
    else
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2, %3;\n"
                     " selp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity), "r"(kSuspendNs) : "memory");
    return ok != 0;
}

// Bounded wait; false on time-out or when another role has aborted the CTA.
template <bool CLUSTER = false>
__device__ __forceinline__ bool mbar_wait(u64* bar, u32 parity, long long budget, volatile int* abort_flag)
{
    if (mbar_try_wait<CLUSTER>(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait<CLUSTER>(bar, parity)) {
        if (*abort_flag) return false;
        if (clock64() - t0 > budget) {
            *abort_flag = 1;
            return false;
        }
    }
    return true;
}

// commit the MMAs issued so far to the barrier at `bar`'s offset in both CTAs
__device__ __forceinline__ void commit_both(u64* bar)
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n"
                 :: "r"(smem_u32(bar)), "h"((unsigned short)3) : "memory");
}

// element word `m` (0..3) of a 32-bit word
template <int M>
__device__ __forceinline__ u32 elems(u32 x)
{
    return M == 0 ? x & 0x11111111u : M == 1 ? x & 0x22222222u : M == 2 ? x & 0x44444444u : (x >> 1) & 0x44444444u;
}

// 16 lanes (rows) x 32 columns of TMEM from row groups 0 (lanes 0-7) and 1
// (lanes 8-15): v[j][g][0..1] are columns 8 j + 2 (lane % 4) + {0, 1} of row
// lane / 4 of group g
__device__ __forceinline__ void tmem_st_half(u32 taddr, const u32 (&v)[4][2][2])
{
    asm volatile("tcgen05.st.sync.aligned.16x256b.x4.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};\n"
                 :: "r"(taddr), "r"(v[0][0][0]), "r"(v[0][0][1]), "r"(v[0][1][0]), "r"(v[0][1][1]), "r"(v[1][0][0]),
                    "r"(v[1][0][1]), "r"(v[1][1][0]), "r"(v[1][1][1]), "r"(v[2][0][0]), "r"(v[2][0][1]),
                    "r"(v[2][1][0]), "r"(v[2][1][1]), "r"(v[3][0][0]), "r"(v[3][0][1]), "r"(v[3][1][0]),
                    "r"(v[3][1][1])
                 : "memory");
}

// element words of a lane's 128 bits (w0, w1), masks 2 AT and 2 AT + 1, in
// K-step order: step 4 AT + 2 q + t holds mask 2 AT + t of the word pair q
template <int AT>
__device__ __forceinline__ void expand_half(u32 (&v)[4][2][2], int g, u64 w0, u64 w1)
{
    const u32 x[2][2] = {{(u32)w0, (u32)(w0 >> 32)}, {(u32)w1, (u32)(w1 >> 32)}};
    #pragma unroll
    for (int q = 0; q < 2; ++q)
        #pragma unroll
        for (int i = 0; i < 2; ++i) {
            v[2 * q][g][i] = elems<2 * AT>(x[q][i]);
            v[2 * q + 1][g][i] = elems<2 * AT + 1>(x[q][i]);
        }
}

// 16 bytes from global to shared memory (8-byte aligned source), the bytes at
// and past `valid` as zeros
__device__ __forceinline__ void copy16(u32 dst, const u64* src, int valid)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n"
                 :: "r"(dst), "l"(src), "r"(valid < 8 ? valid : 8) : "memory");
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n"
                 :: "r"(dst + 8), "l"(valid > 8 ? src + 1 : src), "r"(valid > 8 ? valid - 8 : 0) : "memory");
}

// 128 rows x 128 bytes of the packed matrix (word x on, row y on; zeros
// outside it) to shared memory, 16-byte chunk k of a row at k ^ (row % 8)
__device__ __forceinline__ void tma_rows(u32 dst, const CUtensorMap* map, u64 x, u64 y, u64* bar)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n"
                 :: "r"(dst), "l"(map), "r"((int)x), "r"((int)y), "r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void mbar_expect(u64* bar, u32 bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" :: "r"(smem_u32(bar)), "r"(bytes) : "memory");
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

// tile t -> (ti, tj), tiles ordered column by column: tj = 0, 1, ..., ti = 0..tj
__device__ __forceinline__ void pair_tile(u64 t, u64& r0, u64& c0)
{
    u64 j = 0;
    while (t > j) {
        t -= j + 1;
        ++j;
    }
    r0 = t * kTile;
    c0 = j * kTile;
}

// Work of a cluster: the words are cut into nst units of 1024 bit-rows and
// these into chunks of L; chunk k's (tile, unit) pairs are laid out tile-major
// and cluster c takes the c-th of G equal contiguous shares; every cluster
// walks the chunks at the same pace, so the window of L units of all rows is
// shared in L2.  Odd chunks are walked from the share's last tile to its first, so a chunk
// begins with the tile the one before ended with and its accumulation runs on.
struct WorkIter {
    u64 tiles, nst, L, G, c, KC;
    u64 k, Lk, u, uend;
    __device__ __forceinline__ void init(u64 tiles_, u64 nst_, u64 L_, u64 G_, u64 c_)
    {
        tiles = tiles_; nst = nst_; L = L_; G = G_; c = c_;
        KC = (nst + L - 1) / L;
        k = ~0ull; u = uend = Lk = 0;
    }
    __device__ __forceinline__ bool next(u64& tile, u64& kst, u64& len)
    {
        while (u >= uend) {
            k = (k == ~0ull) ? 0 : k + 1;
            if (k >= KC) return false;
            Lk = min(L, nst - k * L);
            const u64 Uk = tiles * Lk;
            u = c * Uk / G;
            uend = (c + 1) * Uk / G;
        }
        if (k & 1) {
            tile = (uend - 1) / Lk;
            const u64 b = max(u, tile * Lk);
            len = uend - b;
            kst = k * L + (b - tile * Lk);
            uend = b;
        } else {
            tile = u / Lk;
            const u64 e = min(uend, (tile + 1) * Lk);
            len = e - u;
            kst = k * L + (u - tile * Lk);
            u = e;
        }
        return true;
    }
};

// Accumulations in the order the cluster makes them, walked alike by the MMA
// thread and the epilogue: a segment joins the running accumulation when it
// is of the same tile and the exactness cap allows, and starts the next one
// otherwise.
struct Accum {
    u64 tile = ~0ull, fill = 0;
    u32 f = 0;  // index of the running accumulation (valid once tile is set)
    // does a segment of `len` units of tile t start a new accumulation?
    __device__ __forceinline__ bool starts(u64 t, u64 len) const { return tile != t || fill + len > kMaxSegUnits; }
};

// TMA: the packed words come through the tensor map (16-byte aligned rows);
// otherwise the unpacking warps copy their rows 8 bytes at a time.
template <typename CT, bool TMA>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
k_prod_tc2(const __grid_constant__ CUtensorMap map, const u64* __restrict__ X, u64 stride, u64 n, u64 W,
           const u64* Wdev, u64 tiles, u64 L, CT* __restrict__ C, u64 ldc, u32* err, long long budget)
{
    if (Wdev) W = min(W, *Wdev);  // (the words up to the bound are zeros)
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) u64 full_bar[kBufs], ready_bar[kBufs], empty_bar[kBufs], ldf_bar[kSlots],
        lde_bar[kSlots], accf_bar, acce_bar, done_bar;
    __shared__ u32 tmem_slot;
    __shared__ int abort_flag;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const u32 rank = cta_rank();
    const u64 G = gridDim.x / 2, c = blockIdx.x / 2;  // clusters and this CTA's cluster
    const u64 nst = (W + kUnitWords - 1) / kUnitWords;
    // units of this cluster (the same in both CTAs)
    u64 T = 0;
    {
        const u64 KC = (nst + L - 1) / L;
        for (u64 k = 0; k < KC; ++k) {
            const u64 Uk = tiles * min(L, nst - k * L);
            T += (c + 1) * Uk / G - c * Uk / G;
        }
    }
    if (T == 0) return;  // uniform per cluster, before any TMEM, barrier or peer access

    const u32 raw = smem_u32(smem_raw);
    const u32 base = (raw + 1023u) & ~1023u;
    unsigned char* sm = smem_raw + (base - raw);

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;\n"
                     :: "r"(smem_u32(&tmem_slot)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;\n" ::: "memory");
    }
    if (tid == 32) {
        for (int b = 0; b < kBufs; ++b) {
            mbar_init(&full_bar[b], kProducerWarps + 1);  // rank-0 producer warps + the rank-1 signal
            mbar_init(&ready_bar[b], kProducerWarps);      // rank-1 producer warps
            mbar_init(&empty_bar[b], 1);
        }
        for (int y = 0; y < kSlots; ++y) {
            mbar_init(&ldf_bar[y], 1);
            mbar_init(&lde_bar[y], kProducerWarps);
        }
        mbar_init(&accf_bar, 1);
        mbar_init(&acce_bar, 2 * 4);                   // epilogue warps of both CTAs
        mbar_init(&done_bar, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const u32 tmem = tmem_slot;
    if (warp >= kEpiWarp0 && warp < kLoadWarp) {
        // the block scales, in every lane
        const u32 at = tmem + (((u32)(warp - kEpiWarp0 + 1) & 3u) * 32u << 16) + kScaleCol;
        asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%2,%2,%2,%2,%2,%2,%2,%2};\n"
                     "tcgen05.wait::st.sync.aligned;\n" :: "r"(at), "r"(kScales0), "r"(kScales1) : "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    cluster_sync();  // both CTAs' barriers and scales exist before any remote arrival or MMA
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    volatile int* abort_v = &abort_flag;

    if (warp < kProducerWarps) {
        // ---------------- unpack producers ----------------
        // A unit is a 128-byte line of every A and B row, in a slot of shared
        // memory, 16-byte chunk k of row y at k ^ (y % 8).  Lane l reads the
        // 32-byte piece l % 4 of row l / 4 of a group of 8 rows: the piece's
        // low 16 bytes for the unit's first stage, its high 16 bytes for the
        // second (which bits a stage holds is free, as long as A and B agree).
        // Of a K step's eight element words per row, lane l owns words
        // 2 (l % 4) and + 1: the layout of a 16x256b TMEM store.
        const int lr = lane >> 2, h = lane & 3;
        const bool is_a = warp < kProducerWarps / 2;
        const int r0w = (warp & 3) * 32;  // this warp's 32 rows of its operand (A: the TMEM lanes it may write)
        // B: step j of a row is the 32 bytes at chunk 2 (j % 4) of atom column
        // j / 4, chunk c stored at c ^ (row % 8) = c ^ lr.  The 16 lanes of a
        // store phase (4 rows x 4 x 8 bytes) hit all 32 banks when odd rows
        // take their word pairs the other way round (pair q is chunk bit 2).
        const u32 odd = (u32)lr & 1u;
        u32 b_off[4];
        #pragma unroll
        for (int j = 0; j < 4; ++j)
            b_off[j] = (u32)((r0w + lr) * 128 + 8 * (h & 1)) + ((((u32)(2 * j + (h >> 1))) ^ (4u * odd) ^ (u32)lr) << 4);
        const unsigned char* rows_s = sm + kBufs * kStageBytes + (is_a ? 0 : kHalfSlot) + (r0w + lr) * 128;
        const u32 y0 = (u32)lane >> 3;  // !TMA: first row this lane copies (then every fourth)
        const u32 copy_s = smem_u32(sm + kBufs * kStageBytes + (is_a ? 0 : kHalfSlot)) + ((u32)r0w + y0) * 128;
        WorkIter fit;
        u64 f_tile = ~0ull, f_kst = 0, f_left = 0, f_r0 = 0, f_c0 = 0;
        // !TMA: start copying this warp's rows of the next unit into slot y (one
        // group of copies, empty past the end)
        auto fetch = [&](int y) {
            bool more = f_left > 0;
            if (!more) {
                u64 tile;
                more = fit.next(tile, f_kst, f_left);
                if (more && tile != f_tile) { pair_tile(tile, f_r0, f_c0); f_tile = tile; }
            }
            if (more) {
                const u64 gk = f_kst * kUnitWords + 2 * (u64)(lane & 7);
                const int left = gk < W ? (W - gk >= 2 ? 16 : 8) : 0;
                const u64 row = (is_a ? f_r0 : f_c0) + (u64)rank * kHalf + (u64)r0w + y0;
                const int rows = left == 0 || row >= n ? 0 : (int)min(n - row, (u64)kHalf);  // rows left in the matrix
                const u64* src = X + row * stride + gk;
                #pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const bool in = 4 * q < rows;
                    const u32 dst = copy_s + (u32)(y * kSlotBytes + q * 512) +
                                    ((((u32)lane & 7u) ^ ((y0 + 4 * (u32)q) & 7u)) << 4);
                    copy16(dst, in ? src : X, in ? left : 0);
                    src += 4 * stride;
                }
                --f_left;
                ++f_kst;
            }
            asm volatile("cp.async.commit_group;\n" ::: "memory");
        };
        if (!TMA) {
            fit.init(tiles, nst, L, G, c);
            for (int y = 0; y < kSlots; ++y) fetch(y);
        }
        u32 lpar = 0;  // parity of the slot's `ldf` phase
        bool ok = true;
        int b = 0, y = 0;
        u32 par = 1;  // parity of the `empty` phase before this buffer's use
        bool first = true;  // the first use of every buffer waits for none
        for (u64 t = 0; t < T && ok; ++t) {
            if (TMA) {
                ok = mbar_wait(&ldf_bar[y], lpar, budget, abort_v);
            } else {
                asm volatile("cp.async.wait_group %0;\n" :: "n"(kSlots - 1) : "memory");
                __syncwarp();
            }
            #pragma unroll
            for (int hs = 0; hs < kUnitStages; ++hs) {
                u64 w[kWarpGroups][2];  // B, odd rows: the halves swapped
                {
                    const unsigned char* src = rows_s + y * kSlotBytes + ((u32)((2 * h + hs) ^ lr) << 4);
                    #pragma unroll
                    for (int q = 0; q < kWarpGroups; ++q) {
                        if (is_a) {
                            const ulonglong2 v = *(const ulonglong2*)(src + q * 8 * 128);
                            w[q][0] = v.x;
                            w[q][1] = v.y;
                        } else {
                            w[q][0] = *(const u64*)(src + q * 8 * 128 + 8 * odd);
                            w[q][1] = *(const u64*)(src + q * 8 * 128 + 8 * (1 - odd));
                        }
                    }
                }
                if (TMA && hs + 1 == kUnitStages) {
                    // the slot has been read: the fence orders these reads
                    // before the async proxy's next write to it
                    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&lde_bar[y]);
                }
                if (ok && !first && !mbar_wait(&empty_bar[b], par, budget, abort_v)) ok = false;
                ok = __all_sync(0xffffffffu, ok);  // tcgen05.st is warp-wide
                if (!ok) break;
                if (is_a) {
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    const u32 ta = tmem + ((u32)r0w << 16) + kACol + (u32)b * kACols;
                    #pragma unroll
                    for (int q = 0; q < kWarpGroups; q += 2) {
                        const u32 tq = ta + ((u32)(8 * q) << 16);
                        u32 v[4][2][2];
                        expand_half<0>(v, 0, w[q][0], w[q][1]);
                        expand_half<0>(v, 1, w[q + 1][0], w[q + 1][1]);
                        tmem_st_half(tq, v);
                        expand_half<1>(v, 0, w[q][0], w[q][1]);
                        expand_half<1>(v, 1, w[q + 1][0], w[q + 1][1]);
                        tmem_st_half(tq + 32, v);
                    }
                    asm volatile("tcgen05.wait::st.sync.aligned;\n"
                                 "tcgen05.fence::before_thread_sync;\n" ::: "memory");
                } else {
                    unsigned char* st[4];
                    #pragma unroll
                    for (int j = 0; j < 4; ++j) st[j] = sm + b * kStageBytes + b_off[j];
                    #pragma unroll
                    for (int q = 0; q < kWarpGroups; ++q) {
                        u32 v[4][2][2];
                        expand_half<0>(v, 0, w[q][0], w[q][1]);
                        expand_half<1>(v, 1, w[q][0], w[q][1]);
                        #pragma unroll
                        for (int j = 0; j < kSteps; ++j)
                            *(uint2*)(st[j & 3] + q * 8 * 128 + (j >> 2) * kAtom) =
                                make_uint2(v[j & 3][j >> 2][0], v[j & 3][j >> 2][1]);
                    }
                    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                }
                __syncwarp();
                // rank 0: straight to the MMA's barrier; rank 1: to the local
                // barrier its signal thread forwards (one cluster-scope release
                // per stage instead of one per warp)
                if (lane == 0) mbar_arrive(rank == 0 ? &full_bar[b] : &ready_bar[b]);
                if (++b == kBufs) { b = 0; par ^= 1u; first = false; }
            }
            if (!TMA && ok) fetch(y);
            if (++y == kSlots) { y = 0; lpar ^= 1u; }
        }
        if (!TMA) asm volatile("cp.async.wait_all;\n" ::: "memory");
    } else if (warp == kMmaWarp) {
        // ---------------- MMA issuer (rank-0 CTA) ----------------
        if (rank == 0 && lane == 0) {
            WorkIter it;
            it.init(tiles, nst, L, G, c);
            Accum ac;
            u64 tile, kst, len;
            int b = 0;
            u32 par = 0;
            bool ok = true;
            while (ok && it.next(tile, kst, len)) {
                bool fresh = false;
                if (ac.starts(tile, len)) {
                    if (ac.tile != ~0ull) {
                        commit_both(&accf_bar);
                        // the accumulator has been copied out
                        if (!mbar_wait<true>(&acce_bar, ac.f & 1u, budget, abort_v)) {
                            ok = false;
                            break;
                        }
                        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                        ac.f += 1;
                    }
                    ac.tile = tile;
                    ac.fill = 0;
                    fresh = true;
                }
                for (u64 q = 0; q < len * kUnitStages; ++q) {
                    if (!mbar_wait<true>(&full_bar[b], par, budget, abort_v)) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    const u32 bbase = base + b * kStageBytes, ta = tmem + kACol + (u32)b * kACols;
                    #pragma unroll
                    for (int j = 0; j < kSteps; ++j) {
                        // K step j: masks 0-1 in atom column 0, masks 2-3 in atom column 1
                        const u64 db = sw128_desc(bbase + (j >> 2) * kAtom + (j & 3) * 32);
                        const u32 accum = (fresh && q == 0 && j == 0) ? 0u : 1u;
                        asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %5, 0;\n"
                                     " tcgen05.mma.cta_group::2.kind::mxf4.block_scale.scale_vec::2X"
                                     " [%0], [%1], %2, %3, [%4], [%4], p;\n}\n"
                                     :: "r"(tmem), "r"(ta + 8 * j), "l"(db),
                                        "r"(j < 4 && (j & 1) ? kIdesc | kScaleHigh : kIdesc),
                                        "r"(tmem + kScaleCol + (j < 4 ? 0u : kScaleCols)), "r"(accum) : "memory");
                    }
                    commit_both(&empty_bar[b]);
                    if (++b == kBufs) { b = 0; par ^= 1u; }
                }
                ac.fill += len;
            }
            if (ok && ac.tile != ~0ull) commit_both(&accf_bar);
            commit_both(&done_bar);
        } else if (rank == 1 && lane == 0) {
            // signal: forward each stage's local readiness to the MMA's barrier
            // in the rank-0 CTA (release at cluster scope, after acquiring the
            // producers' release at CTA scope)
            int b = 0;
            u32 par = 0;
            for (u64 t = 0; t < T * kUnitStages; ++t) {
                if (!mbar_wait(&ready_bar[b], par, budget, abort_v)) break;
                mbar_arrive_cluster(peer_addr(&full_bar[b], 0));
                if (++b == kBufs) { b = 0; par ^= 1u; }
            }
        }
        __syncwarp();
    } else if (warp == kLoadWarp) {
        // ---------------- packed words (both CTAs) ----------------
        if (TMA && lane == 0) {
            WorkIter it;
            it.init(tiles, nst, L, G, c);
            u64 tile, kst, len, t = 0;
            bool ok = true;
            while (ok && it.next(tile, kst, len)) {
                u64 r0, c0;
                pair_tile(tile, r0, c0);
                r0 += (u64)rank * kHalf;
                c0 += (u64)rank * kHalf;
                for (u64 q = 0; q < len; ++q, ++t) {
                    const int y = (int)(t % kSlots);
                    if (t >= kSlots && !mbar_wait(&lde_bar[y], (u32)((t / kSlots - 1) & 1), budget, abort_v)) {
                        ok = false;
                        break;
                    }
                    mbar_expect(&ldf_bar[y], kSlotBytes);
                    const u32 dst = base + kBufs * kStageBytes + y * kSlotBytes;
                    tma_rows(dst, &map, (kst + q) * kUnitWords, r0, &ldf_bar[y]);
                    tma_rows(dst + kHalfSlot, &map, (kst + q) * kUnitWords, c0, &ldf_bar[y]);
                }
            }
            // no copy of this CTA is in flight when it ends (bounded)
            for (u64 q = t > kSlots ? t - kSlots : 0; q < t; ++q) {
                const long long t0 = clock64();
                while (!mbar_try_wait<false>(&ldf_bar[q % kSlots], (u32)((q / kSlots) & 1)))
                    if (clock64() - t0 > budget) { *abort_v = 1; break; }
            }
        }
        __syncwarp();
    } else {
        // ---------------- epilogue (both CTAs) ----------------
        const int e = (warp - kEpiWarp0 + 1) & 3;  // TMEM lane quarter of this warp (warp % 4)
        // this warp's 32 rows of the copy of half an accumulator: row y at
        // y * 512 bytes, 16-byte chunk k at k ^ (y % 8)
        unsigned char* copy = sm + kBufs * kStageBytes + kRingBytes + e * 32 * (kDrainCols * 4);
        auto drain = [&](u32 f, u64 tile) -> bool {
            int got = 0;
            if (lane == 0) got = mbar_wait(&accf_bar, f & 1u, budget, abort_v) ? 1 : 0;
            got = __shfl_sync(0xffffffffu, got, 0);
            if (!got) return false;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            u64 r0, c0;
            pair_tile(tile, r0, c0);
            #pragma unroll 1
            for (int half = 0; half < kTile / kDrainCols; ++half) {
                #pragma unroll 1
                for (int cb = 0; cb < kDrainCols / 32; ++cb) {
                    u32 r[32];
                    tmem_ld32(tmem + ((u32)(e * 32) << 16) + (u32)(half * kDrainCols + cb * 32), r);
                    #pragma unroll
                    for (int x = 0; x < 8; ++x)
                        *(uint4*)(copy + lane * (kDrainCols * 4) + (((8 * cb + x) ^ (lane & 7)) << 4)) =
                            make_uint4((u32)__uint_as_float(r[4 * x]), (u32)__uint_as_float(r[4 * x + 1]),
                                       (u32)__uint_as_float(r[4 * x + 2]), (u32)__uint_as_float(r[4 * x + 3]));
                }
                if (half + 1 == kTile / kDrainCols) {
                    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(peer_addr(&acce_bar, 0));
                }
                __syncwarp();
                #pragma unroll 2
                for (int y = 0; y < 32; ++y) {
                    const u64 i = r0 + (u64)rank * kHalf + (u64)(e * 32 + y);
                    if (i >= n) break;
                    #pragma unroll
                    for (int cb = 0; cb < kDrainCols / 32; ++cb) {
                        const int k = 8 * cb + (lane >> 2);
                        const u32 v = *(const u32*)(copy + y * (kDrainCols * 4) + ((k ^ (y & 7)) << 4) + 4 * (lane & 3));
                        const u64 j = c0 + (u64)(half * kDrainCols + cb * 32 + lane);
                        if (j < n && i <= j && v) atomicAdd(C + i * ldc + j, (CT)v);
                    }
                }
                __syncwarp();
            }
            return true;
        };
        WorkIter it;
        it.init(tiles, nst, L, G, c);
        Accum ac;
        u64 tile, kst, len;
        bool ok = true;
        while (ok && it.next(tile, kst, len)) {
            if (ac.starts(tile, len)) {
                if (ac.tile != ~0ull) {
                    ok = drain(ac.f, ac.tile);
                    ac.f += 1;
                }
                ac.tile = tile;
                ac.fill = 0;
            }
            ac.fill += len;
        }
        if (ok && ac.tile != ~0ull) drain(ac.f, ac.tile);
    }

    // every MMA of the pair has completed (bounded wait), both CTAs are done
    // with each other's barriers, then TMEM is freed
    if (warp == 0) {
        long long t0 = clock64();
        while (!mbar_try_wait<false>(&done_bar, 0u)) {
            if (clock64() - t0 > budget) { *abort_v = 1; break; }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (tid == 0 && *abort_v) atomicOr(err, kErrTimeout);
    cluster_sync();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;\n" :: "r"(tmem), "r"(kTmemCols)
                     : "memory");
    }
}

template <typename CT, bool TMA>
cudaError_t run(ProductArgs& a, const CUtensorMap& map, cudaStream_t st)
{
    const u64 TT = (a.n + kTile - 1) / kTile;
    const u64 tiles = TT * (TT + 1) / 2;
    const u64 nst = (a.W + kUnitWords - 1) / kUnitWords;
    const u64 total = tiles * nst;
    if (total == 0) return cudaSuccess;
    u64 L = (kWindowMiB << 20) / ((u64)kUnitWords * 8ull * std::max<u64>(a.n, 1));
    L = std::max<u64>(kMinUnits, std::min<u64>(L, kMaxSegUnits));
    cudaError_t e = cudaFuncSetAttribute(k_prod_tc2<CT, TMA>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (e != cudaSuccess) return e;
    // as many clusters as can be resident at once (a GPC with an odd number
    // of free SMs leaves one unused), so no cluster waits for another's SMs
    int dev = 0;
    cudaGetDevice(&dev);
    static std::atomic<int> resident_by_dev[kMaxDevices];
    int resident = dev < kMaxDevices ? resident_by_dev[dev].load(std::memory_order_relaxed) : 0;
    if (resident == 0) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3((unsigned)a.sms & ~1u);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = kSmemBytes;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int nc = 0;
        if (cudaOccupancyMaxActiveClusters(&nc, k_prod_tc2<CT, TMA>, &cfg) != cudaSuccess || nc < 1) {
            cudaGetLastError();
            nc = a.sms / 2;
        }
        resident = nc;
        if (dev < kMaxDevices) resident_by_dev[dev].store(nc, std::memory_order_relaxed);
    }
    const u64 clusters = std::min<u64>((u64)std::min(resident, a.sms / 2), total);
    k_prod_tc2<CT, TMA><<<(unsigned)(2 * clusters), kThreads, kSmemBytes, st>>>(map, a.X, a.stride, a.n, a.W, a.Wdev, tiles, L,
                                                                          (CT*)a.C, a.ldc, a.err, wait_budget(a.timeout_ms));
    a.launches += 1;
    return cudaGetLastError();
}

}  // namespace

cudaError_t product_tc_pair(ProductArgs& a, cudaStream_t st)
{
    CUtensorMap map{};
    if (packed_map(&map, a.X, a.n, a.W, a.stride, kUnitWords, CU_TENSOR_MAP_SWIZZLE_128B))
        return a.count_bits == 64 ? run<u64, true>(a, map, st) : run<u32, true>(a, map, st);
    return a.count_bits == 64 ? run<u64, false>(a, map, st) : run<u32, false>(a, map, st);
}

}  // namespace jsim
