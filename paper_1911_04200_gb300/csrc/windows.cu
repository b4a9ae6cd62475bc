// Windowed construction of the block-sparse path's row classes and class
// matrices: the filter f^(l) of every tile of samples (Eq. 5), the class
// ranks (Eq. 6) and the bitmask compression (Sec. III-B), built range by
// range in shared memory.
//
// A row batch [lo, lo + m) is cut into windows of 2^wl rows.  A sample's
// values are sorted, so its values in a run of rows are one segment.  Set
// sizes vary by two decades, so both passes treat the segments of a tile's
// samples in their run of rows as one flat list of aligned 32-byte pieces of
// four values, split evenly over the warps, one piece a lane and step: a
// lane's position tells its sample (the segments' running starts lie in
// shared memory), no lane idles on a short segment, every load is one full
// sector, and nothing is paid per sample but its two cursors.  What bounds
// them (1024 clade samples, 1.3e9 values, 20 values a sample and window of
// 2^16 rows): pass 1 instruction issue and the values' latency (3.6 ms, 4.1
// TB/s); pass 2 the shared-memory pipe (about 11 cycles of it per 32 values
// and lookup) and the latency of its phases (7.9 ms, 3.3 TB/s), which the
// next tile's loads beside this tile's stores shorten.  Measured on the whole
// call, ms of passes 1 and 2: a warp per sample and range 5.9 + 13.0; a flat
// list of single values 6.5 + 11.8; runs of four values a lane, loaded word
// by word 5.0 + 12.2; aligned pieces in one 32-byte load 3.9 + 9.9 (one CTA
// per range and tile in pass 2); cheaper list entries and one CTA per range,
// its class-0 words placed once for all tiles 3.6 + 9.0; loads beside the
// stores, nothing spilled 3.6 + 7.9 (64 bytes of spills in that loop cost 1.8
// ms: a spilled load waits for its value).  The cursors take 1.4.  Also
// tried in pass 2: ranges of 1 and 4 windows 10.6 and 10.4 against 9.9 (2);
// three pieces a lane in flight 10.2 against 9.9; L2 prefetch of the next
// tile's values 8.5 against 7.9.
//
// k_win_cursors: every sample's position at each group of windows.  Pass 1
// (k_win_tiles, one CTA per group and tile): the tile's filter bitmap of the
// group is set in shared memory and stored, and every sample's position at
// each range of pass 2 noted where its values cross into the range.
// k_win_classify (one CTA per window) classifies the rows - class 0: held by
// two or more tiles; class 1 + t: by tile t alone (with the two-or-more
// filter, by two or more of its samples) - and writes every class word's
// rank within its window and every class's rows per window; k_win_agg sums
// the counts per range.
//
// Ranks: a class's rows are numbered in row order, range after range, and
// each range's count is rounded up to a multiple of 64 - the rows in between
// are zero rows of the packed matrix, which add nothing to C (Eq. 4) - so
// that every packed word belongs to one range.
//
// Pass 2 (k_win_pack, one CTA per range, tile after tile): the tile's samples
// are packed into the class-0 matrix XM and the tile's matrix XS.  A value's
// class and rank come from the range's class words and ranks in shared
// memory; the words of a group of samples (as many as fit, usually the whole
// tile) are gathered there too and stored whole with plain stores.  Every
// word of the batch's part of XM and XS is written exactly once, zero words
// included, so nothing is zeroed beforehand and no global atomics are
// needed.
#include "ingest_dev.cuh"

namespace jsim {

namespace {

constexpr int kWinThreads = 512;
constexpr u32 kRun = 4;           // values of a piece: 32 aligned bytes
constexpr int kClassThreads = 512;
constexpr int kCursChunk = 8;     // consecutive cursors a thread of k_win_cursors finds
constexpr u64 kWinTile = 128;     // samples per tile
constexpr int kMaxClasses = 17;   // class 0 and up to 16 tiles'
constexpr u32 kRoundLen = 1u << 24;     // values of a segment listed at a time (128 of them fit 32-bit positions)
constexpr u32 kStageWords = 5120;       // words gathered at a time in pass 2 (40 KiB)

// The values as 32-byte pieces: piece p is ids[4 p - ph .. 4 p - ph + 3], ph
// the values that ids lies past a 32-byte boundary.
struct Values {
    const u64* ids;
    u64 n;
    u32 ph;
};

// The flat list of up to 128 segments [a, b) of ids, in pieces (a segment's
// first and last piece may hold other values too): segment k's pieces are
// list entries [beg, end).
struct Segment {
    u32 beg, end;
    u32 words;  // list entry f of the segment holds values up to word words - 4 f of its piece
    u32 skip;   // words of other values in its first piece
};
struct PieceList {
    Segment seg[kWinTile];
    const u64* ptr[kWinTile];  // list entry f is the 32 bytes at ptr + 4 f
    u64 a[kWinTile];
    u32 scan[kWinTile / 32];
};

// Listing, in two parts around a barrier: values [r kRoundLen, (r + 1)
// kRoundLen) of every segment whose thread (0 .. 127) has a < b.  count
// returns what place needs; place returns the list's length.  The list may be
// read after a barrier that follows, and rebuilt after another.
struct Listing {
    u64 a;
    u32 len, runs, inc;
};
__device__ __forceinline__ Listing list_count(PieceList& L, const Values& v, u64 a, u64 b, u32 r)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    Listing x{0, 0, 0, 0};
    if (tid < (int)kWinTile) {
        x.a = min(b, a + (u64)r * kRoundLen);
        x.len = (u32)min(b - x.a, (u64)kRoundLen);
        x.runs = x.len ? (u32)(((x.a + x.len - 1 + v.ph) >> 2) - ((x.a + v.ph) >> 2)) + 1 : 0;
        x.inc = x.runs;
        #pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const u32 y = __shfl_up_sync(0xffffffffu, x.inc, o);
            if (lane >= o) x.inc += y;
        }
        if (lane == 31) L.scan[warp] = x.inc;
    }
    return x;
}
__device__ __forceinline__ u32 list_place(PieceList& L, const Values& v, const Listing& x)
{
    const int tid = threadIdx.x, warp = tid >> 5;
    u32 total = 0, before = 0;
    #pragma unroll
    for (int w = 0; w < (int)kWinTile / 32; ++w) {
        if (w < warp) before += L.scan[w];
        total += L.scan[w];
    }
    if (tid < (int)kWinTile) {
        const u32 beg = before + x.inc - x.runs, skip = (u32)(x.a + v.ph) & 3u;
        L.seg[tid] = Segment{beg, beg + x.runs, 4 * beg + skip + x.len, skip};
        L.ptr[tid] = v.ids + ((long long)((x.a + v.ph) >> 2) * 4 - (long long)v.ph - 4ll * beg);
        L.a[tid] = x.a;
    }
    return total;
}

// A lane's walk through a list, forward: its segment k, its piece's address
// and the words [lo, hi) of the piece that belong to the segment.
struct Walk {
    u32 k, lo, hi;
    Segment sg;
    const u64* ptr;
    const u64* at;
    // at list position f (below the list's length)
    __device__ __forceinline__ void init(const PieceList& L, u32 f)
    {
        u32 l = 0, h = kWinTile - 1;
        while (l < h) {
            const u32 mid = (l + h + 1) >> 1;
            if (L.seg[mid].beg <= f) l = mid; else h = mid - 1;
        }
        k = l;
        sg = L.seg[k];
        ptr = L.ptr[k];
    }
    __device__ __forceinline__ void to(const PieceList& L, u32 f)
    {
        if (f >= sg.end) {
            do {
                ++k;
                sg = L.seg[k];
            } while (f >= sg.end);
            ptr = L.ptr[k];
        }
        at = ptr + 4ull * f;
        lo = f == sg.beg ? sg.skip : 0;
        hi = min(kRun, sg.words - 4 * f);
    }
};

// The low words of a piece's four values (with edge, where a list may reach
// either end of ids, a piece that does is read value by value).
__device__ __forceinline__ void load_piece(const Values& v, const Walk& w, bool edge, u32 (&x)[kRun])
{
    if (!edge || (w.at >= v.ids && w.at + kRun <= v.ids + v.n)) {
        u64 y[kRun];
        asm volatile("ld.global.nc.v4.u64 {%0,%1,%2,%3}, [%4];\n"
                     : "=l"(y[0]), "=l"(y[1]), "=l"(y[2]), "=l"(y[3]) : "l"(w.at));
        #pragma unroll
        for (u32 i = 0; i < kRun; ++i) x[i] = (u32)y[i];
    } else {
        #pragma unroll
        for (u32 i = 0; i < kRun; ++i) x[i] = i >= w.lo && i < w.hi ? (u32)w.at[i] : 0u;
    }
}

// Rows of a piece's values: those outside [lo, hi) take the nearest one
// inside (a bit set twice is set once).
__device__ __forceinline__ void rows_of(u32 (&x)[kRun], u32 lo, u32 hi, u32 origin, u32 mask)
{
    #pragma unroll
    for (u32 i = 0; i < kRun; ++i) x[i] = (x[i] - origin) & mask;
    #pragma unroll
    for (int i = (int)kRun - 2; i >= 0; --i) x[i] = (u32)i < lo ? x[i + 1] : x[i];
    #pragma unroll
    for (u32 i = 1; i < kRun; ++i) x[i] = i >= hi ? x[i - 1] : x[i];
}

// Does the segment [a, b) reach a first or last piece of ids?
__device__ __forceinline__ bool at_edge(const Values& v, u64 a, u64 b) { return a < b && (a < kRun || b + kRun > v.n); }

// Every sample's position at the start of each group of g.gw windows (and at
// the batch end): gcurs[g n + k] for entry k of the plan.  A thread bisects
// for its first group and gallops on from there, by the sample's mean
// distance.
__global__ void k_win_cursors(const u64* __restrict__ ids, Plan plan, WinGeom g, u64* __restrict__ gcurs)
{
    const u32 i = blockIdx.x * blockDim.x + threadIdx.x, c = i / (u32)g.n, k = i - c * (u32)g.n;
    const u64 g0 = (u64)c * kCursChunk, g1 = min(g0 + kCursChunk, g.NG);
    if (g0 >= g.NG) return;
    const u64 b = plan.beg[k], e = b + plan.len[k];
    const u64 mean = (e - b) / g.NG + 1;
    u64 pos = b;
    for (u64 gi = g0; gi < g1; ++gi) {
        const u64 bound = g.lo + ((gi * g.gw) << g.wl);
        if (gi == g0) {
            pos = gi ? lower_bound_u64(ids, b, e, bound) : b;
        } else {
            // from the expected place outward in steps of a sector, then 2, 4 .. of them
            u64 lo = pos, hi = min(e, pos + mean), step = 4;
            if (hi < e && ids[hi] < bound) {
                do {
                    lo = hi + 1;
                    hi = min(e, lo + step);
                    step *= 2;
                } while (hi < e && ids[hi] < bound);
            } else {
                while (hi > lo + step && ids[hi - step] >= bound) {
                    hi -= step;
                    step *= 2;
                }
                if (hi > lo + step) lo = hi - step;
            }
            pos = lower_bound_u64(ids, lo, hi, bound);
        }
        gcurs[gi * g.n + k] = pos;
    }
    if (g1 == g.NG) gcurs[g.NG * g.n + k] = e;
}

// Pass 1: CTA (group gi, tile t) = blockIdx.x (gi * T + t) sets the rows that
// tile t's samples hold in the group's windows (Eq. 5 over the tile; TWICE:
// also the rows two or more of them hold) in shared memory and stores the
// bitmaps to B (and B2), tile-major.  curs gets every sample's position at
// the start of each pass-2 range.  Shared memory: the bitmaps (64 KiB: groups
// of 8 windows, 4 with TWICE), then the list.
template <bool TWICE>
__global__ void __launch_bounds__(kWinThreads, 2)
k_win_tiles(Values v, WinGeom g, const u64* __restrict__ gcurs, u64* __restrict__ B,
            u64* __restrict__ B2, u64* __restrict__ curs)
{
    extern __shared__ __align__(16) unsigned char win_smem[];
    const u32 gi = blockIdx.x / (u32)g.T, t = blockIdx.x - gi * (u32)g.T;
    const u64 w0 = gi * g.gw, w1 = min(w0 + g.gw, g.nwin);
    const u64 rows = (w1 - w0) << g.wl;
    const u32 glo32 = (u32)(g.lo + (w0 << g.wl));
    u32* bm = reinterpret_cast<u32*>(win_smem);
    u32* bm2 = bm + (g.gw << (g.wl - 5));
    PieceList& L = *reinterpret_cast<PieceList*>(bm + (TWICE ? 2 : 1) * (g.gw << (g.wl - 5)));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const u64 k0 = t * kWinTile, m = min(kWinTile, g.n - k0);
    // pass-2 ranges of the group: r0 on; a row of the group >> rsh is its range
    const u64 r0 = w0 >> g.wpc_log;
    const u32 nr = (u32)((w1 - w0 + g.wpc - 1) >> g.wpc_log);
    const int rsh = g.wl + g.wpc_log;

    // everything the group needs first, in flight together
    u64 a = 0, b = 0;
    if (tid < m) {
        a = gcurs[gi * g.n + k0 + tid];
        b = max(a, gcurs[(gi + 1) * g.n + k0 + tid]);
    }
    {
        uint4* z = reinterpret_cast<uint4*>(bm);
        const u32 nz = (u32)((TWICE ? 2 : 1) * (g.gw << (g.wl - 5)) / 4);
        for (u32 i = tid; i < nz; i += kWinThreads) z[i] = make_uint4(0u, 0u, 0u, 0u);
    }
    if (tid < m) {
        // the ranges no value crosses into start at the segment's end
        curs[r0 * g.n + k0 + tid] = a;
        for (u32 r = 1; r < nr; ++r) curs[(r0 + r) * g.n + k0 + tid] = b;
        if (w1 == g.nwin) curs[g.G * g.n + k0 + tid] = b;
    }
    // Rows are taken modulo the bitmap: a row outside the group only comes
    // from unsorted input, whose results are dropped.
    const u32 mask = (u32)(g.gw << g.wl) - 1;
    auto walk = [&](bool edge, u32 F, u32 rd) {
        const u32 cw = (F + kWinThreads - 1) / kWinThreads * 32;  // a warp's share: whole steps of a piece a lane
        const u32 f0 = warp * cw, f1 = min(F, f0 + cw);
        if (f0 >= f1) return;
        Walk wk;
        wk.init(L, min(f0 + lane, f1 - 1));
        wk.to(L, min(f0 + lane, f1 - 1));
        u32 nx[kRun];  // the next piece's values, loaded ahead
        load_piece(v, wk, edge, nx);
        u32 cd = 0;    // the row before the step's first piece
        if (lane == 0 && f0 != wk.sg.beg) cd = ((u32)wk.at[-1] - glo32) & mask;
        for (u32 f = f0 + lane; f - lane < f1; f += 32) {
            u32 x[kRun];
            #pragma unroll
            for (u32 i = 0; i < kRun; ++i) x[i] = nx[i];
            rows_of(x, wk.lo, wk.hi, glo32, mask);
            const u32 k = wk.k, lo = wk.lo;
            const u64* at = wk.at;
            const bool in = f < f1, first = f == wk.sg.beg;
            // the row before the piece, if it is of the sample's segment of the
            // group (else 0: the first range's start)
            u32 pd = __shfl_up_sync(0xffffffffu, x[kRun - 1], 1);
            if (lane == 0) pd = cd;
            cd = __shfl_sync(0xffffffffu, x[kRun - 1], 31);
            if (first) pd = rd > 0 ? ((u32)at[(int)lo - 1] - glo32) & mask : 0u;  // rd > 0: the list begins inside the segment
            const bool prev = !first || rd > 0;
            if (f + 32 < f1) {
                wk.to(L, f + 32);
                load_piece(v, wk, edge, nx);
            }
            if (!in) continue;
            if ((x[kRun - 1] >> rsh) > (pd >> rsh)) {
                // the values cross into further ranges
                const u64 s = (u64)(at - v.ids);
                u32 pr = pd >> rsh;
                #pragma unroll
                for (u32 i = 0; i < kRun; ++i) {
                    const u32 rg = min(x[i] >> rsh, nr - 1);
                    for (; pr < rg; ++pr) curs[(r0 + pr + 1) * g.n + k0 + k] = s + max(i, lo);
                }
            }
            #pragma unroll
            for (u32 i = 0; i < kRun; ++i) {
                const u32 d = x[i], bit = 1u << (d & 31);
                if (TWICE) {
                    if (i ? d != x[i - 1] : !prev || d != pd) {
                        const u32 old = atomicOr(bm + (d >> 5), bit);
                        if (old & bit) atomicOr(bm2 + (d >> 5), bit);
                    }
                } else {
                    atomicOr(bm + (d >> 5), bit);
                }
            }
        }
    };
    for (u32 rd = 0;; ++rd) {
        const Listing x = list_count(L, v, a, b, rd);
        const bool edge = __syncthreads_or(at_edge(v, a, b));
        const u32 F = list_place(L, v, x);
        const int more = __syncthreads_or(b - a > (u64)(rd + 1) * kRoundLen);  // segments beyond this round
        walk(edge, F, rd);
        __syncthreads();  // the list is rebuilt, the bitmaps are stored
        if (!more) break;
    }
    const u32 n16 = (u32)(rows >> 7);
    const uint4* b16 = reinterpret_cast<const uint4*>(bm);
    uint4* out = reinterpret_cast<uint4*>(B + t * g.nw + (w0 << (g.wl - 6)));
    for (u32 j = tid; j < n16; j += kWinThreads) out[j] = b16[j];
    if (TWICE) {
        const uint4* c16 = reinterpret_cast<const uint4*>(bm2);
        uint4* out2 = reinterpret_cast<uint4*>(B2 + t * g.nw + (w0 << (g.wl - 6)));
        for (u32 j = tid; j < n16; j += kWinThreads) out2[j] = c16[j];
    }
}

// Classes of window w's rows = blockIdx.x from the tiles' bitmaps: class 0
// = rows of two or more tiles, class 1 + t = rows of tile t alone (with the
// two-or-more filter: rows tile t holds twice or more and no other tile
// holds); the class words, every word's rank within the window (the class's
// rows of the window below the word, 16 bits: a window has at most 2^16
// rows), and the window's rows per class.  Thread i takes the window's words
// 2 i and 2 i + 1, every tile's in registers (up to MT tiles), so each is
// read once; the counts of three classes share a 64-bit scan, and all scans
// one pair of barriers.
template <int MT>
__global__ void __launch_bounds__(kClassThreads)
k_win_classify(const u64* __restrict__ B, const u64* __restrict__ B2, WinGeom g, u64* __restrict__ cls,
               unsigned short* __restrict__ pre, u32* __restrict__ cnt)
{
    constexpr int kScans = (MT + 3) / 3;  // of MT + 1 classes, three a scan (fields of 21 bits)
    __shared__ u64 s_scan[kScans][kClassThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const u64 w = blockIdx.x, W64 = 1ull << (g.wl - 6);
    const u64 j0 = w * W64 + 2 * (u64)tid;
    const bool mine = 2 * (u64)tid < W64;
    ulonglong2 c[MT + 1];
    {
        ulonglong2 ones = make_ulonglong2(0, 0), twos = ones;
        #pragma unroll
        for (int q = 0; q < MT; ++q) {
            const ulonglong2 v = mine && q < (int)g.T ? *(const ulonglong2*)(B + q * g.nw + j0) : make_ulonglong2(0, 0);
            twos.x |= ones.x & v.x;
            twos.y |= ones.y & v.y;
            ones.x |= v.x;
            ones.y |= v.y;
            c[q + 1] = v;
        }
        c[0] = twos;
        #pragma unroll
        for (int q = 0; q < MT; ++q) {
            if (B2 && mine && q < (int)g.T) c[q + 1] = *(const ulonglong2*)(B2 + q * g.nw + j0);
            c[q + 1].x &= ~twos.x;
            c[q + 1].y &= ~twos.y;
        }
    }
    u64 own[kScans], inc[kScans];
    #pragma unroll
    for (int s = 0; s < kScans; ++s) {
        u64 packed = 0;
        #pragma unroll
        for (int f = 0; f < 3; ++f)
            if (3 * s + f <= MT) packed |= (u64)(__popcll(c[3 * s + f].x) + __popcll(c[3 * s + f].y)) << (21 * f);
        own[s] = packed;
        u64 x = packed;
        #pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const u64 y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        inc[s] = x;
        if (lane == 31) s_scan[s][warp] = x;
    }
    __syncthreads();
    if (warp == 0) {
        #pragma unroll
        for (int s = 0; s < kScans; ++s) {
            u64 x = lane < kClassThreads / 32 ? s_scan[s][lane] : 0;
            #pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const u64 y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (lane < kClassThreads / 32) s_scan[s][lane] = x;
        }
    }
    __syncthreads();
    #pragma unroll
    for (int q = 0; q <= MT; ++q) {
        if (q > (int)g.T) break;
        const int s = q / 3, sh = 21 * (q % 3);
        const u64 ex = (warp ? s_scan[s][warp - 1] : 0) + inc[s] - own[s];
        const u32 run = (u32)(ex >> sh) & 0x1fffffu;
        if (mine) {
            *(ulonglong2*)(cls + q * g.nw + j0) = c[q];
            *(ushort2*)(pre + q * g.nw + j0) =
                make_ushort2((unsigned short)run, (unsigned short)(run + (u32)__popcll(c[q].x)));
        }
        if (tid == 0) cnt[q * g.nwin + w] = (u32)(s_scan[s][kClassThreads / 32 - 1] >> sh) & 0x1fffffu;
    }
}

// Every range's rows per class, rounded up to 64 (one thread per class and
// range), and the rows of all classes into plan.totals.
__global__ void k_win_agg(const u32* __restrict__ cnt, WinGeom g, Plan plan, u64* __restrict__ agg)
{
    const u32 i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (g.T + 1) * g.G) return;
    const u32 c = i / (u32)g.G, r = i - c * (u32)g.G;
    const u64 w0 = r * g.wpc, w1 = min(w0 + g.wpc, g.nwin);
    u64 s = 0;
    for (u64 w = w0; w < w1; ++w) s += cnt[c * g.nwin + w];
    agg[i] = (s + 63) / 64 * 64;
    if (s) atomicAdd((unsigned long long*)(plan.totals + kPlanRowsTotal), (unsigned long long)s);
}

// Pass 2: CTA r = blockIdx.x packs range r, tile after tile.  Shared memory:
// per class (0, and 1 + t of the tile at hand) and 32 rows the class bits and
// the place of the first of them among a sample's gathered bits, then the
// gathered words, then the list.  A value costs one or two of these lookups
// and one shared OR.  A tile's class words, ranks and cursors are loaded
// while the words of the tile before are stored.
__global__ void __launch_bounds__(kWinThreads, 2)
k_win_pack(Values v, WinGeom g, const u64* __restrict__ cls,
           const unsigned short* __restrict__ pre, const u32* __restrict__ cnt, const u64* __restrict__ boff,
           const u64* __restrict__ curs, const u64* __restrict__ kbase, u64* XM, u64 stride_m, u64* XS, u64 stride_s)
{
    extern __shared__ __align__(16) unsigned char win_smem[];
    const u32 r = blockIdx.x, T = (u32)g.T;
    const u64 w0 = (u64)r << g.wpc_log, w1 = min(w0 + g.wpc, g.nwin);
    const u32 nwr = (u32)(w1 - w0), RW = nwr << (g.wl - 6);  // the range's windows and words per class
    uint2* e0 = reinterpret_cast<uint2*>(win_smem);
    uint2* e1 = e0 + (g.wpc << (g.wl - 5));
    u64* stage = reinterpret_cast<u64*>(e1 + (g.wpc << (g.wl - 5)));
    u32* stage32 = reinterpret_cast<u32*>(stage);
    PieceList& L = *reinterpret_cast<PieceList*>(stage + kStageWords);
    // per class: rows of the range's windows; the range's first word in the class's matrix
    __shared__ u32 s_cnt[kMaxClasses][kMaxWinPerRange];
    __shared__ u64 s_at[kMaxClasses];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wsh = g.wl - 6;  // words of a window = 1 << wsh

    // words and ranks of class c: kWords words a thread, in flight together
    constexpr u32 kWords = 4;  // (a range of 2^17 rows has 2048)
    u64 cw[kWords];
    u32 cp[kWords];
    auto load_class = [&](u32 c) {
        const u64* w = cls + (c * g.nw + (w0 << wsh));
        const unsigned short* q = pre + (c * g.nw + (w0 << wsh));
        #pragma unroll
        for (u32 i = 0; i < kWords; ++i) {
            const u32 j = tid + i * kWinThreads;
            if (j < RW) {
                cw[i] = w[j];
                cp[i] = q[j];
            }
        }
    };
    // .. into e, the class's bits placed from bit `base` of a sample's gathered words
    auto place_class = [&](uint2* e, u32 c, bool any, u32 base) {
        #pragma unroll
        for (u32 i = 0; i < kWords; ++i) {
            const u32 j = tid + i * kWinThreads;
            if (j < RW) {
                const u64 w = any ? cw[i] : 0;
                const u32 p = base + (j >> wsh ? s_cnt[c][0] : 0) + cp[i];
                reinterpret_cast<uint4*>(e)[j] = make_uint4((u32)w, p, (u32)(w >> 32), p + (u32)__popc((u32)w));
            }
        }
    };
    u64 a = 0, b = 0;  // (b is raised to a where they are used: unsorted input)
    auto load_cursors = [&](u32 t) {
        a = b = 0;
        if (tid < (int)kWinTile && t * kWinTile + tid < g.n) {
            a = curs[r * g.n + t * kWinTile + tid];
            b = curs[(r + 1) * g.n + t * kWinTile + tid];
        }
    };
    load_class(0);
    if (tid < (int)(T + 1)) {
        #pragma unroll
        for (u32 w = 0; w < kMaxWinPerRange; ++w) s_cnt[tid][w] = w < nwr ? cnt[tid * g.nwin + w0 + w] : 0;
        s_at[tid] = kbase[tid] + (boff[tid * g.G + r] - boff[tid * g.G]) / 64;  // ranges start on whole words
    }
    load_cursors(0);
    __syncthreads();
    auto words_of = [&](u32 c) { return (s_cnt[c][0] + s_cnt[c][1] + 63) / 64; };
    const u32 q0 = XM ? words_of(0) : 0;
    place_class(e0, 0, q0 > 0, 0);
    load_class(1);
    // rows modulo the range (see pass 1): a row has a place only where its class bit is set
    const u32 rlo32 = (u32)(g.lo + (w0 << g.wl)), mask = (nwr << g.wl) - 1;

    for (u32 t = 0; t < T; ++t) {
        const u32 m = (u32)min(kWinTile, g.n - t * kWinTile);
        const u32 q1 = XS ? words_of(1 + t) : 0, Lw = q0 + q1;
        auto load_next = [&]() {
            if (t + 1 < T) {
                load_class(2 + t);
                load_cursors(t + 1);
            }
        };
        if (Lw == 0) {  // nothing of this tile in the range
            load_next();
            continue;
        }
        // samples gathered at a time: all, or as many as fit (Lw <= 2 * 2048 words: at least one)
        const u32 gs = m * Lw <= kStageWords ? m : kStageWords / Lw;
        // (the stores of the tile before read only the gathered words)
        b = max(a, b);
        const Listing x0 = list_count(L, v, a, b, 0);
        place_class(e1, 1 + t, q1 > 0, q0 * 64);
        const bool edge = __syncthreads_or(at_edge(v, a, b));
        for (u32 i = tid; i < (min(m, gs) * Lw + 1) / 2; i += kWinThreads)
            reinterpret_cast<uint4*>(stage)[i] = make_uint4(0u, 0u, 0u, 0u);
        const u32 F0 = list_place(L, v, x0);
        const bool whole = !__syncthreads_or(gs < m || b - a > kRoundLen);
        // the listed values into the gathered words of samples g0 on
        auto gather = [&](u32 F, u32 g0) {
            const u32 cs = (F + kWinThreads - 1) / kWinThreads * 32;  // a warp's share: whole steps of a piece a lane
            const u32 f1 = min(F, (warp + 1) * cs);
            u32 f = warp * cs + lane;
            if (f >= f1) return;
            Walk wk;
            wk.init(L, f);
            wk.to(L, f);
            u32 nx[kRun];  // the next piece's values, loaded ahead
            load_piece(v, wk, edge, nx);
            while (f < f1) {
                u32 x[kRun];
                #pragma unroll
                for (u32 i = 0; i < kRun; ++i) x[i] = nx[i];
                rows_of(x, wk.lo, wk.hi, rlo32, mask);
                u32* to = stage32 + (wk.k - g0) * 2 * Lw;
                f += 32;
                if (f < f1) {
                    wk.to(L, f);
                    load_piece(v, wk, edge, nx);
                }
                #pragma unroll
                for (u32 i = 0; i < kRun; ++i) {
                    // class 0 if two or more tiles hold the row, else the tile's
                    // class if the row is kept there
                    const u32 d = x[i], bit = 1u << (d & 31);
                    uint2 e = e0[d >> 5];
                    if (!(e.x & bit)) e = e1[d >> 5];
                    if (e.x & bit) {
                        const u32 rk = e.y + (u32)__popc(e.x & (bit - 1));
                        atomicOr(to + (rk >> 5), 1u << (rk & 31));
                    }
                }
            }
        };
        // i / Lw by a multiplication (exact: i Lw < 2^32; Lw = 1 has no 32-bit reciprocal)
        const u32 inv = Lw > 1 ? 0xffffffffu / Lw + 1 : 0;
        for (u32 g0 = 0; g0 < m; g0 += gs) {
            const u32 g1 = min(m, g0 + gs);
            if (!whole && g0) {
                __syncthreads();  // the words of the samples before are stored
                for (u32 i = tid; i < (g1 - g0) * Lw; i += kWinThreads) stage[i] = 0ull;
            }
            int more = 1;
            for (u32 rd = 0; more; ++rd) {
                u32 F = F0;
                if (whole) {
                    more = 0;
                } else {
                    __syncthreads();  // the list before has been walked
                    load_cursors(t);
                    b = (u32)tid >= g0 && (u32)tid < g1 ? max(a, b) : a;
                    const Listing x = list_count(L, v, a, b, rd);
                    more = __syncthreads_or(b - a > (u64)(rd + 1) * kRoundLen);
                    F = list_place(L, v, x);
                    __syncthreads();
                }
                gather(F, g0);
            }
            __syncthreads();
            if (g1 == m) load_next();
            u64* dm = XM + (t * kWinTile + g0) * stride_m + s_at[0];
            u64* ds = XS + (t * kWinTile + g0) * stride_s + s_at[1 + t];
            for (u32 i = tid; i < (g1 - g0) * Lw; i += kWinThreads) {
                const u32 y = Lw > 1 ? __umulhi(i, inv) : i, x = i - y * Lw;
                u64* row = x < q0 ? dm + y * stride_m + x : ds + y * stride_s + (x - q0);
                *row = stage[i];
            }
        }
    }
}

size_t win_tiles_smem(const WinGeom& g, bool twice)
{
    return (size_t)(twice ? 2 : 1) * ((size_t)g.gw << (g.wl - 3)) + sizeof(PieceList);
}

size_t win_pack_smem(const WinGeom& g)
{
    return 2 * ((size_t)g.wpc << (g.wl - 5)) * sizeof(uint2) + kStageWords * sizeof(u64) + sizeof(PieceList);
}

}  // namespace

WinGeom win_geom(u64 n, u64 T, u64 lo, u64 width, int wl, bool twice)
{
    WinGeom g{};
    g.n = n;
    g.T = T;
    g.lo = lo;
    g.wl = wl;
    g.nwin = width >> wl;
    g.nw = width / 64;
    g.wpc_log = 1;
    g.wpc = 2;
    g.G = (g.nwin + g.wpc - 1) / g.wpc;
    g.gw = twice ? 4 : 8;
    g.NG = (g.nwin + g.gw - 1) / g.gw;
    return g;
}

namespace {
Values values_of(const u64* ids, u64 N) { return Values{ids, N, (u32)((uintptr_t)ids / 8 % 4)}; }
}  // namespace

cudaError_t launch_win_classes(const u64* ids, u64 N, Plan plan, const WinGeom& g, bool twice, u64* B, u64* B2, u64* cls,
                               unsigned short* pre, u32* cnt, u64* agg, u64* gcurs, u64* curs, cudaStream_t st)
{
    if (g.nwin == 0) return cudaSuccess;
    const u64 searches = (g.NG + kCursChunk - 1) / kCursChunk * g.n;
    k_win_cursors<<<(unsigned)((searches + 127) / 128), 128, 0, st>>>(ids, plan, g, gcurs);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const size_t smem = win_tiles_smem(g, twice);
    const unsigned grid = (unsigned)(g.NG * g.T);
    if (twice) {
        e = cudaFuncSetAttribute(k_win_tiles<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k_win_tiles<true><<<grid, kWinThreads, smem, st>>>(values_of(ids, N), g, gcurs, B, B2, curs);
    } else {
        e = cudaFuncSetAttribute(k_win_tiles<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k_win_tiles<false><<<grid, kWinThreads, smem, st>>>(values_of(ids, N), g, gcurs, B, nullptr, curs);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const u64* b2 = twice ? B2 : nullptr;
    if (g.T <= 4) k_win_classify<4><<<(unsigned)g.nwin, kClassThreads, 0, st>>>(B, b2, g, cls, pre, cnt);
    else if (g.T <= 8) k_win_classify<8><<<(unsigned)g.nwin, kClassThreads, 0, st>>>(B, b2, g, cls, pre, cnt);
    else k_win_classify<16><<<(unsigned)g.nwin, kClassThreads, 0, st>>>(B, b2, g, cls, pre, cnt);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_win_agg<<<(unsigned)(((g.T + 1) * g.G + 255) / 256), 256, 0, st>>>(cnt, g, plan, agg);
    return cudaGetLastError();
}

cudaError_t launch_win_pack(const u64* ids, u64 N, const WinGeom& g, const u64* cls, const unsigned short* pre,
                            const u32* cnt, const u64* boff, const u64* curs, const u64* kbase, u64* XM, u64 stride_m,
                            u64* XS, u64 stride_s, cudaStream_t st)
{
    if (g.G == 0 || g.T == 0 || (!XM && !XS)) return cudaSuccess;
    const size_t smem = win_pack_smem(g);
    cudaError_t e = cudaFuncSetAttribute(k_win_pack, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_win_pack<<<(unsigned)g.G, kWinThreads, smem, st>>>(values_of(ids, N), g, cls, pre, cnt, boff, curs, kbase, XM,
                                                                 stride_m, XS, stride_s);
    return cudaGetLastError();
}

}  // namespace jsim
