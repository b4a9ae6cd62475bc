// Batched all-pairs: many independent collections per call.
//
// Each collection is one run of the paper's method (Listing 1): its own row
// batches, its own zero-row filter and prefix sum (Eq. 5, Eq. 6), its own
// bitmask words, its own product (Eq. 7, Eq. 4).  What is shared is the
// execution:
//   * one validation pass per collection, then a single host
//     synchronisation for the whole call (errors, value ranges, sizes);
//   * every row batch of every collection appends its words after the
//     previous batch's along the word axis of that collection's packed matrix
//     (a running word offset kept on the device), so no batch needs the host
//     to learn its nonzero-row count;
//   * the products of all collections run as one persistent tcgen05 launch
//     over a table of collections (or, if the tuner prefers, one CUDA-core
//     launch per collection), reading the word counts from device memory;
//   * with device-resident inputs and outputs, the whole launch sequence is
//     captured once into a CUDA graph and replayed by later calls on the same
//     collections.
// An autotuner times the candidate products (tcgen05 on SM pairs and diagonal
// tiles, tcgen05 over the table, CUDA-core with 64-bit and 32-bit words) on the
// first call of a collection shape and keeps the fastest for that shape.
#include <algorithm>
#include <memory>
#include "ctx.cuh"

namespace {

struct Col {
    u64 n = 0, N = 0;
    std::vector<u64> hoff;
    const u64* d_off = nullptr;
    const u64* d_ids = nullptr;
    u64 minid = 0, maxid = 0, mt = 0, lo0 = 0, rounds = 0;
    u64 stride = 0, n_pad = 0, max_chunks = 0;
    size_t x_off = 0, c_off = 0, s_off = 0, p_off = 0;  // offsets into the pools
    bool empty = false;
};

// Independent collections are ingested, multiplied (CUDA-core product) and
// finished on kLanes side streams at once: their kernels are small, and one
// stream would run them one after another.
constexpr int kLanes = 4;
// What a batch costs a lane whatever it holds, the lanes running beside one
// another: up to 1e7 values a collection take 2^30 rows, up to 4e6 2^31.
// Values in [0, 2^32) unless said, whole calls in 2^29-row and wider batches:
// 13 collections of 31 to 231 samples x 20,000 values 7.5 and 6.8 ms; 60 of 20
// to 120 x 20,000 in [0, 2^30) 10.7 and 10.4; 12 of 150 to 255 x 60,000 (1.2e7
// values or more each) 11.3 and 11.8, so these keep 2^29.
constexpr double kWaveBatchMs = 0.04;

// Everything one wave of collections needs on the device; kept alive by the
// graph cache so a replay finds the same addresses.
struct Wave {
    std::vector<Col> cols;
    DevBuf xpool, cpool, spool, ppool, scal, ids_pool, off_pool;
    // per lane: bitmap (the rows kept), seen (every row, filter_min 2), rank
    // directory and row count of the collection the lane is packing
    DevBuf bitmap[kLanes], seen[kLanes], dir[kLanes], bsum[kLanes], boff[kLanes], R[kLanes];
    DevBuf jobtab;          // tensor-core job table
    DevBuf cstage, jstage;  // host-output staging
    u64 max_mt = 0, batches = 0;
    int variant = JSIM_VARIANT_TC;
    int word_bits = 64;
    int tile_n = 256;       // tensor-core tile width (128 x tile_n tiles)
    cudaGraphExec_t exec = nullptr;
    u64 signature = 0;
    ~Wave()
    {
        if (exec) cudaGraphExecDestroy(exec);
    }
};

u64 mix(u64 h, u64 v)
{
    h ^= v + 0x9E3779B97F4A7C15ull + (h << 6) + (h >> 2);
    return h;
}

// the tensor-core job table of the wave (one entry per nonempty collection)
std::vector<TcJobDesc> wave_jobs(Wave& w)
{
    std::vector<TcJobDesc> jobs;
    u64* scal = w.scal.as<u64>();
    for (size_t c = 0; c < w.cols.size(); ++c) {
        const Col& cl = w.cols[c];
        if (cl.empty || cl.n == 0) continue;
        jobs.push_back(TcJobDesc{w.xpool.as<u64>() + cl.x_off, scal + 2 * c, (char*)w.cpool.p + cl.c_off,
                                 cl.stride, cl.n, 0, cl.n});
    }
    return jobs;
}

// Launch sequence of one wave after validation: zero, ingest every batch of
// every collection, product, epilogue.  No host synchronisation inside; the
// job table must already be in device memory.
int enqueue_wave(jsim_ctx* ctx, Wave& w, void* const* C, double* const* J, bool dev_out, size_t first,
                 bool run_product_only, int variant, int word_bits, int tile_n)
{
    const size_t cb = ctx->opt.count_bits == 64 ? 8 : 4;
    cudaStream_t st = ctx->stream;
    u64* scal = w.scal.as<u64>();  // per collection: ktotal, kbase
    if (!run_product_only) {
        CK(cudaMemsetAsync(w.xpool.p, 0, w.xpool.bytes, st));
        CK(cudaMemsetAsync(scal, 0, w.cols.size() * 2 * sizeof(u64), st));
        int rc = lanes_fork(ctx, kLanes);
        if (rc) return rc;
        for (size_t c = 0; c < w.cols.size(); ++c) {
            const Col& cl = w.cols[c];
            if (cl.empty) continue;
            const int ln = (int)(c % kLanes);
            cudaStream_t ls = ctx->lanes[ln];
            Plan plan;
            u64* pb = w.ppool.as<u64>() + cl.p_off;
            plan.beg = pb; plan.len = pb + cl.n; plan.cofs = pb + 2 * cl.n; plan.totals = pb + 3 * cl.n + 1;
            u64* X = w.xpool.as<u64>() + cl.x_off;
            const u64 nwords = cl.mt / 64;
            for (u64 l = 0; l < cl.rounds; ++l) {
                const u64 lo = cl.lo0 + l * cl.mt;
                CK(launch_plan(cl.d_off, cl.d_ids, cl.n, lo, lo + cl.mt, false, plan, ls));
                CK(cudaMemsetAsync(w.bitmap[ln].p, 0, nwords * sizeof(u64), ls));
                if (ctx->opt.filter_min == 2) {
                    CK(cudaMemsetAsync(w.seen[ln].p, 0, nwords * sizeof(u64), ls));
                    CK(launch_filter(cl.d_ids, cl.n, plan, cl.max_chunks, lo, cl.mt, w.seen[ln].as<u32>(), ctx->sms,
                                     ls, w.bitmap[ln].as<u32>()));
                } else {
                    CK(launch_filter(cl.d_ids, cl.n, plan, cl.max_chunks, lo, cl.mt, w.bitmap[ln].as<u32>(),
                                     ctx->sms, ls));
                }
                CK(launch_scan(w.bitmap[ln].as<u64>(), nwords, w.dir[ln].as<u32>(), w.bsum[ln].as<u64>(),
                               w.boff[ln].as<u64>(), w.R[ln].as<u64>(), ls, scal + 2 * c, scal + 2 * c + 1));
                CK(launch_pack_full(cl.d_ids, cl.n, plan, cl.max_chunks, lo, cl.mt, w.bitmap[ln].as<u64>(),
                                    w.dir[ln].as<u32>(), w.boff[ln].as<u64>(), X, cl.stride, w.R[ln].as<u64>(),
                                    ctx->sms, ls, scal + 2 * c + 1));
                ctx->stats.launches += 5;
            }
        }
        rc = lanes_join(ctx, kLanes);
        if (rc) return rc;
    }
    CK(cudaMemsetAsync(w.cpool.p, 0, w.cpool.bytes, st));
    // product: all collections
    if (variant == JSIM_VARIANT_TC) {
        std::vector<TcJobDesc> jobs = wave_jobs(w);
        int launches = 0;
        cudaError_t e = product_tc_jobs(jobs.data(), (int)jobs.size(), w.jobtab.p, false, ctx->opt.count_bits,
                                        ctx->sms, ctx->d_err, ctx->opt.timeout_ms > 0 ? ctx->opt.timeout_ms : 2000,
                                        st, &launches, tile_n);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "batched tcgen05 product");
        ctx->stats.product_launches += launches;
        ctx->stats.launches += launches;
    } else if (variant == JSIM_VARIANT_TC2) {
        // 4-bit operands: collections of one tile together, the others one by one
        const int to = ctx->opt.timeout_ms > 0 ? ctx->opt.timeout_ms : 2000;
        std::vector<TcJobDesc> small;
        for (TcJobDesc& j : wave_jobs(w)) {
            if (j.n <= 128) {
                j.W = j.stride;
                small.push_back(j);
                continue;
            }
            ProductArgs a{};
            a.X = j.X; a.stride = j.stride; a.n = j.n; a.W = j.stride; a.Wdev = j.Wdev; a.C = j.C; a.ldc = j.ldc;
            a.count_bits = ctx->opt.count_bits; a.sms = ctx->sms; a.timeout_ms = to; a.err = ctx->d_err;
            cudaError_t e = product_tc_pair(a, st);
            if (e != cudaSuccess) return cuda_fail(ctx, e, "batched SM-pair product");
            ctx->stats.product_launches += a.launches;
            ctx->stats.launches += a.launches;
        }
        int launches = 0;
        bool taken = true;
        if (!small.empty())
            CK(product_tc_diag(small.data(), (int)small.size(), ctx->opt.count_bits, ctx->sms, ctx->d_err, to, st,
                               &launches, &taken));
        if (!taken) return JSIM_ERR_UNSUPPORTED;  // (only a candidate where the rows are aligned)
        ctx->stats.product_launches += launches;
        ctx->stats.launches += launches;
    } else {
        int rc = lanes_fork(ctx, kLanes);
        if (rc) return rc;
        for (size_t c = 0; c < w.cols.size(); ++c) {
            const Col& cl = w.cols[c];
            if (cl.empty || cl.n == 0) continue;
            cudaStream_t ls = ctx->lanes[c % kLanes];
            ProductArgs a{};
            a.X = w.xpool.as<u64>() + cl.x_off; a.stride = cl.stride; a.n = cl.n; a.W = cl.stride;
            a.Wdev = scal + 2 * c; a.C = (char*)w.cpool.p + cl.c_off; a.ldc = cl.n;
            a.count_bits = ctx->opt.count_bits; a.word_bits = word_bits; a.sms = ctx->sms;
            a.timeout_ms = ctx->opt.timeout_ms; a.err = ctx->d_err;
            cudaError_t e = product_popc(a, ls);
            if (e != cudaSuccess) return cuda_fail(ctx, e, "batched CUDA-core product");
            ctx->stats.product_launches += a.launches;
            ctx->stats.launches += a.launches;
        }
        rc = lanes_join(ctx, kLanes);
        if (rc) return rc;
    }
    if (run_product_only) return JSIM_OK;
    // epilogue per collection, into the outputs (device) or staging (host)
    size_t cs = 0, js = 0;
    int rce = lanes_fork(ctx, kLanes);
    if (rce) return rce;
    for (size_t c = 0; c < w.cols.size(); ++c) {
        const Col& cl = w.cols[c];
        const size_t gi = first + c;
        void* Cd = C ? C[gi] : nullptr;
        double* Jd = J ? J[gi] : nullptr;
        if (!dev_out) {
            Cd = Cd ? (void*)((char*)w.cstage.p + cs) : nullptr;
            Jd = Jd ? (double*)((char*)w.jstage.p + js) : nullptr;
        }
        cs += cl.n * cl.n * cb;
        js += cl.n * cl.n * sizeof(double);
        if (cl.n == 0 || (!Cd && !Jd)) continue;
        CK(launch_epilogue((char*)w.cpool.p + cl.c_off, cl.n, ctx->opt.count_bits, w.spool.as<u64>() + cl.s_off, Cd,
                           Jd, ctx->lanes[c % kLanes], ctx->opt.filter_min == 2, ctx->opt.distance, ctx->d_err));
        ctx->stats.launches += 1;
    }
    return lanes_join(ctx, kLanes);
}

// word counts of the call (device running totals) into the statistics
int finish_stats(jsim_ctx* ctx, Wave& w)
{
    const size_t k = w.cols.size();
    std::vector<u64> sc(2 * k);
    CK(cudaMemcpyAsync(sc.data(), w.scal.p, 2 * k * sizeof(u64), cudaMemcpyDeviceToHost, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    ctx->stats.words = 0;
    ctx->stats.bitops_dense = 0;
    ctx->stats.batches = 0;
    for (size_t c = 0; c < k; ++c) {
        const Col& x = w.cols[c];
        ctx->stats.words += sc[2 * c];
        ctx->stats.batches += x.rounds;
        ctx->stats.bitops_dense += 64.0 * (double)sc[2 * c] * (double)x.n * (double)(x.n + 1) / 2.0;
    }
    return JSIM_OK;
}

// time the product of the wave with one variant (CUDA events), ms
int time_product(jsim_ctx* ctx, Wave& w, int variant, int word_bits, int tile_n, float& ms)
{
    cudaEvent_t a = take_event(ctx), b = take_event(ctx);
    if (!a || !b) return JSIM_ERR_CUDA;
    CK(cudaEventRecord(a, ctx->stream));
    int rc = enqueue_wave(ctx, w, nullptr, nullptr, true, 0, true, variant, word_bits, tile_n);
    if (rc) return rc;
    CK(cudaEventRecord(b, ctx->stream));
    CK(cudaEventSynchronize(b));
    CK(cudaEventElapsedTime(&ms, a, b));
    return JSIM_OK;
}

}  // namespace

// Tuning cache: shape signature -> (variant, word bits, tile width).
struct jsim_tuned {
    int variant, word_bits, tile_n;
};
struct jsim_tuning {
    std::vector<std::pair<u64, jsim_tuned>> entries;
};

namespace {
jsim_tuning* tuning_of(jsim_ctx* ctx)
{
    static std::vector<std::pair<jsim_ctx*, jsim_tuning*>> tab;  // one per context
    for (auto& e : tab)
        if (e.first == ctx) return e.second;
    tab.push_back({ctx, new jsim_tuning()});
    return tab.back().second;
}

// The wave kept for a replay, taken by a call (so that no request of the call
// gives it back) and kept again when the call is done with it.
struct KeptWave {
    jsim_ctx* ctx;
    std::unique_ptr<Wave> w;
    explicit KeptWave(jsim_ctx* c) : ctx(c), w((Wave*)c->kept_wave) { c->kept_wave = nullptr; }
    ~KeptWave() { ctx->kept_wave = w.release(); }
};

// The wave of a call that replays nothing; one that an error ends goes once the
// side streams are through with it.
struct FreshWave {
    jsim_ctx* ctx;
    std::unique_ptr<Wave> w;
    bool done = false;
    ~FreshWave()
    {
        if (done) return;
        for (cudaStream_t s : ctx->lanes) cudaStreamSynchronize(s);
        cudaGetLastError();
    }
};
}  // namespace

bool jsim_batched_release(jsim_ctx* ctx)
{
    if (!ctx->kept_wave) return false;
    delete (Wave*)ctx->kept_wave;
    ctx->kept_wave = nullptr;
    return true;
}

// The batched machinery over k collections (statistics into the caller's
// scope).
static int batched_body(jsim_ctx* ctx, const jsim_sets* cols, uint64_t k, void* const* C, uint64_t* const* sizes,
                        double* const* J, int out_mem)
{
    if (k == 0) return JSIM_OK;
    const bool dev_out = out_mem == JSIM_MEM_DEVICE;
    const size_t cb = ctx->opt.count_bits == 64 ? 8 : 4;

    // ---- host-side checks and the shape signature ----
    bool all_dev = true;
    u64 sig = mix(0x5151, k);
    sig = mix(sig, ctx->opt.batch_rows);
    sig = mix(sig, (u64)ctx->opt.variant * 131 + ctx->opt.count_bits * 7 + ctx->opt.id_bits);
    sig = mix(sig, (u64)ctx->opt.filter_min);
    std::vector<Col> cl(k);
    for (u64 c = 0; c < k; ++c) {
        int rc = check_sets(&cols[c]);
        if (rc) return rc;
        if (cols[c].n > (1ull << 20)) return JSIM_ERR_ARG;
        rc = load_offsets(ctx, &cols[c], cl[c].hoff);
        if (rc) return rc;
        cl[c].n = cols[c].n;
        cl[c].N = cl[c].hoff[cl[c].n];
        all_dev = all_dev && cols[c].mem == JSIM_MEM_DEVICE;
        sig = mix(sig, cl[c].n);
        for (u64 v : cl[c].hoff) sig = mix(sig, v);
        sig = mix(sig, (u64)(uintptr_t)cols[c].ids);
        sig = mix(sig, (u64)(uintptr_t)cols[c].offsets);
        // a captured graph writes C and J through the pointers it saw
        sig = mix(sig, (u64)(uintptr_t)(C ? C[c] : nullptr));
        sig = mix(sig, (u64)(uintptr_t)(J ? J[c] : nullptr));
    }
    const bool use_graph = all_dev && dev_out;
    CK(cudaMemsetAsync(ctx->d_err, 0, sizeof(u32), ctx->stream));

    // ---- replay a captured call on the same collections ----
    {
        KeptWave kept(ctx);
        if (use_graph) {
            if (kept.w && kept.w->signature == sig && kept.w->exec) {
                // validation still runs: the values may have changed
                Wave& w = *kept.w;
                DevBuf flags;
                ALLOC(flags, 3 * sizeof(u64) * k);
                CK(cudaMemsetAsync(flags.p, 0, 3 * sizeof(u64) * k, ctx->stream));
                CK(cudaMemsetAsync(w.spool.p, 0, w.spool.bytes, ctx->stream));
                for (u64 c = 0; c < k; ++c) {
                    Col& x = w.cols[c];
                    CK(cudaMemsetAsync(flags.as<u64>() + 3 * c + 2, 0xff, 8, ctx->stream));
                    if (x.n == 0) continue;
                    Plan plan;
                    u64* pb = w.ppool.as<u64>() + x.p_off;
                    plan.beg = pb; plan.len = pb + x.n; plan.cofs = pb + 2 * x.n; plan.totals = pb + 3 * x.n + 1;
                    CK(launch_plan(x.d_off, x.d_ids, x.n, 0, 0, true, plan, ctx->stream));
                    CK(launch_validate(x.d_off, x.d_ids, x.n, plan, x.max_chunks, ctx->opt.id_bits,
                                       w.spool.as<u64>() + x.s_off, (u32*)(flags.as<u64>() + 3 * c),
                                       flags.as<u64>() + 3 * c + 1, flags.as<u64>() + 3 * c + 2, ctx->sms,
                                       ctx->stream));
                }
                std::vector<u64> hf(3 * k);
                CK(cudaMemcpyAsync(hf.data(), flags.p, 3 * sizeof(u64) * k, cudaMemcpyDeviceToHost, ctx->stream));
                CK(cudaStreamSynchronize(ctx->stream));
                for (u64 c = 0; c < k; ++c) {
                    if (w.cols[c].n == 0) continue;
                    u32 f = (u32)hf[3 * c];
                    if (f & kFlagUnsorted) return JSIM_ERR_UNSORTED;
                    if (f & kFlagIdRange) return JSIM_ERR_ID_RANGE;
                    // a changed value range would need a new plan: fall through
                    if (hf[3 * c + 1] != w.cols[c].maxid || (w.cols[c].N && hf[3 * c + 2] != w.cols[c].minid))
                        goto replan;
                }
                {
                    StageTimer t(ctx, &ctx->stats.ms_product);
                    CK(cudaGraphLaunch(w.exec, ctx->stream));
                }
                // nothing is written when a bounded device wait ran out, as on the captured call
                const int rcw = check_device_waits(ctx, ctx->d_err);
                if (rcw) return rcw;
                if (sizes)
                    for (u64 c = 0; c < k; ++c)
                        if (sizes[c] && w.cols[c].n)
                            CK(cudaMemcpyAsync(sizes[c], w.spool.as<u64>() + w.cols[c].s_off, w.cols[c].n * 8,
                                               cudaMemcpyDeviceToDevice, ctx->stream));
                CK(cudaStreamSynchronize(ctx->stream));
                ctx->stats.variant = w.variant;
                ctx->stats.tile_n = w.variant == JSIM_VARIANT_TC ? (u64)w.tile_n : 0;
                return finish_stats(ctx, w);
            }
        }
    }
replan:
    jsim_batched_release(ctx);
    FreshWave fresh{ctx, std::unique_ptr<Wave>(new Wave())};
    Wave& w = *fresh.w;
    w.signature = sig;
    w.cols = std::move(cl);

    // ---- inputs on the device ----
    {
        StageTimer t(ctx, &ctx->stats.ms_h2d);
        u64 tot_ids = 0, tot_off = 0;
        for (auto& x : w.cols) { tot_ids += x.N; tot_off += x.n + 1; }
        if (!all_dev) {
            ALLOC(w.ids_pool, std::max<u64>(tot_ids, 1) * 8);
            ALLOC(w.off_pool, std::max<u64>(tot_off, 1) * 8);
        }
        u64 io = 0, oo = 0;
        for (u64 c = 0; c < k; ++c) {
            Col& x = w.cols[c];
            if (cols[c].mem == JSIM_MEM_DEVICE) {
                x.d_off = (const u64*)cols[c].offsets;
                x.d_ids = (const u64*)cols[c].ids;
            } else {
                u64* doff = w.off_pool.as<u64>() + oo;
                u64* dids = w.ids_pool.as<u64>() + io;
                CK(cudaMemcpyAsync(doff, x.hoff.data(), (x.n + 1) * 8, cudaMemcpyHostToDevice, ctx->stream));
                if (x.N) CK(cudaMemcpyAsync(dids, cols[c].ids, x.N * 8, cudaMemcpyHostToDevice, ctx->stream));
                x.d_off = doff;
                x.d_ids = dids;
                oo += x.n + 1;
                io += x.N;
            }
        }
    }

    // ---- validation of every collection, one synchronisation ----
    size_t s_tot = 0, p_tot = 0;
    for (auto& x : w.cols) {
        x.s_off = s_tot; s_tot += x.n;
        x.p_off = p_tot; p_tot += plan_words(x.n);
        x.max_chunks = x.N / kChunk + x.n + 1;
    }
    ALLOC(w.spool, std::max<size_t>(s_tot, 1) * 8);
    ALLOC(w.ppool, std::max<size_t>(p_tot, 1) * 8);
    DevBuf flags;
    ALLOC(flags, 3 * sizeof(u64) * k);
    {
        StageTimer t(ctx, &ctx->stats.ms_validate);
        CK(cudaMemsetAsync(w.spool.p, 0, w.spool.bytes, ctx->stream));
        CK(cudaMemsetAsync(flags.p, 0, 3 * sizeof(u64) * k, ctx->stream));
        for (u64 c = 0; c < k; ++c) CK(cudaMemsetAsync(flags.as<u64>() + 3 * c + 2, 0xff, 8, ctx->stream));
        int rc = lanes_ensure(ctx, kLanes);
        if (rc) return rc;
        rc = lanes_fork(ctx, kLanes);
        if (rc) return rc;
        for (u64 c = 0; c < k; ++c) {
            Col& x = w.cols[c];
            if (x.n == 0) continue;
            cudaStream_t ls = ctx->lanes[c % kLanes];
            Plan plan;
            u64* pb = w.ppool.as<u64>() + x.p_off;
            plan.beg = pb; plan.len = pb + x.n; plan.cofs = pb + 2 * x.n; plan.totals = pb + 3 * x.n + 1;
            CK(launch_plan(x.d_off, x.d_ids, x.n, 0, 0, true, plan, ls));
            CK(launch_validate(x.d_off, x.d_ids, x.n, plan, x.max_chunks, ctx->opt.id_bits, w.spool.as<u64>() + x.s_off,
                               (u32*)(flags.as<u64>() + 3 * c), flags.as<u64>() + 3 * c + 1,
                               flags.as<u64>() + 3 * c + 2, ctx->sms, ls));
            ctx->stats.launches += 2;
        }
        rc = lanes_join(ctx, kLanes);
        if (rc) return rc;
    }
    std::vector<u64> hf(3 * k), hs(std::max<size_t>(s_tot, 1));
    CK(cudaMemcpyAsync(hf.data(), flags.p, 3 * sizeof(u64) * k, cudaMemcpyDeviceToHost, ctx->stream));
    CK(cudaMemcpyAsync(hs.data(), w.spool.p, s_tot * 8, cudaMemcpyDeviceToHost, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    for (u64 c = 0; c < k; ++c) {
        Col& x = w.cols[c];
        if (x.n == 0) continue;
        u32 f = (u32)hf[3 * c];
        if (f & kFlagUnsorted) return JSIM_ERR_UNSORTED;
        if (f & kFlagIdRange) return JSIM_ERR_ID_RANGE;
        for (u64 i = 0; i < x.n; ++i)
            if (ctx->opt.count_bits == 32 && hs[x.s_off + i] > 0xffffffffull) return JSIM_ERR_OVERFLOW;
        x.maxid = hf[3 * c + 1];
        x.minid = hf[3 * c + 2];
    }

    // ---- batch plan and packed-matrix bound of every collection ----
    // A lane's batch costs kWaveBatchMs whatever it holds: few values take
    // wide batches, as in the plain call (dense_batch_rows), as far as the
    // lanes' bitmaps stay within what the packed matrices take (a call's
    // scratch at most doubles).
    size_t x_tot = 0, c_tot = 0, cs_tot = 0, js_tot = 0;
    auto plan_wave = [&](u64 widest) -> int {
        x_tot = c_tot = cs_tot = js_tot = 0;
        w.max_mt = 0;
        u64 batches = 0;
        for (auto& x : w.cols) {
            x.empty = x.N == 0;
            const u64 span = x.empty ? 0 : x.maxid - x.minid;
            u64 one = 64;
            while (one < span + 1 && one < (1ull << 29)) one <<= 1;
            x.mt = ctx->opt.batch_rows ? ctx->opt.batch_rows : one;
            if (!x.empty && x.maxid / x.mt - x.minid / x.mt + 1 > 4096)
                return JSIM_ERR_UNSUPPORTED;  // value span too wide for one batched plan
            if (widest > x.mt && !x.empty && !ctx->opt.batch_rows)
                x.mt = std::max(x.mt, std::min(widest, dense_batch_rows(ctx, x.n, x.N, x.minid, x.maxid, nullptr,
                                                                        nullptr, kWaveBatchMs, kLanes)));
            x.lo0 = x.empty ? 0 : x.minid / x.mt * x.mt;
            x.rounds = x.empty ? 0 : x.maxid / x.mt - x.minid / x.mt + 1;
            // sum_l ceil(R_l / 64) <= N / 64 + rounds
            x.stride = round_up(x.N / 64 + x.rounds + 1, kWordPad);
            x.n_pad = round_up(std::max<u64>(x.n, 1), kRowPad);
            x.x_off = x_tot;
            x_tot += x.n_pad * x.stride;
            x.c_off = c_tot;
            c_tot += x.n * x.n * cb;
            cs_tot += x.n * x.n * cb;
            js_tot += x.n * x.n * sizeof(double);
            w.max_mt = std::max(w.max_mt, x.mt);
            batches += x.rounds;
        }
        w.batches = batches;
        return JSIM_OK;
    };
    auto alloc_wave = [&]() -> int {
        const u64 nwords = std::max<u64>(w.max_mt / 64, 1);
        const u64 nb = (nwords + kScanBlockWords - 1) / kScanBlockWords;
        for (int l = 0; l < kLanes; ++l) {
            ALLOC(w.bitmap[l], nwords * 8);
            if (ctx->opt.filter_min == 2) ALLOC(w.seen[l], nwords * 8);
            ALLOC(w.dir[l], nwords * 4);
            ALLOC(w.bsum[l], std::max<u64>(nb, 1) * 8);
            ALLOC(w.boff[l], std::max<u64>(nb, 1) * 8);
            ALLOC(w.R[l], 8);
        }
        ALLOC(w.xpool, std::max<size_t>(x_tot, 1) * 8);
        ALLOC(w.cpool, std::max<size_t>(c_tot, 8));
        ALLOC(w.scal, 2 * sizeof(u64) * k);
        ALLOC(w.jobtab, sizeof(TcJobDesc) * std::max<u64>(k, 1));
        if (!dev_out) {
            if (C) ALLOC(w.cstage, std::max<size_t>(cs_tot, 8));
            if (J) ALLOC(w.jstage, std::max<size_t>(js_tot, 8));
        }
        return JSIM_OK;
    };
    {
        const u64 narrow = 1ull << 29;
        int rc = plan_wave(narrow);
        if (rc) return rc;
        u64 widest = narrow;
        const double bits = ctx->opt.filter_min == 2 ? 2.5 : 1.5;  // bitmap, directory (and every row's bitmap)
        while (widest < (1ull << 32) && kLanes * bits * (double)(2 * widest) / 8.0 <= 8.0 * (double)x_tot) widest *= 2;
        if (widest > narrow) {
            rc = plan_wave(widest);
            if (rc) return rc;
        }
        rc = alloc_wave();
        if (rc == JSIM_ERR_OOM && w.max_mt > narrow && !ctx->opt.batch_rows) {
            // no room for the wide batches and what lies behind them
            for (int l = 0; l < kLanes; ++l)
                for (DevBuf* d : {&w.bitmap[l], &w.seen[l], &w.dir[l], &w.bsum[l], &w.boff[l]}) d->release();
            for (DevBuf* d : {&w.xpool, &w.cpool, &w.scal, &w.jobtab, &w.cstage, &w.jstage}) d->release();
            rc = plan_wave(narrow);
            if (!rc) rc = alloc_wave();
        }
        if (rc) return rc;
        ctx->stats.batches += w.batches;
        std::vector<TcJobDesc> jobs = wave_jobs(w);
        if (!jobs.empty())
            CK(cudaMemcpyAsync(w.jobtab.p, jobs.data(), sizeof(TcJobDesc) * jobs.size(), cudaMemcpyHostToDevice,
                               ctx->stream));
        CK(cudaStreamSynchronize(ctx->stream));
    }

    // ---- variant: the caller's, or the tuned one for this shape ----
    int variant = ctx->opt.variant, word_bits = ctx->opt.word_bits;
    int tile_n = ctx->opt.tile_n ? ctx->opt.tile_n : 256;
    const bool tc_ok = product_tc_supported(ctx->opt.device);
    if (variant == JSIM_VARIANT_TC && !tc_ok) return JSIM_ERR_UNSUPPORTED;
    if (variant != JSIM_VARIANT_AUTO && variant != JSIM_VARIANT_TC && variant != JSIM_VARIANT_POPC)
        return JSIM_ERR_UNSUPPORTED;
    jsim_tuning* tun = tuning_of(ctx);
    u64 shape = 0x77;
    for (auto& x : w.cols) shape = mix(shape, (x.n + 31) / 32 * 1000003 + (64 - __builtin_clzll(x.N | 1)));
    shape = mix(shape, (u64)ctx->opt.tile_n);
    // (the 4-bit products load rows by TMA: a choice made with 16-byte aligned
    // matrices does not hold for others)
    const bool aligned = (uintptr_t)w.xpool.p % 16 == 0;
    shape = mix(shape, aligned ? 1 : 0);
    if (variant == JSIM_VARIANT_AUTO) {
        for (auto& e : tun->entries)
            if (e.first == shape) {
                variant = e.second.variant;
                word_bits = e.second.word_bits;
                tile_n = e.second.tile_n;
            }
    }

    // ---- ingest all collections (and tune the product on the packed words) ----
    if (variant == JSIM_VARIANT_AUTO) {
        int rc = enqueue_wave(ctx, w, nullptr, nullptr, true, 0, false, JSIM_VARIANT_POPC, 64, 256);
        if (rc) return rc;
        // the first call above also ran one product; now time each candidate:
        // tensor-core tiles of 128 x 256 and of 128 x 128 (collections of at
        // most 128 samples then fill whole tiles, and diagonal tiles unpack
        // their rows once), CUDA-core products on 64- and 32-bit words
        std::vector<jsim_tuned> cands;
        if (tc_ok) {
            static_assert(kWordPad % 2 == 0, "16-byte aligned rows");
            // 4-bit operands (13 collections of 31 to 231 samples x 20,000 values,
            // whole call: 6.8 ms with byte tiles, 6.1)
            if (!ctx->opt.tile_n && aligned) cands.push_back({JSIM_VARIANT_TC2, 64, 256});
            if (ctx->opt.tile_n != 128) cands.push_back({JSIM_VARIANT_TC, 64, 256});
            if (ctx->opt.tile_n != 256) cands.push_back({JSIM_VARIANT_TC, 64, 128});
        }
        cands.push_back({JSIM_VARIANT_POPC, 64, 256});
        cands.push_back({JSIM_VARIANT_POPC, 32, 256});
        float best = 1e30f;
        for (auto& cd : cands) {
            float ms = 0;
            int r2 = time_product(ctx, w, cd.variant, cd.word_bits, cd.tile_n, ms);
            if (r2) return r2;
            if (ms < best) {
                best = ms;
                variant = cd.variant;
                word_bits = cd.word_bits;
                tile_n = cd.tile_n;
            }
        }
        tun->entries.push_back({shape, {variant, word_bits, tile_n}});
    }
    w.variant = variant;
    w.word_bits = word_bits;
    w.tile_n = tile_n;
    ctx->stats.variant = variant;
    ctx->stats.tile_n = variant == JSIM_VARIANT_TC ? (u64)tile_n : 0;

    // ---- the launch sequence: captured once when inputs and outputs are on the device ----
    if (use_graph) {
        cudaGraph_t g = nullptr;
        CK(cudaStreamBeginCapture(ctx->stream, cudaStreamCaptureModeThreadLocal));
        int rc = enqueue_wave(ctx, w, C, J, dev_out, 0, false, variant, word_bits, tile_n);
        cudaError_t e = cudaStreamEndCapture(ctx->stream, &g);
        if (rc) { if (g) cudaGraphDestroy(g); return rc; }
        if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaStreamEndCapture");
        e = cudaGraphInstantiate(&w.exec, g, 0);
        cudaGraphDestroy(g);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaGraphInstantiate");
        StageTimer t(ctx, &ctx->stats.ms_product);
        CK(cudaGraphLaunch(w.exec, ctx->stream));
    } else {
        StageTimer t(ctx, &ctx->stats.ms_product);
        int rc = enqueue_wave(ctx, w, C, J, dev_out, 0, false, variant, word_bits, tile_n);
        if (rc) return rc;
    }

    // ---- outputs (none when a bounded device wait ran out: the epilogues
    // skipped their writes) ----
    {
        int rc = check_device_waits(ctx, ctx->d_err);
        if (rc) return rc;
    }
    {
        StageTimer t(ctx, &ctx->stats.ms_d2h);
        const cudaMemcpyKind kind = dev_out ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
        size_t cs = 0, js = 0;
        for (u64 c = 0; c < k; ++c) {
            const Col& x = w.cols[c];
            if (!dev_out && x.n) {
                if (C && C[c]) CK(cudaMemcpyAsync(C[c], (char*)w.cstage.p + cs, x.n * x.n * cb, kind, ctx->stream));
                if (J && J[c]) CK(cudaMemcpyAsync(J[c], (char*)w.jstage.p + js, x.n * x.n * 8, kind, ctx->stream));
            }
            cs += x.n * x.n * cb;
            js += x.n * x.n * 8;
            if (sizes && sizes[c] && x.n)
                CK(cudaMemcpyAsync(sizes[c], w.spool.as<u64>() + x.s_off, x.n * 8, kind, ctx->stream));
        }
    }
    CK(cudaStreamSynchronize(ctx->stream));
    int rc = finish_stats(ctx, w);
    fresh.done = !rc;
    if (use_graph && !rc) ctx->kept_wave = fresh.w.release();  // (else there is nothing to replay)
    return rc;
}

// Collections the block-sparse product may take (variant AUTO, 256 to 2048
// samples, tensor cores, device-resident input): they gain more from
// skipping blocks than from sharing launches, and run as plain calls (which
// decide, by the sketch, between the block-sparse and the dense product);
// the others share the batched launches.  The plain calls' inputs are
// validated first, so an input error still leaves every output unwritten.
extern "C" int jsim_all_pairs_batched(jsim_ctx* ctx, const jsim_sets* cols, uint64_t k, void* const* C,
                                      uint64_t* const* sizes, double* const* J, int out_mem)
{
    if (!ctx || (!cols && k)) return JSIM_ERR_ARG;
    if (out_mem != JSIM_MEM_HOST && out_mem != JSIM_MEM_DEVICE) return JSIM_ERR_ARG;
    CK(cudaSetDevice(ctx->opt.device));
    CallScope scope(ctx);
    StageTimer total(ctx, &ctx->stats.ms_total);
    if (k == 0) return JSIM_OK;
    for (u64 c = 0; c < k; ++c) {
        const int rc = check_sets(&cols[c]);
        if (rc) return rc;
    }
    const bool split = ctx->opt.variant == JSIM_VARIANT_AUTO && !ctx->opt.count_useful &&
                       (ctx->opt.batch_rows == 0 || ctx->opt.batch_rows % (1ull << 18) == 0) &&
                       product_tc_supported(ctx->opt.device);
    std::vector<u64> big, rest;
    for (u64 c = 0; c < k; ++c)
        (split && cols[c].n >= 256 && cols[c].n <= 2048 ? big : rest).push_back(c);
    // device-resident inputs only, so that every collection is validated
    // before any output is written
    for (u64 c : big)
        if (cols[c].mem != JSIM_MEM_DEVICE) big.clear();
    if (big.empty()) return batched_body(ctx, cols, k, C, sizes, J, out_mem);
    for (u64 c : big) {
        std::vector<u64> hoff;
        int r = load_offsets(ctx, &cols[c], hoff);
        if (r) return r;
        Staged st;
        r = stage_input(ctx, &cols[c], st, hoff, false);
        if (r) return r;
        r = validate_staged(ctx, st, ctx->stream);
        if (r) return r;
        r = check_staged(ctx, st);
        if (r) return r;
    }
    rest.clear();
    for (u64 c = 0; c < k; ++c)
        if (std::find(big.begin(), big.end(), c) == big.end()) rest.push_back(c);
    int rc = JSIM_OK;
    if (!rest.empty()) {
        std::vector<jsim_sets> rc_cols;
        std::vector<void*> rc_C;
        std::vector<uint64_t*> rc_s;
        std::vector<double*> rc_J;
        for (u64 c : rest) {
            rc_cols.push_back(cols[c]);
            rc_C.push_back(C ? C[c] : nullptr);
            rc_s.push_back(sizes ? sizes[c] : nullptr);
            rc_J.push_back(J ? J[c] : nullptr);
        }
        rc = batched_body(ctx, rc_cols.data(), rest.size(), C ? rc_C.data() : nullptr, sizes ? rc_s.data() : nullptr,
                          J ? rc_J.data() : nullptr, out_mem);
        if (rc) return rc;
    }
    // the batched part carried out its dense work; the plain calls add theirs
    const int wave_variant = ctx->stats.variant;
    const u64 wave_tile = ctx->stats.tile_n;
    if (ctx->stats.bitops_done == 0) ctx->stats.bitops_done = ctx->stats.bitops_dense;
    for (u64 c : big) {
        rc = all_pairs_impl(ctx, &cols[c], C ? C[c] : nullptr, sizes ? sizes[c] : nullptr, J ? J[c] : nullptr,
                            out_mem, 0, 1, false, false);
        if (rc) return rc;
    }
    if (!rest.empty()) {
        ctx->stats.variant = wave_variant;
        ctx->stats.tile_n = wave_tile;
    }
    return JSIM_OK;
}
