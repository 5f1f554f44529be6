// fim_api.cu -- the C ABI of include/fim.h: context, memory, and the order of
// the three stages of Section III (matrix construction, support calculation,
// frequent-itemset extraction).  No exception crosses the boundary; every
// entry point returns a FIM_* status.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>

#include "fim_common.cuh"


namespace {

thread_local char g_last_cuda[256] = {0};

// Restores the caller's current device on scope exit.
struct DeviceGuard {
    int prev = -1;
    bool ok = false;
    explicit DeviceGuard(int dev) {
        if (cudaGetDevice(&prev) == cudaSuccess && cudaSetDevice(dev) == cudaSuccess) ok = true;
    }
    ~DeviceGuard() {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

constexpr unsigned long long kTaskCap = 1ull << 20;
constexpr unsigned long long kCandPoolCap = 1ull << 24;
constexpr size_t kStackBudget = 8ull << 30;   // first try; grows on FIM_E_STACK
constexpr size_t kStackBudgetMax = 64ull << 30;
constexpr int64_t kDirectWords = 1 << 16;        // frequent columns up to this many words: no projection
constexpr int64_t kDirectWordsShort = 3 << 17;   // the same for few items in short rows
constexpr unsigned long long kSmallPlanWords = 64ull << 20;  // worst-case projection of a device-planned mine
constexpr unsigned long long kProjWords = 1ull << 30;  // largest projection (words)
constexpr unsigned long long kTriples = 64ull << 20;   // largest table of triple supports
constexpr int64_t kLongWords = 4096;             // columns from which the CTA workers may be the better ones
constexpr uint32_t kProjWmax = 1u << 15;         // longest projected column (words)
constexpr size_t kProjStackBudget = 4ull << 30;  // warp workers' global stacks

// Read back a device struct, or two (the stream is synchronised): through
// page-locked memory, which the copy engine writes without a staging pass.
template <class T, class U>
int read_back(fim_ctx *ctx, T *host, const void *dev, U *host2, const void *dev2) {
    constexpr size_t at2 = (sizeof(T) + 15) / 16 * 16;
    static_assert(at2 + sizeof(U) <= kPinnedBytes, "landing place");
    char *const land = static_cast<char *>(ctx->pinned);
    FIM_CUDA_TRY(cudaMemcpyAsync(land, dev, sizeof(T), cudaMemcpyDeviceToHost, ctx->stream));
    if (host2) FIM_CUDA_TRY(cudaMemcpyAsync(land + at2, dev2, sizeof(U), cudaMemcpyDeviceToHost, ctx->stream));
    FIM_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
    memcpy((void *)host, land, sizeof(T));
    if (host2) memcpy((void *)host2, land + at2, sizeof(U));
    return FIM_OK;
}
template <class T>
int read_back(fim_ctx *ctx, T *host, const void *dev) {
    return read_back(ctx, host, dev, static_cast<int *>(nullptr), nullptr);
}

}  // namespace

void fim_set_cuda_error(cudaError_t e, const char *what, const char *file, int line) {
    snprintf(g_last_cuda, sizeof(g_last_cuda), "%s (%s) at %s:%d: %s", cudaGetErrorName(e), what,
             file, line, cudaGetErrorString(e));
    (void)cudaGetLastError();  // clear a sticky-free error so the ctx stays usable
}

// The ctx's side stream, at the device's highest priority: work put there
// (a group's pair pass beside the next group's build) is scheduled first
// where the two kernels compete for an SM.
int fim_aux_stream(fim_ctx *ctx) {
    if (ctx->aux_stream) return FIM_OK;
    int least = 0, greatest = 0;
    FIM_CUDA_TRY(cudaDeviceGetStreamPriorityRange(&least, &greatest));
    FIM_CUDA_TRY(cudaStreamCreateWithPriority(&ctx->aux_stream, cudaStreamNonBlocking, greatest));
    return FIM_OK;
}

int queue_compact_status(fim_ctx *ctx) {
    if (ctx->compact_waits)
        FIM_CUDA_TRY(cudaMemcpyAsync(ctx->pinned, ctx->dev_flag.as<int>() + kCompactErr, sizeof(int),
                                     cudaMemcpyDeviceToHost, ctx->stream));
    return FIM_OK;
}
int compact_status(fim_ctx *ctx) {
    return ctx->compact_waits && *static_cast<const int *>(ctx->pinned) ? FIM_E_TIMEOUT : FIM_OK;
}

// Workers reserve record slots ahead.  A used slot past the arena's end is an
// overflow; a reservation that only ends past it is not, and its slots there
// are holes that exist in the counts alone: the compaction must not look at
// them.
void drop_slots_past_arena(fim_ctx *ctx) {
    MineCounters &c = ctx->host_ctr;
    if (c.n_records <= ctx->rec_cap) return;
    c.rec_holes -= c.n_records - ctx->rec_cap;
    c.n_records = ctx->rec_cap;
}

// Phase times of the last single-database mine, once its work has finished
// (events ev[1..4] of that mine; called before anything records them again).
int fim_finish_phase_times(fim_ctx *ctx) {
    if (!ctx->phase_times_pending) return FIM_OK;
    ctx->phase_times_pending = false;
    FIM_CUDA_TRY(cudaEventSynchronize(ctx->ev[4]));
    cudaEventElapsedTime(&ctx->stats.ms_pairs, ctx->ev[1], ctx->ev[2]);
    cudaEventElapsedTime(&ctx->stats.ms_dfs, ctx->ev[2], ctx->ev[3]);
    cudaEventElapsedTime(&ctx->stats.ms_compact, ctx->ev[3], ctx->ev[4]);
    return FIM_OK;
}

// Device memory for b, `want` bytes or at least `bytes`.
static int dev_alloc(fim_ctx *ctx, DevBuf &b, size_t want, size_t bytes) {
    const size_t limit = (size_t)ctx->test_memory_mb << 20;
    for (size_t n = want;; n = bytes) {
        if (limit && ctx->bytes_held + n > limit) b.p = nullptr;  // (the fault-injection hook)
        else if (cudaMalloc(&b.p, n) != cudaSuccess) {
            (void)cudaGetLastError();
            b.p = nullptr;
        }
        if (b.p) {
            b.bytes = n;
            return FIM_OK;
        }
        if (n == bytes) return FIM_E_NOMEM;
    }
}

void drop_rows(fim_ctx *ctx) {
    ctx->rows_kept = false;
    ctx->row_cap = 0;
    fim_release(ctx, ctx->row_ptr);
    fim_release(ctx, ctx->row_idx);
}

int fim_reserve(fim_ctx *ctx, DevBuf &b, size_t bytes) {
    if (bytes == 0) bytes = 16;
    if (bytes <= b.bytes) return FIM_OK;
    if (b.p) {
        FIM_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
        cudaFree(b.p);
        ctx->bytes_held -= b.bytes;
        b.p = nullptr;
        b.bytes = 0;
    }
    size_t nb = bytes + bytes / 4;
    nb = (nb + 255) & ~(size_t)255;
    int rc = dev_alloc(ctx, b, nb, bytes);
    if (rc == FIM_E_NOMEM && ctx->row_idx.p && &b != &ctx->row_ptr && &b != &ctx->row_idx) {
        // the kept rows only make the pair pass faster: their room first
        FIM_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
        drop_rows(ctx);
        rc = dev_alloc(ctx, b, nb, bytes);
    }
    if (rc != FIM_OK) return rc;
    ctx->bytes_held += b.bytes;
    if (ctx->bytes_held > ctx->stats.peak_device_bytes) ctx->stats.peak_device_bytes = ctx->bytes_held;
    return FIM_OK;
}

void fim_release(fim_ctx *ctx, DevBuf &b) {
    if (b.p) {
        cudaFree(b.p);
        ctx->bytes_held -= b.bytes;
    }
    b.p = nullptr;
    b.bytes = 0;
}

extern "C" {

uint32_t fim_version(void) { return (1u << 16) | 0u; }

const char *fim_strerror(int s) {
    switch (s) {
        case FIM_OK: return "ok";
        case FIM_E_INVAL: return "invalid argument or malformed database";
        case FIM_E_NOMEM: return "out of memory";
        case FIM_E_CUDA: return g_last_cuda[0] ? g_last_cuda : "CUDA error";
        case FIM_E_TIMEOUT: return "bounded device wait expired";
        case FIM_E_STACK: return "DFS stack budget exceeded";
        case FIM_E_TOO_SMALL: return "output buffer too small";
        case FIM_E_STATE: return "call out of order";
        case FIM_E_NODEV: return "no such CUDA device";
        case FIM_E_CHECK: return "a debug_checks invariant failed (internal error)";
        default: return "unknown status";
    }
}

uint64_t fim_minsup_from_ppm(int64_t n_trans, uint32_t ppm) {
    if (n_trans <= 0) return 1;
    const unsigned __int128 num = (unsigned __int128)(uint64_t)n_trans * ppm + 999999u;
    const uint64_t v = (uint64_t)(num / 1000000u);
    return v ? v : 1;
}

int fim_create(fim_ctx **out, int device, void *cuda_stream) {
    FIM_NVTX("fim_create");
    if (!out) return FIM_E_INVAL;
    *out = nullptr;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev <= 0) {
        (void)cudaGetLastError();
        return FIM_E_NODEV;
    }
    if (device < 0 || device >= ndev) return FIM_E_NODEV;
    DeviceGuard g(device);
    if (!g.ok) return FIM_E_CUDA;
    fim_ctx *ctx = new (std::nothrow) fim_ctx();
    if (!ctx) return FIM_E_NOMEM;
    ctx->device = device;
    cudaDeviceGetAttribute(&ctx->num_sms, cudaDevAttrMultiProcessorCount, device);
    cudaDeviceGetAttribute(&ctx->l2_bytes, cudaDevAttrL2CacheSize, device);
    if (cuda_stream) {
        ctx->stream = (cudaStream_t)cuda_stream;
    } else {
        if (cudaStreamCreateWithFlags(&ctx->stream, cudaStreamNonBlocking) != cudaSuccess) {
            delete ctx;
            return FIM_E_CUDA;
        }
        ctx->own_stream = true;
    }
    for (auto &e : ctx->ev) cudaEventCreate(&e);
    if (cudaHostAlloc(&ctx->pinned, kPinnedBytes, cudaHostAllocDefault) != cudaSuccess) {
        (void)cudaGetLastError();
        ctx->pinned = nullptr;
        fim_destroy(ctx);
        return FIM_E_NOMEM;
    }
    int rc = fim_reserve(ctx, ctx->counters, sizeof(MineCounters));
    if (rc == FIM_OK) rc = fim_reserve(ctx, ctx->dev_flag, kFlagBytes);
    if (rc == FIM_OK) rc = fim_reserve(ctx, ctx->epoch, sizeof(uint32_t));
    if (rc == FIM_OK && cudaMemsetAsync(ctx->epoch.p, 0, sizeof(uint32_t), ctx->stream) != cudaSuccess) rc = FIM_E_CUDA;
    if (rc != FIM_OK) {
        fim_destroy(ctx);
        return rc;
    }
    *out = ctx;
    return FIM_OK;
}

void fim_destroy(fim_ctx *ctx) {
    FIM_NVTX("fim_destroy");
    if (!ctx) return;
    DeviceGuard g(ctx->device);
    cudaStreamSynchronize(ctx->stream);
    DevBuf *all[] = {&ctx->csr_ptr, &ctx->csr_idx, &ctx->bm, &ctx->row_ptr, &ctx->row_idx, &ctx->item_sup, &ctx->perm, &ctx->rank,
                     &ctx->dev_flag, &ctx->pair_cnt, &ctx->pairbits, &ctx->roots, &ctx->tasks,
                     &ctx->cand_pool, &ctx->stack_bits, &ctx->frame_items, &ctx->frame_sups,
                     &ctx->rec_off, &ctx->rec_len, &ctx->rec_sup, &ctx->rec_items, &ctx->counters,
                     &ctx->keys, &ctx->idx_a, &ctx->idx_b, &ctx->hist, &ctx->scan_tmp, &ctx->kv_a, &ctx->kv_b,
                     &ctx->out_off,
                     &ctx->out_items, &ctx->out_sup, &ctx->rule_base, &ctx->rule_part, &ctx->rule_bits,
                     &ctx->rule_hash, &ctx->rule_set, &ctx->rule_mask,
                     &ctx->rule_conf, &ctx->rule_lift, &ctx->rule_sets, &ctx->probe_buf, &ctx->shard_cost, &ctx->merge_off, &ctx->mlp_w32, &ctx->mlp_wbf, &ctx->trace_x,
                     &ctx->trace_y, &ctx->mlp_scratch, &ctx->root_order, &ctx->root_bucket,
                     &ctx->root_hist, &ctx->rec_db, &ctx->dbdesc, &ctx->epoch, &ctx->sp_idx,
                     &ctx->sp_val, &ctx->sp_z, &ctx->proj_items, &ctx->proj_tiles, &ctx->proj_totals,
                     &ctx->proj_mat, &ctx->proj_list, &ctx->proj_cands, &ctx->proj_triple, &ctx->proj_roots};
    for (DevBuf *b : all) fim_release(ctx, *b);
    fim_release(ctx, ctx->batch_prefix);
    fim_release(ctx, ctx->batch_units);
    fim_release(ctx, ctx->batch_unit_db);
    fim_release(ctx, ctx->batch_plan);
    fim_release(ctx, ctx->batch_windows);
    fim_release(ctx, ctx->batch_slices);
    if (ctx->batch_graph_exec) cudaGraphExecDestroy((cudaGraphExec_t)ctx->batch_graph_exec);
    for (void *g : ctx->compact_graph_exec)
        if (g) cudaGraphExecDestroy((cudaGraphExec_t)g);
    for (cudaStream_t u : ctx->up_stream)
        if (u) cudaStreamDestroy(u);
    if (ctx->aux_stream) cudaStreamDestroy(ctx->aux_stream);
    for (cudaEvent_t e : ctx->seg_ev)
        if (e) cudaEventDestroy(e);
    if (ctx->copy_stream) cudaStreamDestroy(ctx->copy_stream);
    for (cudaEvent_t e : ctx->copy_ev)
        if (e) cudaEventDestroy(e);
    for (cudaEvent_t e : ctx->aux_ev)
        if (e) cudaEventDestroy(e);
    for (cudaEvent_t e : ctx->pair_ev)
        if (e) cudaEventDestroy(e);
    for (cudaEvent_t e : ctx->up_ev)
        if (e) cudaEventDestroy(e);
    for (auto &e : ctx->ev)
        if (e) cudaEventDestroy(e);
    if (ctx->own_stream && ctx->stream) cudaStreamDestroy(ctx->stream);
    if (ctx->pinned) cudaFreeHost(ctx->pinned);
    delete ctx;
}

int fim_build_bitmaps(fim_ctx *ctx, const void *indptr, const void *indices, int64_t n_trans,
                      int32_t n_items, uint32_t flags) {
    FIM_NVTX("fim_build_bitmaps");
    if (!ctx) return FIM_E_INVAL;
    if (n_trans < 0 || n_trans > FIM_MAX_TRANS || n_items < 0 || n_items > FIM_MAX_ITEMS) return FIM_E_INVAL;
    if (!indptr) return FIM_E_INVAL;
    DeviceGuard g(ctx->device);
    if (!g.ok) return FIM_E_CUDA;
    FIM_TRY(fim_finish_phase_times(ctx));  // before the events are recorded again
    ctx->built = false;
    ctx->mined = false;
    ctx->n = n_trans;
    ctx->m = n_items;
    ctx->nw = ceil_div64(n_trans, 32);
    ctx->nwp = round_up64(ctx->nw, FIM_WORDS_ALIGN);
    cudaStream_t st = ctx->stream;
    cudaEventRecord(ctx->ev[0], st);
    const uint64_t launches0 = ctx->launches;

    // the CSR's element types (FIM_CSR_COMPACT: uint32 row offsets, uint16 ids)
    const bool cmp = (flags & FIM_CSR_COMPACT) != 0;
    const size_t pb = csr_off_bytes(cmp), ib = csr_id_bytes(cmp);
    const void *d_ptr = indptr;
    const void *d_idx = indices;
    int64_t h_nnz = -1;
    bool mapped = false;  // pinned host CSR read by the build kernel in place
    if (!(flags & FIM_INPUT_DEVICE)) {
        const int64_t nnz = csr_off(indptr, cmp, n_trans);
        if (csr_off(indptr, cmp, 0) != 0 || nnz < 0 || (nnz > 0 && !indices)) return FIM_E_INVAL;
        if (ctx->upload_mapped) {
            // page-locked, mapped host memory is addressable from the GPU: the
            // kernel streams it over the host link, no staging copy
            cudaPointerAttributes ap{}, ai{};
            const bool ok_p = cudaPointerGetAttributes(&ap, indptr) == cudaSuccess &&
                              ap.type == cudaMemoryTypeHost && ap.devicePointer != nullptr;
            const bool ok_i = nnz == 0 || (cudaPointerGetAttributes(&ai, indices) == cudaSuccess &&
                                           ai.type == cudaMemoryTypeHost && ai.devicePointer != nullptr);
            cudaGetLastError();  // a query on unregistered memory leaves no sticky error
            if (ok_p && ok_i) {
                d_ptr = ap.devicePointer;
                d_idx = nnz ? ai.devicePointer : indices;
                h_nnz = nnz;
                mapped = true;
            }
        }
    }
    if (!(flags & FIM_INPUT_DEVICE) && !mapped) {
        const int64_t nnz = csr_off(indptr, cmp, n_trans);
        FIM_TRY(fim_reserve(ctx, ctx->csr_ptr, pb * (size_t)(n_trans + 1)));
        FIM_TRY(fim_reserve(ctx, ctx->csr_idx, ib * (size_t)(nnz > 0 ? nnz : 1)));
        FIM_CUDA_TRY(cudaMemcpyAsync(ctx->csr_ptr.p, indptr, pb * (size_t)(n_trans + 1), cudaMemcpyHostToDevice, st));
        // (the indices go up inside launch_build_bitmaps, overlapped with the build)
        d_ptr = ctx->csr_ptr.p;
        d_idx = ctx->csr_idx.p;
        h_nnz = nnz;
    }
    // device input: indptr[0] == 0 and indptr[n] >= 0 are checked by the build
    // kernel (no host round trip)
    const size_t mm = (size_t)(n_items > 0 ? n_items : 1);
    FIM_TRY(fim_reserve(ctx, ctx->bm, sizeof(uint32_t) * (size_t)ctx->nwp * mm));
    FIM_TRY(fim_reserve(ctx, ctx->item_sup, sizeof(uint32_t) * mm));
    FIM_TRY(fim_reserve(ctx, ctx->perm, sizeof(int32_t) * mm));
    FIM_TRY(fim_reserve(ctx, ctx->rank, sizeof(int32_t) * mm));
    if (flags & FIM_INPUT_DEVICE) FIM_TRY(launch_build_bitmaps(ctx, d_ptr, d_idx, -1, nullptr, nullptr, cmp));
    else if (mapped) FIM_TRY(launch_build_bitmaps(ctx, d_ptr, d_idx, h_nnz, nullptr, nullptr, cmp));
    else FIM_TRY(launch_build_bitmaps(ctx, d_ptr, d_idx, h_nnz, indptr, h_nnz > 0 ? indices : nullptr, cmp));
    cudaEventRecord(ctx->ev[1], st);
    BuildFlags bf{};
    FIM_TRY(read_back(ctx, &bf, ctx->dev_flag.p));
    if (bf.bad) return FIM_E_INVAL;
    ctx->max_row_len = bf.max_len;
    ctx->row_nnz = bf.nnz;
    ctx->row_pairs = bf.row_pairs;
    ctx->tile_pairs = bf.tile_pairs;
    ctx->rows_kept = ctx->row_cap > 0 && (uint64_t)bf.nnz <= ctx->row_cap;
    cudaEventElapsedTime(&ctx->stats.ms_build, ctx->ev[0], ctx->ev[1]);
    ctx->stats.ms_singletons = 0.f;  // counted by the build kernel
    if (ctx->debug_checks) FIM_TRY(run_check_pads(ctx));
    ctx->stats.launches_build = ctx->launches - launches0;
    ctx->built = true;
    return FIM_OK;
}

}  // extern "C"

namespace {

struct MineState {
    int depth_cap = 0;
    int64_t frame_pool = 0;
    size_t stack_budget = kStackBudget;
    bool cta_dfs = false;  // the warp workers' stack was too small: CTA workers
};

// The search runs on warp workers (k_proj.cu); the trace and no-split
// options, and searches too deep for a warp worker's stack, on the CTA
// workers, which look at whole columns.
bool search_on_warps(uint32_t flags, const MineState &ms) {
    return !ms.cta_dfs && !(flags & (FIM_TRACE | FIM_NO_SPLIT));
}

// The largest projection that mf frequent items can have.
ProjTotals worst_projection(const fim_ctx *ctx, int mf) {
    ProjTotals t{};
    const unsigned long long np = (unsigned long long)mf * (unsigned long long)(mf > 0 ? mf - 1 : 0) / 2;
    t.wmax = (uint32_t)(ceil_div64(ctx->n, 128) * 4);
    t.words = np * t.wmax;
    t.rows = (unsigned long long)mf * (unsigned long long)ctx->n;
    t.cands = np;
    t.tiles = (unsigned long long)mf * ((t.wmax + 31) / 32);
    t.triples = (unsigned long long)mf * mf * mf;
    t.units = (unsigned long long)mf * proj_triple_units(mf);
    return t;
}

// Whether two items of average support share enough rows, if they are independent.
bool avg_pair_frequent(const fim_ctx *ctx, uint32_t thr) {
    if (ctx->m <= 0) return false;
    const double s = (double)ctx->row_nnz / (double)ctx->m;
    return s * s >= (double)thr * (double)ctx->n;
}

// Whether warps on projected columns mine a matrix of long columns sooner than
// CTAs on the whole ones.  A CTA pass costs a column's length per level and
// support; the projection costs its gathered bits, and one warp then walks a
// projected column (about as long where the items are dense) per class.  The
// levels and supports to expect come from the plan: the frequent pairs' mean
// support, the share q of an item's rows that a partner holds, and sets of k
// of as many items as make that many pairs while pair support times q^(k - 2)
// passes.  The factors (us per 1,000 words or million bits) were fitted to 843 mines
// of 100,000 to 3 million rows, 6 to 400 items, independent, Zipf and
// correlated: the choice is within 10% of the better one in 833 of them.
// 1 million rows, us on CTAs and on projected columns: 64 items at density 0.5,
// pairs only 795 and 2,038; 24 items at 0.5, sets of up to four 1,586 and
// 2,081, up to six 14,870 and 8,789; 250 Zipf items at 0.8% 388 and 507, at
// 0.3% 602 and 631; 40 items at 0.05, sets of four 7,375 and 1,187.
bool projection_pays(const ProjTotals &t, int64_t nw, double n, uint32_t thr) {
    const double pairs = (double)t.cands, bits = 32.0 * (double)t.words;
    const double rows = bits / pairs;  // of an item with candidates
    const double q = std::min(1.0, t.pair_sum ? (double)t.pair_sum / bits : rows / n);
    double sup = t.pair_sum ? (double)t.pair_sum / pairs : rows * q;
    int levels = 2;
    while (levels < 12 && sup * q >= (double)thr) {
        sup *= q;
        levels++;
    }
    const double items = (1.0 + sqrt(1.0 + 8.0 * pairs)) / 2.0;
    double sets = pairs, supports = 0;
    for (int k = 3; k <= levels + 1 && items > k - 1; k++) {
        sets *= (items - k + 1) / k;
        supports += sets;
    }
    supports = std::max(supports, ((double)t.triples - pairs) / 2.0);
    const double L = std::min(levels, 7), kw = (double)nw / 1e3, kmax = (double)t.wmax / 1e3;
    const double cta_us = 20.0 + 1.27 * L * kw + 0.23 * supports / 1e3 * kw;
    const double warp_us = (15.0 + 4.6 * L) * kmax + 0.84 * bits / 1e6;
    return warp_us <= cta_us;
}

bool small_plan_takes(const fim_ctx *ctx, int mf, uint32_t flags, const MineState &ms) {
    const ProjTotals t = worst_projection(ctx, mf);
    return search_on_warps(flags, ms) && ctx->n_shards == 1 && !((flags & FIM_LEARNED) && ctx->learned_order) &&
           proj_small_plan_fits(mf) && t.wmax <= kProjWmax && t.words <= kSmallPlanWords && t.rows <= kSmallPlanWords;
}

// One attempt at the whole mine with the current capacities.  Returns
// FIM_OK, or an error; *retry is set when a capacity must grow first.
int mine_once(fim_ctx *ctx, uint32_t thr, uint32_t flags, MineState &ms, bool *retry) {
    cudaStream_t st = ctx->stream;
    *retry = false;
    ctx->cur_thr = thr;
    if ((flags & FIM_LEARNED) && !ctx->has_weights) return FIM_E_STATE;
    MineCounters *d_ctr = ctx->counters.as<MineCounters>();
    const uint32_t maxlen = flags >> 24;
    DbDesc &d = ctx->host_db;  // the one-entry database table of a single-database mine (DFS, compactor)
    d = DbDesc{};
    d.n = ctx->n;
    d.nw = ctx->nw;
    d.nwp = ctx->nwp;
    d.m = ctx->m;
    d.thr = thr;
    d.maxlen = maxlen;
    FIM_TRY(fim_reserve(ctx, ctx->dbdesc, sizeof(DbDesc)));
    ctx->up_desc.clear();  // the batched mine's table is overwritten
    // Few items, and a search the one-launch plan takes: the whole mine is
    // queued at once, sized for m' = m, and m' is read on the device (its
    // read-back in mid-mine left the GPU idle for some 12 us).
    const bool blind = mine_begin_fits(ctx->m) && ctx->m >= 3 && ctx->nw > 0 && (maxlen == 0 || maxlen >= 3) &&
                       !(flags & FIM_PAIRS_POPC) && small_plan_takes(ctx, ctx->m, flags, ms);
    cudaEventRecord(ctx->ev[0], st);
    if (blind) {
        FIM_TRY(fim_reserve(ctx, ctx->pair_cnt, sizeof(int) * (size_t)ctx->m * (size_t)ctx->m + 16));
        FIM_TRY(launch_mine_begin(ctx, d, d_ctr));
        ctx->mfreq = ctx->m;
    } else {
        FIM_CUDA_TRY(cudaMemsetAsync(d_ctr, 0, sizeof(MineCounters), st));
        FIM_TRY(launch_rank_items(ctx, thr, d_ctr));
        if (ctx->shard == 0) FIM_TRY(launch_emit_singletons(ctx, d_ctr));
        FIM_TRY(read_back(ctx, &ctx->host_ctr, d_ctr));
        ctx->mfreq = ctx->host_ctr.m_freq;
        d.mfreq = ctx->mfreq;
        FIM_CUDA_TRY(cudaMemcpyAsync(ctx->dbdesc.p, &d, sizeof(DbDesc), cudaMemcpyHostToDevice, st));
    }
    const int mf = ctx->mfreq;  // m', or its bound m
    cudaEventRecord(ctx->ev[1], st);
    const bool do_pairs = mf >= 2 && (maxlen == 0 || maxlen >= 2);
    const bool do_dfs = do_pairs && mf >= 3 && (maxlen == 0 || maxlen >= 3);
    const bool rep = (flags & (FIM_LEARNED | FIM_DIFFSET_RULE)) != 0;  // classes choose their representation
    const bool net_order = (flags & FIM_LEARNED) && ctx->learned_order;  // the network orders the pair roots
    const bool warp_dfs = do_dfs && search_on_warps(flags, ms);
    // Small matrices of short rows in which an average pair is infrequent: few
    // triples, which the bit columns themselves count sooner than three more
    // launches would (zipf baskets at 2%, us a mine, bit columns against
    // projected: 2,000 x 169 155 and 169, 50,000 x 60 172 and 182).  Where the
    // average pair is frequent, nearly all triples are counted, and whole columns
    // cost more the longer they are (64 items in 5% of the rows each: 8,000 rows
    // 213 and 195, 64,000 341 and 218, 128,000 464 and 231, CTA workers 296); the
    // same for rows that hold a third of the frequent items, which make wide
    // classes (12,060 x 46 at density 0.29: 507 and 343).  With more items than
    // the one-launch plan takes, the plan's totals come back to the host, and the
    // line lies lower.
    bool direct = warp_dfs && (proj_small_plan_fits(mf) ? (int64_t)mf * ctx->nwp <= kDirectWordsShort &&
                                                              3 * ctx->max_row_len <= mf && !avg_pair_frequent(ctx, thr)
                                                        : (int64_t)mf * ctx->nwp <= kDirectWords);
    if (warp_dfs && ctx->dfs_proj >= 0) direct = ctx->dfs_proj == 2;
    // Few frequent items: one launch plans the whole search (pair threshold,
    // roots, projection), sized for the worst case, so that nothing has to
    // come back to the host before the search.
    const size_t npairs_all = (size_t)mf * (size_t)(mf > 0 ? mf - 1 : 0) / 2;
    ProjTotals proj = worst_projection(ctx, mf);
    const bool small_plan = do_dfs && small_plan_takes(ctx, mf, flags, ms);
    // long columns: the plan's totals come back first, to choose the workers
    const bool ask = small_plan && !direct && (ctx->dfs_proj == 0 || (ctx->dfs_proj < 0 && ctx->nw >= kLongWords));
    // automatic: keep low-support classes sparse when the frequent item
    // columns do not fit in half of L2 (streaming whole columns from HBM
    // is latency-bound; from L2 the dense pass is as fast)
    const int sparse_div = ctx->sparse_div >= 0 ? ctx->sparse_div
                           : ((double)mf * (double)ctx->nwp * 4.0 > 0.5 * (double)ctx->l2_bytes ? 4 : 0);
    // sparse copies of the low-support item columns, for the root classes
    // (bounded: at most 1 GiB of (index, word) pairs); a child of a sparse
    // parent is stored sparse, so the copies must fit half a stack level.
    // They depend only on the ranking, so they are made on a side stream
    // while the pair pass runs (their kernel fits beside its CTAs).
    int64_t sp_cap = sparse_div > 0 ? ctx->nw / sparse_div : 0;
    if (sp_cap > ctx->nwp / 2) sp_cap = ctx->nwp / 2;
    const bool sp_fits = do_dfs && sp_cap > 0 && (double)mf * (double)sp_cap * 8.0 <= (double)(1ull << 30);
    const bool sp_items = sp_fits && !warp_dfs;
    if (sp_items) {
        FIM_TRY(reserve_sparse_items(ctx, mf, sp_cap));
        FIM_TRY(fim_aux_stream(ctx));
        for (auto &e : ctx->aux_ev)
            if (!e) FIM_CUDA_TRY(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
        FIM_CUDA_TRY(cudaEventRecord(ctx->aux_ev[0], st));
        FIM_CUDA_TRY(cudaStreamWaitEvent(ctx->aux_stream, ctx->aux_ev[0], 0));
    }
    ctx->stats.pair_path = ctx->stats.pair_rows = 0;
    if (do_pairs) {
        const int mpw = (int)ceil_div64(mf, 32);
        const size_t npairs = (size_t)mf * (mf - 1) / 2;
        FIM_TRY(fim_reserve(ctx, ctx->pair_cnt, sizeof(int) * (size_t)mf * mf));
        FIM_TRY(fim_reserve(ctx, ctx->pairbits, sizeof(uint32_t) * (size_t)mf * mpw));
        FIM_TRY(fim_reserve(ctx, ctx->roots, sizeof(uint32_t) * 3 * npairs));
        const bool rows = !blind && !(flags & FIM_PAIRS_POPC) && pairs_rows_pays(ctx);
        int rc = FIM_E_INVAL;
        if (blind) rc = launch_pairs_tc_blind(ctx);
        else if (!(flags & FIM_PAIRS_POPC))
            rc = rows ? launch_pairs_rows(ctx) : launch_pairs_tc(ctx, 0, true, st, ctx->num_sms);
        if (rc == FIM_OK) {
            ctx->stats.pair_path = 1;
            ctx->stats.pair_rows = rows;
        } else FIM_TRY(launch_pairs_popc(ctx));
        if (sp_items) {  // launched after the pair pass, so that its CTAs take the SMs first
            FIM_TRY(launch_sparse_items(ctx, mf, sp_cap, ctx->aux_stream));
            FIM_CUDA_TRY(cudaEventRecord(ctx->aux_ev[1], ctx->aux_stream));
        }
        if (small_plan) {
            FIM_TRY(reserve_root_plan(ctx, npairs));
            FIM_TRY(launch_proj_small_plan(ctx, mf, thr, d_ctr, !direct && !ask, ask));
        } else {
            FIM_TRY(launch_pairs_finalize(ctx, thr, d_ctr));
        }
        // a shard of a split mine takes only the root classes it owns
        if (ctx->n_shards > 1) FIM_TRY(launch_shard_roots(ctx, d_ctr, ctx->shard, ctx->n_shards));
    }
    cudaEventRecord(ctx->ev[2], st);
    bool on_warps = warp_dfs;
    bool search = do_dfs;
    ctx->dfs_workers = ctx->num_sms * ctx->dfs_ctas_per_sm;
    int items = mf;  // m', or its bound
    if (warp_dfs && !direct && (ask || !small_plan)) {
        if (ask) FIM_TRY(read_back(ctx, &proj, ctx->proj_totals.p, &items, &d_ctr->m_freq));
        else FIM_TRY(launch_proj_plan(ctx, &proj));
        on_warps = proj.words <= kProjWords && proj.wmax <= kProjWmax && proj.cands < 0xFFFFFFFFull;
        if (ctx->dfs_proj == 0) on_warps = false;
        else if (ctx->dfs_proj < 0 && ctx->nw >= kLongWords && proj.cands > 0)
            on_warps = on_warps && projection_pays(proj, ctx->nw, (double)ctx->n, thr);
        // no item has two later partners: there is no third item to try, and
        // neither triples nor root classes are planned for a search
        search = proj.cands > 0;
    }
    if (search) {
        const int workers = ctx->dfs_workers * (on_warps ? proj_workers_per_cta() : 1);
        ctx->dfs_workers = workers;
        // deepest class: a prefix can hold at most min(longest row, m') items
        int bound = ctx->max_row_len < mf ? ctx->max_row_len : mf;
        if (maxlen && (int)maxlen < bound) bound = (int)maxlen;
        if (bound > 240) bound = 240;  // the worker's shared-memory frame arrays hold 256 levels
        const int levels_needed = bound > 2 ? bound - 1 : 1;
        ProjParams q{};
        if (on_warps) {
            const bool triples = !direct && ctx->n_shards == 1 && !net_order && proj.triples <= kTriples;
            if (ask && triples)  // the plan has counted the pairs as roots; the triple pass brings its own
                FIM_CUDA_TRY(cudaMemsetAsync(&d_ctr->pending, 0, sizeof(d_ctr->pending), st));
            if (!direct) FIM_TRY(launch_projection(ctx, mf, proj, small_plan, triples, thr));
            if (triples) {
                q.triple = ctx->proj_triple.as<uint32_t>();
                q.roots = ctx->proj_roots.as<unsigned long long>();
            } else if (!small_plan) {  // candidate-less pairs dropped, the others ordered
                FIM_TRY(reserve_root_plan(ctx, npairs_all));
                FIM_TRY(launch_root_plan(ctx, d_ctr, npairs_all, nullptr, net_order ? 2 : ctx->root_sort, nullptr, st));
            }
            q.items = ctx->proj_items.as<ProjItem>();
            q.mat = ctx->proj_mat.as<uint32_t>();
            q.cands = ctx->proj_cands.as<uint32_t>();
            q.direct = direct ? 1 : 0;
            q.direct_words = (int)round_up64(ctx->nw, 4);
            const int64_t level = direct ? q.direct_words : (int64_t)proj.wmax;
            // one level more than the classes: a queued task's own prefix
            q.gstack = min64((int64_t)(levels_needed + 1) * level,
                             (int64_t)(kProjStackBudget / sizeof(uint32_t)) / workers / 4 * 4);
            if (q.gstack < 4) q.gstack = 4;
            FIM_TRY(fim_reserve(ctx, ctx->stack_bits, sizeof(uint32_t) * (size_t)workers * (size_t)q.gstack));
        } else {
            const size_t per_level = (size_t)workers * (size_t)ctx->nwp * sizeof(uint32_t);
            if (ms.depth_cap == 0) {
                size_t cap = ms.stack_budget / (per_level ? per_level : 1);
                ms.depth_cap = (int)(cap < (size_t)levels_needed ? cap : (size_t)levels_needed);
                if (ms.depth_cap < 2) ms.depth_cap = 2;
            }
            FIM_TRY(fim_reserve(ctx, ctx->stack_bits, per_level * (size_t)ms.depth_cap));
        }
        if (ms.frame_pool == 0) ms.frame_pool = 4LL * mf + 1024;
        FIM_TRY(fim_reserve(ctx, ctx->frame_items, sizeof(uint32_t) * (size_t)workers * ms.frame_pool));
        if (!on_warps || rep) FIM_TRY(fim_reserve(ctx, ctx->frame_sups, sizeof(uint32_t) * (size_t)workers * ms.frame_pool));
        FIM_TRY(prepare_task_queue(ctx, sizeof(Task) * kTaskCap));
        FIM_TRY(fim_reserve(ctx, ctx->cand_pool, sizeof(uint32_t) * kCandPoolCap));
        if (!small_plan) FIM_TRY(launch_epoch_bump(ctx));
        const size_t npairs = (size_t)mf * (mf - 1) / 2;
        DfsParams p{};
        p.dbs = ctx->dbdesc.as<DbDesc>();
        p.bm = ctx->bm.as<uint32_t>();
        p.perm = ctx->perm.as<int32_t>();
        p.pairbits = ctx->pairbits.as<uint32_t>();
        p.nwp_max = ctx->nwp;
        p.root_a = ctx->roots.as<uint32_t>();
        p.root_b = p.root_a + npairs;
        p.root_sup = p.root_a + 2 * npairs;
        p.root_db = nullptr;
        p.rec_db = ctx->rec_db.as<uint32_t>();
        p.tasks = ctx->tasks.as<Task>();
        p.task_cap = kTaskCap;
        p.cand_pool = ctx->cand_pool.as<uint32_t>();
        p.cand_pool_cap = kCandPoolCap;
        p.split_depth = (flags & FIM_NO_SPLIT) ? 0 : ctx->split_depth;
        p.stack_bits = ctx->stack_bits.as<uint32_t>();
        p.frame_items = ctx->frame_items.as<uint32_t>();
        p.frame_sups = ctx->frame_sups.as<uint32_t>();
        p.frame_pool = ms.frame_pool;
        p.depth_cap = ms.depth_cap;
        p.rec_off = ctx->rec_off.as<unsigned long long>();
        p.rec_len = ctx->rec_len.as<uint32_t>();
        p.rec_sup = ctx->rec_sup.as<uint32_t>();
        p.rec_items = ctx->rec_items.as<uint32_t>();
        p.rec_cap = ctx->rec_cap;
        p.rec_items_cap = ctx->rec_items_cap;
        p.ctr = d_ctr;
        p.spin_limit = (unsigned long long)ctx->spin_limit_ms * 1000000ull;
        p.withhold_slot = ctx->test_withhold_task;
        p.sparse_div = sparse_div;
        p.epoch = ctx->epoch.as<uint32_t>();
        p.learned_kmin = ctx->learned_kmin;
        p.rec_chunk = ctx->rec_chunk;
        p.root_reverse = ctx->root_reverse;
        const bool sp_late = sp_fits && warp_dfs && !on_warps;
        if (sp_late) {  // the warp workers' projection was too large, or did not pay, after all
            FIM_TRY(reserve_sparse_items(ctx, items, sp_cap));
            FIM_TRY(launch_sparse_items(ctx, items, sp_cap, st));
        }
        if (sp_items || sp_late) {
            if (sp_items) FIM_CUDA_TRY(cudaStreamWaitEvent(st, ctx->aux_ev[1], 0));
            p.item_idx = ctx->sp_idx.as<uint32_t>();
            p.item_val = ctx->sp_val.as<uint32_t>();
            p.item_z = ctx->sp_z.as<int>();
            p.item_cap = sp_cap;
        }
        p.pair_cnt = ctx->pair_cnt.as<int>();
        p.item_sup = ctx->item_sup.as<uint32_t>();
        p.root_order = nullptr;
        p.learned = (flags & FIM_LEARNED) ? 1 : 0;
        p.diffset_rule = (flags & FIM_DIFFSET_RULE) ? 1 : 0;
        p.mlp_w = ctx->mlp_wbf.as<__nv_bfloat16>();
        if (on_warps) {
            p.root_order = q.triple ? nullptr : ctx->root_order.as<uint32_t>();
        } else {  // candidate-less roots dropped, the others ordered
            if (!small_plan) {  // (the one-launch plan has done so)
                const int mode = (p.learned && ctx->learned_order) ? 2 : ctx->root_sort;
                FIM_TRY(reserve_root_plan(ctx, npairs));
                FIM_TRY(launch_root_plan(ctx, d_ctr, npairs, nullptr, mode, nullptr, st));
            }
            p.root_order = ctx->root_order.as<uint32_t>();
        }
        p.trace = (flags & FIM_TRACE) ? 1 : 0;
        if (p.trace) {
            // complete subtree totals need every subtree inside one worker
            p.split_depth = 0;
            if (ctx->trace_cap == 0) ctx->trace_cap = 1ull << 21;
            FIM_TRY(fim_reserve(ctx, ctx->trace_x, sizeof(float) * FIM_MLP_FEATURES * ctx->trace_cap));
            FIM_TRY(fim_reserve(ctx, ctx->trace_y, sizeof(float) * 2 * ctx->trace_cap));
            p.trace_x = ctx->trace_x.as<float>();
            p.trace_y = ctx->trace_y.as<float>();
            p.trace_cap = ctx->trace_cap;
        }
        if (on_warps) FIM_TRY(launch_dfs_proj(ctx, p, q, ctx->dfs_ctas_per_sm));
        else FIM_TRY(launch_dfs(ctx, p, workers, ctx->dfs_block));
    }
    cudaEventRecord(ctx->ev[3], st);
    FIM_TRY(read_back(ctx, &ctx->host_ctr, d_ctr));
    const MineCounters &c = ctx->host_ctr;
    ctx->mfreq = c.m_freq;
    if (c.err == FIM_E_STACK && on_warps) {
        ms.cta_dfs = true;
        *retry = true;
        return FIM_OK;
    }
    if (c.err == FIM_E_STACK) {
        if (ms.stack_budget >= kStackBudgetMax) return FIM_E_STACK;
        ms.stack_budget *= 2;
        ms.depth_cap = ms.depth_cap * 2 > 240 ? 240 : ms.depth_cap * 2;
        ms.frame_pool *= 2;
        *retry = true;
        return FIM_OK;
    }
    if (c.err != 0) return c.err;
    if (c.overflow) {
        ctx->rec_cap = c.n_records + c.n_records / 4 + 1024;
        ctx->rec_items_cap = c.n_rec_items + c.n_rec_items / 4 + 4096;
        FIM_TRY(fim_reserve(ctx, ctx->rec_off, sizeof(unsigned long long) * ctx->rec_cap));
        FIM_TRY(fim_reserve(ctx, ctx->rec_len, sizeof(uint32_t) * ctx->rec_cap));
        FIM_TRY(fim_reserve(ctx, ctx->rec_sup, sizeof(uint32_t) * ctx->rec_cap));
        FIM_TRY(fim_reserve(ctx, ctx->rec_items, sizeof(uint32_t) * ctx->rec_items_cap));
    FIM_TRY(fim_reserve(ctx, ctx->rec_db, sizeof(uint32_t) * ctx->rec_cap));
        *retry = true;
        return FIM_OK;
    }
    drop_slots_past_arena(ctx);
    int lmax = c.max_len;
    if (ctx->shard == 0 && c.m_freq >= 1 && lmax < 1) lmax = 1;
    const unsigned long long n_sets = c.n_records - c.rec_holes;
    if (ctx->shard == 0 && n_sets > (unsigned long long)c.m_freq && lmax < 2) lmax = 2;
    ctx->host_ctr.max_len = lmax;
    FIM_TRY(launch_compact(ctx, c.n_records, n_sets, 1, ctx->m));
    cudaEventRecord(ctx->ev[4], st);
    FIM_CUDA_TRY(cudaGetLastError());
    // the mine returns with the compaction queued: the next call that reads
    // results (or these phase times) synchronises the stream first
    ctx->phase_times_pending = true;
    return FIM_OK;
}

}  // namespace

extern "C" {

int fim_mine(fim_ctx *ctx, uint64_t minsup, uint32_t flags) {
    FIM_NVTX("fim_mine");
    if (!ctx) return FIM_E_INVAL;
    if (!ctx->built) return FIM_E_STATE;
    if (!(flags & FIM_STRICT) && minsup == 0) return FIM_E_INVAL;
    DeviceGuard g(ctx->device);
    if (!g.ok) return FIM_E_CUDA;
    FIM_TRY(fim_finish_phase_times(ctx));  // before the events are recorded again
    ctx->mined = false;
    ctx->mflags = flags;
    uint64_t thr64 = (flags & FIM_STRICT) ? minsup + 1 : minsup;
    if ((flags & FIM_STRICT) && minsup == UINT64_MAX) thr64 = UINT64_MAX;
    const uint32_t thr = thr64 > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)thr64;
    if (ctx->test_record_cap > 0) {
        ctx->rec_cap = (unsigned long long)ctx->test_record_cap;
        if (ctx->rec_items_cap == 0) ctx->rec_items_cap = 1ull << 23;
    } else if (ctx->rec_cap == 0) {
        ctx->rec_cap = 1ull << 20;
        ctx->rec_items_cap = 1ull << 23;
    }
    FIM_TRY(fim_reserve(ctx, ctx->rec_off, sizeof(unsigned long long) * ctx->rec_cap));
    FIM_TRY(fim_reserve(ctx, ctx->rec_len, sizeof(uint32_t) * ctx->rec_cap));
    FIM_TRY(fim_reserve(ctx, ctx->rec_sup, sizeof(uint32_t) * ctx->rec_cap));
    FIM_TRY(fim_reserve(ctx, ctx->rec_items, sizeof(uint32_t) * ctx->rec_items_cap));
    FIM_TRY(fim_reserve(ctx, ctx->rec_db, sizeof(uint32_t) * ctx->rec_cap));
    const uint64_t launches0 = ctx->launches;
    MineState ms;
    bool retry = true;
    for (int attempt = 0; retry && attempt < 8; attempt++) FIM_TRY(mine_once(ctx, thr, flags, ms, &retry));
    if (retry) return FIM_E_NOMEM;
    const MineCounters &c = ctx->host_ctr;
    fim_stats &s = ctx->stats;
    s.n_trans = (uint64_t)ctx->n;
    s.n_items = (uint64_t)ctx->m;
    s.n_frequent_items = (uint64_t)ctx->mfreq;
    s.n_sets = c.n_records - c.rec_holes;
    s.max_len = (uint64_t)c.max_len;
    s.supports_singletons = (uint64_t)ctx->m;
    const uint64_t mf = (uint64_t)ctx->mfreq;
    const uint32_t maxlen = flags >> 24;
    s.supports_pairs = (mf >= 2 && (maxlen == 0 || maxlen >= 2)) ? mf * (mf - 1) / 2 : 0;
    s.supports_dfs = c.supports_dfs;
    s.dfs_words = c.dfs_words;
    s.dfs_bytes = c.dfs_bytes;
    s.dfs_touched_bytes = c.dfs_touched;
    s.classes = c.classes;
    s.tasks_pushed = c.pushed;
    s.diffset_classes = c.diffset;
    s.launches_mine = ctx->launches - launches0;
    s.dfs_busy_ns = c.busy_ns;
    s.dfs_span_ns = c.t_last > c.t_first && c.t_first != 0 ? c.t_last - c.t_first : 0;
    s.dfs_workers = (uint64_t)ctx->dfs_workers;
    s.dfs_root_ns = c.root_ns;
    if (ctx->bytes_held > s.peak_device_bytes) s.peak_device_bytes = ctx->bytes_held;
    if (ctx->debug_checks) FIM_TRY(run_check_output(ctx, thr));
    ctx->out_n = ctx->n;
    ctx->mined = true;
    ctx->mine_serial++;
    return FIM_OK;
}

int fim_mine_shard(fim_ctx *ctx, uint64_t minsup, uint32_t flags, int shard, int n_shards) {
    FIM_NVTX("fim_mine_shard");
    if (!ctx || n_shards < 1 || n_shards > FIM_MAX_SHARDS || shard < 0 || shard >= n_shards) return FIM_E_INVAL;
    ctx->shard = shard;
    ctx->n_shards = n_shards;
    const int rc = fim_mine(ctx, minsup, flags);
    ctx->shard = 0;
    ctx->n_shards = 1;
    return rc;
}

int fim_fetch_results(fim_ctx *ctx, uint64_t *n_sets, uint64_t *n_items_total, uint64_t *offsets,
                      uint32_t *items, uint32_t *supports, uint64_t cap_sets, uint64_t cap_items,
                      uint32_t flags) {
    FIM_NVTX("fim_fetch_results");
    if (!ctx || !n_sets || !n_items_total) return FIM_E_INVAL;
    if (!ctx->mined) return FIM_E_STATE;
    *n_sets = ctx->out_sets;
    *n_items_total = ctx->out_items_total;
    if (!offsets && !items && !supports) return FIM_OK;
    if (!offsets || !supports || (!items && ctx->out_items_total)) return FIM_E_INVAL;
    if (cap_sets < ctx->out_sets || cap_items < ctx->out_items_total) return FIM_E_TOO_SMALL;
    DeviceGuard g(ctx->device);
    if (!g.ok) return FIM_E_CUDA;
    const cudaMemcpyKind k = (flags & FIM_OUTPUT_DEVICE) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    cudaStream_t st = ctx->stream;
    FIM_CUDA_TRY(cudaMemcpyAsync(offsets, ctx->out_off.p, sizeof(uint64_t) * (ctx->out_sets + 1), k, st));
    if (ctx->out_items_total)
        FIM_CUDA_TRY(cudaMemcpyAsync(items, ctx->out_items.p, sizeof(uint32_t) * ctx->out_items_total, k, st));
    if (ctx->out_sets)
        FIM_CUDA_TRY(cudaMemcpyAsync(supports, ctx->out_sup.p, sizeof(uint32_t) * ctx->out_sets, k, st));
    FIM_TRY(queue_compact_status(ctx));
    FIM_CUDA_TRY(cudaStreamSynchronize(st));
    return compact_status(ctx);
}

int fim_get_stats(const fim_ctx *ctx, fim_stats *out) {
    FIM_NVTX("fim_get_stats");
    if (!ctx || !out) return FIM_E_INVAL;
    // the ctx is the caller's own (non-const) object; the phase times of a
    // mine still in flight are read here, after it has finished
    FIM_TRY(fim_finish_phase_times(const_cast<fim_ctx *>(ctx)));
    *out = ctx->stats;
    return FIM_OK;
}

int fim_set_tuning(fim_ctx *ctx, const char *key, int64_t v) {
    FIM_NVTX("fim_set_tuning");
    if (!ctx || !key) return FIM_E_INVAL;
    struct Knob { const char *name; int *field; int64_t lo, hi; } knobs[] = {
        {"dfs_ctas_per_sm", &ctx->dfs_ctas_per_sm, 1, 4},
        {"dfs_threads", &ctx->dfs_block, 256, 512},
        {"split_depth", &ctx->split_depth, 0, FIM_TASK_MAXR},
        {"sparse_div", &ctx->sparse_div, -1, 64},
        {"learned_kmin", &ctx->learned_kmin, 1, 1 << 20},
        {"learned_order", &ctx->learned_order, 0, 1},
        {"root_reverse", &ctx->root_reverse, 0, 1},
        {"pairs_split", &ctx->pairs_split, 0, 4096},
        {"pairs_kdrain", &ctx->pairs_kdrain, 0, 32768},
        {"pairs_rows", &ctx->pairs_rows, -1, 1},
        {"upload_chunks", &ctx->upload_chunks, 1, 16},
        {"compact_cluster", &ctx->compact_cluster, 0, 1},
        {"upload_mapped", &ctx->upload_mapped, 0, 1},
        {"batch_stream_copies", &ctx->batch_stream_copies, 0, 1},
        {"spin_limit_ms", &ctx->spin_limit_ms, 1, 600000},
        {"debug_checks", &ctx->debug_checks, 0, 1},
        {"test_withhold_task", &ctx->test_withhold_task, -1, 1 << 20},
        {"test_withhold_tile", &ctx->test_withhold_tile, -1, 1 << 20},
        {"test_memory_mb", &ctx->test_memory_mb, 0, 1 << 30},
        {"test_record_cap", &ctx->test_record_cap, 0, 1 << 30},
        {"upload_streams", &ctx->upload_streams, 1, 2},
        {"batch_pairs_shape", &ctx->batch_pairs_shape, 0, kBatchPairsShapeCount - 1},
        {"batch_build_block", &ctx->batch_build_block, 16, 64},
        {"batch_build_coal", &ctx->batch_build_coal, 0, 1},
        {"batch_pairs_pack", &ctx->batch_pairs_pack, 0, 1},
        {"batch_group_dfs", &ctx->batch_group_dfs, 0, 1},
        {"root_sort", &ctx->root_sort, 0, 1},
        {"record_chunk", &ctx->rec_chunk, 1, 1024},
        {"batch_segments", &ctx->batch_segments, 0, 16},
        {"dfs_proj", &ctx->dfs_proj, -1, 2},
        {"dfs_warp", &ctx->dfs_warp, 0, 1},
        {"dfs_warp_ctas", &ctx->dfs_warp_ctas, 2, 3},
    };
    for (const Knob &k : knobs)
        if (strcmp(k.name, key) == 0) {
            if (v < k.lo || v > k.hi) return FIM_E_INVAL;
            // the DFS worker exists in two widths; a worker is capped at 64
            // registers a thread, so at most 1024 worker threads fit an SM
            if (k.field == &ctx->dfs_block && v != 256 && v != 512) return FIM_E_INVAL;
            if (k.field == &ctx->batch_build_block && v != 16 && v != 32 && v != 64) return FIM_E_INVAL;
            const int64_t block = k.field == &ctx->dfs_block ? v : ctx->dfs_block;
            const int64_t per_sm = k.field == &ctx->dfs_ctas_per_sm ? v : ctx->dfs_ctas_per_sm;
            if (block * per_sm > 1024) return FIM_E_INVAL;
            *k.field = (int)v;
            return FIM_OK;
        }
    return FIM_E_INVAL;
}

}  // extern "C"
