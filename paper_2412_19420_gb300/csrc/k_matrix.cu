// k_matrix.cu -- matrix construction (Eq. 1), singleton support (Eq. 3) and the
// internal ids.
//
// build_bitmaps_kernel: one CTA owns a block of WB words (32*WB transactions)
// and a range of IB items.  Each warp streams a 32-row group's elements
// (coalesced) and ORs every (transaction, item) pair into a shared-memory
// tile with atomicOr -- OR makes repeated items idempotent, which is the set
// membership of Eq. 1 -- and the tile goes out as WB-word (64- or 32-byte)
// runs of each item column with 16-byte stores.  The CTA also validates
// its slice of the CSR (monotone indptr, items in [0, m)).  CMP: the CSR is
// compact (uint32 row offsets, uint16 item ids) instead of int64 / int32.
#include <type_traits>

#include "fim_common.cuh"

namespace {

// WB: words per CTA tile row; T: threads; T / 32 / WB warps share a 32-row group.
template <bool CMP, int WB, int T>
__global__ void __launch_bounds__(T)
build_bitmaps_kernel(const void *__restrict__ indptr_v, const void *__restrict__ indices_v,
                     int64_t n, int32_t m, int64_t nnz, int64_t nwp, int ib, int ms, int64_t blk0,
                     uint32_t *__restrict__ bm, uint32_t *__restrict__ sup, BuildFlags *__restrict__ flags,
                     RowCopy rows) {
    using Off = typename std::conditional<CMP, uint32_t, int64_t>::type;
    using Id = typename std::conditional<CMP, unsigned short, int32_t>::type;
    const Off *const indptr = static_cast<const Off *>(indptr_v);
    const Id *const indices = static_cast<const Id *>(indices_v);
    // [WB][ms], word-major and padded: the 32 rows of a warp's group share
    // their word, so their items' bits spread over the banks
    extern __shared__ __align__(16) uint32_t tile[];
    __shared__ int s_max;
    __shared__ unsigned s_tile;
    __shared__ unsigned long long s_pairs;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int SPLIT = T / 32 / WB;
    static_assert(T == 32 * WB * SPLIT && (WB == 8 || WB == 16), "whole warps per row group");
    const int sub = warp % SPLIT;  // of the warps sharing a group
    const int64_t w0 = (blk0 + (int64_t)blockIdx.x) * WB;
    const int i0 = blockIdx.y * ib;
    const int icount = min(ib, m - i0);
    const int64_t t0 = w0 * 32;
    const int64_t t1 = min(n, t0 + WB * 32);
    int bad = 0, my_max = 0;
    unsigned long long my_pairs = 0;
    unsigned my_tile = 0;
    if (nnz < 0) {  // device input: indptr[n] read here, and indptr[0] checked once
        nnz = (int64_t)indptr[n];
        if (nnz < 0) bad = 1;
        if (blockIdx.x == 0 && blockIdx.y == 0 && blk0 == 0 && threadIdx.x == 0 && indptr[0] != 0) bad = 1;
    }
    const bool first = blockIdx.y == 0;  // this CTA's items are the first: it also sees to the rows
    // (a matrix without ids is within a cap of 0: where no rows are kept there is nowhere to write)
    const bool copy = first && rows.ptr != nullptr && (uint64_t)nnz <= rows.cap;
    if (first && blk0 == 0 && blockIdx.x == 0 && threadIdx.x == 0) flags->nnz = nnz;

    for (int k = threadIdx.x; k < WB / 4 * ms; k += T) reinterpret_cast<uint4 *>(tile)[k] = make_uint4(0, 0, 0, 0);
    if (threadIdx.x == 0) {
        s_max = 0;
        s_tile = 0;
        s_pairs = 0;
    }
    __syncthreads();
    // warp w takes 32-row groups: lane i holds the group's start of row i, the
    // warp streams the group's elements 32 at a time (coalesced) and each
    // element finds its row by a binary search over the lanes' starts
    for (int64_t rb = t0 + 32 * (warp / SPLIT); rb < t1; rb += 32 * WB) {
        const int nr = (int)min64(32, t1 - rb);
        const int64_t off = (int64_t)indptr[rb + (lane < nr ? lane : nr)];
        const int64_t e_end = (int64_t)indptr[rb + nr];
        int64_t off_next = __shfl_down_sync(0xffffffffu, off, 1);
        if (lane == nr - 1) off_next = e_end;
        unsigned pairs = 0;  // of this row, for the group's sum
        if (lane < nr) {
            if (off_next < off || off < 0 || off_next > nnz) bad = 1;
            else if (sub == 0) {
                const int64_t len = off_next - off;
                my_max = max(my_max, (int)min64(len, 1 << 30));
                const unsigned long long np = (unsigned long long)len * (unsigned long long)(len - 1) / 2;
                my_pairs += np;
                pairs = (unsigned)min64((int64_t)(len > kRowLong ? 2 * np : np), 1 << 26);
                if (copy) rows.ptr[rb + lane] = (uint32_t)off;
                if (copy && rb + lane == n - 1) rows.ptr[n] = (uint32_t)off_next;
            }
        }
        if (__any_sync(0xffffffffu, bad)) continue;  // malformed: flagged, not read
        if (first && sub == 0) my_tile = max(my_tile, __reduce_add_sync(0xffffffffu, pairs));
        const int64_t e_begin = __shfl_sync(0xffffffffu, off, 0);
        const uint32_t wl = (uint32_t)((rb - t0) >> 5);
        // Rows all hold an id (the usual case): their starts are distinct, one
        // OR over the lanes marks those inside a chunk of 32 ids, and an id's
        // row is a popcount away; else a binary search over the starts.
        const bool dense = e_end - e_begin < (1ll << 30) && !__any_sync(0xffffffffu, lane < nr && off_next == off);
        const int ar = dense ? (int)(off - e_begin) : 0;
        int before = -1;  // rows begun before the chunk, less one
        for (int64_t e0 = e_begin + 32 * sub; e0 < e_end; e0 += 32 * SPLIT) {
            const int64_t e = e0 + lane;
            const bool v = e < e_end;
            const int32_t it = v ? (int32_t)indices[e] : 0;
            int r = 0;  // largest r < nr with start(r) <= e
            if (dense) {
                const int at = (int)(e0 - e_begin);
                const unsigned in = (unsigned)(ar - at);
                if (SPLIT > 1) before = __popc(__ballot_sync(0xffffffffu, lane < nr && ar < at)) - 1;
                const uint32_t heads = __reduce_or_sync(0xffffffffu, lane < nr && in < 32u ? 1u << in : 0u);
                r = before + __popc(heads & (0xFFFFFFFFu >> (31 - lane)));
                if (SPLIT == 1) before += __popc(heads);
            } else {
#pragma unroll
                for (int step = 16; step > 0; step >>= 1) {
                    const int c = r + step;
                    const int64_t oc = __shfl_sync(0xffffffffu, off, c < 32 ? c : 31);
                    if (c < nr && oc <= e) r = c;
                }
            }
            if (!v) continue;
            if (it < 0 || it >= m) { bad = 1; continue; }
            if (copy) rows.idx[e] = (unsigned short)it;
            if (it < i0 || it >= i0 + icount) continue;
            atomicOr(&tile[wl * ms + (it - i0)], 1u << r);
        }
    }
    if (bad) atomicExch(&flags->bad, 1);
    if (first) {  // one pair of global atomics per CTA
        my_max = (int)__reduce_max_sync(0xffffffffu, (unsigned)my_max);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) my_pairs += __shfl_xor_sync(0xffffffffu, my_pairs, o);
        if (lane == 0) {
            atomicMax(&s_max, my_max);
            atomicMax(&s_tile, my_tile);
            atomicAdd(&s_pairs, my_pairs);
        }
    }
    __syncthreads();
    if (first && threadIdx.x == 0 && s_max > 0) {
        atomicMax(&flags->max_len, s_max);
        atomicMax(&flags->tile_pairs, s_tile);
        atomicAdd(&flags->row_pairs, s_pairs);
    }
    // write-out: 16-byte stores, WB / 4 consecutive threads per column; the
    // column's popcount rides along into S(I_j) (Eq. 3).  (A pass of its own over
    // the columns read all of them back: 0.9 ms on 10^7 x 5,000.)
    for (int b = 0; b < icount * (WB / 4); b += T) {  // block-uniform trips
        const int k = b + threadIdx.x;
        const int r = k / (WB / 4), c = k % (WB / 4);
        uint32_t cnt = 0;
        if (r < icount) {
            const uint4 v = make_uint4(tile[(4 * c + 0) * ms + r], tile[(4 * c + 1) * ms + r],
                                       tile[(4 * c + 2) * ms + r], tile[(4 * c + 3) * ms + r]);
            *reinterpret_cast<uint4 *>(bm + (int64_t)(i0 + r) * nwp + w0 + 4 * c) = v;
            cnt = __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
        }
        cnt += __shfl_xor_sync(0xffffffffu, cnt, 1);
        if (WB == 16) cnt += __shfl_xor_sync(0xffffffffu, cnt, 2);
        if (c == 0 && cnt) atomicAdd(&sup[i0 + r], cnt);
    }
}

// Internal ids: frequent items ordered by (support, id) ascending.  One warp
// per item counts the frequent items with a smaller key (ties impossible).
__global__ void rank_items_kernel(const uint32_t *__restrict__ sup, int32_t m, uint32_t thr,
                                  int32_t *__restrict__ perm, int32_t *__restrict__ rank,
                                  MineCounters *ctr) {
    const int lane = threadIdx.x & 31;
    const int j = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (j >= m) return;
    if (j == 0) {  // the supports' sum tells whether a row repeats an item
        unsigned long long t = 0;
        for (int i = lane; i < m; i += 32) t += sup[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) ctr->sup_sum = t;
    }
    const uint32_t sj = sup[j];
    if (sj < thr) {
        if (lane == 0) rank[j] = -1;
        return;
    }
    uint32_t below = 0;
    for (int i = lane; i < m; i += 32) {
        uint32_t si = sup[i];
        below += (si >= thr) && (si < sj || (si == sj && i < j));
    }
    below = warp_sum_u32(below);
    if (lane == 0) {
        rank[j] = (int32_t)below;
        perm[below] = j;
        atomicAdd(&ctr->m_freq, 1);
    }
}

// Singletons are the first m' records: record r = {r} with support S(perm[r]).
__global__ void emit_singletons_kernel(const uint32_t *__restrict__ sup, const int32_t *__restrict__ perm,
                                       MineCounters *ctr, unsigned long long *rec_off,
                                       uint32_t *rec_len, uint32_t *rec_sup, uint32_t *rec_items,
                                       unsigned long long rec_cap, unsigned long long items_cap) {
    const int mf = ctr->m_freq;
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r == 0) {
        ctr->n_records = (unsigned long long)mf;
        ctr->n_rec_items = (unsigned long long)mf;
        if ((unsigned long long)mf > rec_cap) atomicOr(&ctr->overflow, 1);
        if ((unsigned long long)mf > items_cap) atomicOr(&ctr->overflow, 2);
    }
    if (r < mf && (unsigned long long)r < rec_cap && (unsigned long long)r < items_cap) {
        rec_off[r] = (unsigned long long)r;
        rec_len[r] = 1;
        rec_sup[r] = sup[perm[r]];
        rec_items[r] = (uint32_t)r;
    }
}

// The start of a mine with at most MB_MAX items, in one CTA: the counters and the
// pair counts cleared, internal ids, singleton records and the database table.
// (A clear, two kernels, a read-back of m' and an upload of the table before:
// with the read-back in the middle of the mine gone, and the others through
// page-locked memory, a 10,000 x 169 mine went from 205 to 173 us.)
constexpr int MB_T = 1024, MB_MAX = 256;
__global__ void __launch_bounds__(MB_T)
mine_begin_kernel(DbDesc d, const uint32_t *__restrict__ sup, MineCounters *ctr, DbDesc *__restrict__ dbs,
                  int32_t *__restrict__ perm, int32_t *__restrict__ rank, int *__restrict__ pair_cnt,
                  unsigned long long *__restrict__ rec_off, uint32_t *__restrict__ rec_len,
                  uint32_t *__restrict__ rec_sup, uint32_t *__restrict__ rec_items, unsigned long long rec_cap,
                  unsigned long long items_cap) {
    __shared__ uint32_t s[MB_MAX];
    const int j = threadIdx.x, m = d.m;
    for (int i = j; i < (int)(sizeof(MineCounters) / 4); i += MB_T) reinterpret_cast<uint32_t *>(ctr)[i] = 0u;
    for (int i = j; i < (m * m + 3) / 4; i += MB_T) reinterpret_cast<int4 *>(pair_cnt)[i] = make_int4(0, 0, 0, 0);
    const uint32_t sj = j < m ? sup[j] : 0u;
    if (j < m) s[j] = sj;
    const bool f = j < m && sj >= d.thr;
    const int mf = __syncthreads_count(f);
    if (j < m && !f) rank[j] = -1;
    if (f) {
        int below = 0;
        for (int i = 0; i < m; i++) {
            const uint32_t si = s[i];
            below += si >= d.thr && (si < sj || (si == sj && i < j));
        }
        rank[j] = below;
        perm[below] = j;
        if ((unsigned long long)below < rec_cap && (unsigned long long)below < items_cap) {
            rec_off[below] = (unsigned long long)below;
            rec_len[below] = 1;
            rec_sup[below] = sj;
            rec_items[below] = (uint32_t)below;
        }
    }
    if (j == 0) {
        ctr->m_freq = mf;
        ctr->n_records = (unsigned long long)mf;
        ctr->n_rec_items = (unsigned long long)mf;
        if ((unsigned long long)mf > rec_cap) ctr->overflow = 1;
        else if ((unsigned long long)mf > items_cap) ctr->overflow = 2;
        d.mfreq = mf;
        *dbs = d;
    }
}

}  // namespace

bool mine_begin_fits(int m) { return m <= MB_MAX; }

int launch_mine_begin(fim_ctx *ctx, const DbDesc &d, MineCounters *d_ctr) {
    ctx->launches++;
    mine_begin_kernel<<<1, MB_T, 0, ctx->stream>>>(
        d, ctx->item_sup.as<uint32_t>(), d_ctr, ctx->dbdesc.as<DbDesc>(), ctx->perm.as<int32_t>(),
        ctx->rank.as<int32_t>(), ctx->pair_cnt.as<int>(), ctx->rec_off.as<unsigned long long>(),
        ctx->rec_len.as<uint32_t>(), ctx->rec_sup.as<uint32_t>(), ctx->rec_items.as<uint32_t>(), ctx->rec_cap,
        ctx->rec_items_cap);
    FIM_CUDA_TRY(cudaGetLastError());
    return FIM_OK;
}

int launch_build_bitmaps(fim_ctx *ctx, const void *d_indptr, const void *d_indices, int64_t nnz,
                         const void *h_indptr, const void *h_indices, bool cmp) {
    const size_t ib_bytes = csr_id_bytes(cmp);
    // Up to 1,024 items: 64-byte runs, several CTAs an SM.  More: 32-byte runs of
    // up to 7,200 items and one CTA an SM, four warps to a row group, so that
    // every id is read once (blocks of 1,024 items read the ids m / 1,024
    // times): 10^7 x 5,000 3.13 -> 2.92 ms, 100,000 x 2,000 75 -> 67 us from
    // device memory; from mapped host memory the ids cross the link once.  (512
    // threads 3.25 ms, two blocks of 2,500 items 2.95, two CTAs an SM 3.85.)
    const bool wide = ctx->m > 1024;
    const int WB = wide ? 8 : 16, T = wide ? 1024 : 512, most = wide ? 7200 : 1024;
    auto kern = cmp ? build_bitmaps_kernel<true, 16, 512> : build_bitmaps_kernel<false, 16, 512>;
    if (wide) kern = cmp ? build_bitmaps_kernel<true, 8, 1024> : build_bitmaps_kernel<false, 8, 1024>;
    const int64_t nblk = ctx->nwp / WB;
    const int niblk = (int)ceil_div64(ctx->m > 0 ? ctx->m : 1, most);
    int ib = (int)ceil_div64(ctx->m, niblk);
    if (ib < 1) ib = 1;
    // the write-out's four (two) threads of a column on banks of their own
    // (10^7 x 5,000 3.31 -> 3.13 ms)
    const int ms = ib + ((WB == 16 ? 2 : 4) - ib % 8 + 8) % 8;
    const size_t smem = (size_t)ms * WB * sizeof(uint32_t);
    FIM_CUDA_TRY(fim_allow_smem(kern, (size_t)(most + 8) * WB * sizeof(uint32_t)));
    BuildFlags *flags = ctx->dev_flag.as<BuildFlags>();
    cudaStream_t st = ctx->stream;
    FIM_CUDA_TRY(cudaMemsetAsync(flags, 0, sizeof(BuildFlags), st));
    FIM_CUDA_TRY(cudaMemsetAsync(ctx->item_sup.p, 0, sizeof(uint32_t) * (size_t)ctx->m, st));
    // the rows, kept as 32-bit offsets and 16-bit ids for the pair pass, where
    // they hold at most kRowCopyItems items on average (longer rows make more
    // pairs than the tensor cores' pass costs) and there are items outside the
    // tensor cores' block, which that pass never reads the rows for
    RowCopy rows{};
    if (ctx->n > 0 && ctx->m > kRowPairsTop) {
        uint64_t cap = row_copy_cap(ctx->n);
        if (nnz >= 0) cap = (uint64_t)nnz <= cap ? (uint64_t)nnz : 0;  // host input: known, so no more than that
        if (cap > 0) {
            int rc = fim_reserve(ctx, ctx->row_ptr, sizeof(uint32_t) * (size_t)(ctx->n + 1));
            if (rc == FIM_OK) rc = fim_reserve(ctx, ctx->row_idx, sizeof(unsigned short) * (size_t)cap);
            if (rc == FIM_OK) {
                rows.ptr = ctx->row_ptr.as<uint32_t>();
                rows.idx = ctx->row_idx.as<unsigned short>();
                rows.cap = cap;
            } else if (rc == FIM_E_NOMEM) {
                drop_rows(ctx);  // without them the pair pass takes the columns
            } else {
                return rc;
            }
        }
    }
    ctx->row_cap = rows.cap;
    if (nblk <= 0 || ctx->m <= 0) return FIM_OK;
    // device input (nnz < 0): the kernel reads indptr[n] itself
    // Host input: the indices go up in chunks of row blocks on side streams,
    // and each chunk's blocks are built as soon as its copy has landed, so the
    // upload overlaps the construction.  A chunk needs the elements
    // [indptr[t0], indptr[t1]) of its transactions; an indptr that is not
    // monotone there is flagged by the kernel, which then reads nothing.
    int chunks = h_indices ? ctx->upload_chunks : 1;
    if (chunks > nblk) chunks = (int)nblk;
    if (chunks < 1) chunks = 1;
    const int nstreams = h_indices ? ctx->upload_streams : 0;
    for (int s = 0; s < nstreams; s++) {
        if (!ctx->up_stream[s]) FIM_CUDA_TRY(cudaStreamCreateWithFlags(&ctx->up_stream[s], cudaStreamNonBlocking));
        // the copies overwrite the staging buffer: after all earlier work on the ctx stream
        FIM_CUDA_TRY(cudaStreamWaitEvent(ctx->up_stream[s], ctx->ev[0], 0));
    }
    for (int c = 0; c < chunks && h_indices; c++)
        if (!ctx->up_ev[c]) FIM_CUDA_TRY(cudaEventCreateWithFlags(&ctx->up_ev[c], cudaEventDisableTiming));
    const int64_t per = ceil_div64(nblk, chunks);
    const int64_t tpb = (int64_t)WB * 32;  // transactions per row block
    for (int c = 0; c < chunks; c++) {
        const int64_t b0 = (int64_t)c * per, b1 = min64(nblk, b0 + per);
        if (b0 >= b1) break;
        if (h_indices) {
            const int64_t t0 = min64(ctx->n, b0 * tpb), t1 = min64(ctx->n, b1 * tpb);
            int64_t lo = csr_off(h_indptr, cmp, t0), hi = csr_off(h_indptr, cmp, t1);
            lo = lo < 0 ? 0 : (lo > nnz ? nnz : lo);
            hi = hi < lo ? lo : (hi > nnz ? nnz : hi);
            if (hi > lo) {
                cudaStream_t cs = ctx->up_stream[c % nstreams];
                FIM_CUDA_TRY(cudaMemcpyAsync(static_cast<char *>(const_cast<void *>(d_indices)) + ib_bytes * (size_t)lo,
                                             static_cast<const char *>(h_indices) + ib_bytes * (size_t)lo,
                                             ib_bytes * (size_t)(hi - lo), cudaMemcpyHostToDevice, cs));
                FIM_CUDA_TRY(cudaEventRecord(ctx->up_ev[c], cs));
                FIM_CUDA_TRY(cudaStreamWaitEvent(st, ctx->up_ev[c], 0));
            }
        }
        dim3 grid((unsigned)(b1 - b0), (unsigned)niblk);
        ctx->launches++;
        kern<<<grid, T, smem, st>>>(d_indptr, d_indices, ctx->n, ctx->m, nnz, ctx->nwp, ib, ms, b0,
                                                ctx->bm.as<uint32_t>(), ctx->item_sup.as<uint32_t>(), flags, rows);
        FIM_CUDA_TRY(cudaGetLastError());
    }
    return FIM_OK;
}

int launch_rank_items(fim_ctx *ctx, uint32_t thr, MineCounters *d_ctr) {
    if (ctx->m == 0) return FIM_OK;
    const int threads = 256;
    const int blocks = (int)ceil_div64((int64_t)ctx->m * 32, threads);
    ctx->launches++;
    rank_items_kernel<<<blocks, threads, 0, ctx->stream>>>(
        ctx->item_sup.as<uint32_t>(), ctx->m, thr, ctx->perm.as<int32_t>(),
        ctx->rank.as<int32_t>(), d_ctr);
    FIM_CUDA_TRY(cudaGetLastError());
    return FIM_OK;
}

int launch_emit_singletons(fim_ctx *ctx, MineCounters *d_ctr) {
    const int threads = 256;
    const int blocks = (int)ceil_div64(ctx->m > 0 ? ctx->m : 1, threads);
    ctx->launches++;
    emit_singletons_kernel<<<blocks, threads, 0, ctx->stream>>>(
        ctx->item_sup.as<uint32_t>(), ctx->perm.as<int32_t>(), d_ctr,
        ctx->rec_off.as<unsigned long long>(), ctx->rec_len.as<uint32_t>(),
        ctx->rec_sup.as<uint32_t>(), ctx->rec_items.as<uint32_t>(), ctx->rec_cap,
        ctx->rec_items_cap);
    FIM_CUDA_TRY(cudaGetLastError());
    return FIM_OK;
}
