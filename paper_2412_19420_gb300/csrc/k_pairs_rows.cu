// k_pairs_rows.cu -- pair supports from the rows (Eq. 2), for short rows.
//
// S(I_a n I_b) can be summed over the matrix's columns (A^T A, k_pairs_tc.cu)
// or over its rows: a row of L frequent items adds 1 to L (L - 1) / 2 pair
// counts.  The contraction costs n m'^2 / 2 multiply-adds whatever the matrix
// holds; on basket data with thousands of items, where a row holds about ten,
// the rows hold five orders of magnitude fewer pairs: 6.6e8 of them against
// 9.2e13 on 10^7 x 5,000.
//
// pairs_rows_kernel: a warp takes 32 rows, reads their ids 32 at a time
// (coalesced), maps them to internal ids through a table in shared memory and
// packs the frequent ones, row after row, in its slice of shared memory.  Then
// each lane takes packed elements: element p of a row of L pairs with
// (p + d) mod L for d = 1 .. (L - 1) / 2 (and, L even, the first half of the
// row with d = L / 2), which meets every pair once with equal work for a row's
// elements.  Each pair is one reduction (RED) at pair_cnt[a][b].  The kernel is
// bound by those: an SM issues one lane of a scattered RED per cycle and the
// L2 takes 220 G/s of them over a 73 MB table (measured).
//
// The pairs among the kTop most frequent items are the hottest addresses and a
// dense block: they go to the tensor cores, on the side stream, and are skipped
// here.
//
// Pair pass, ms (tensor cores alone -> rows and the top block): 10^7 x 5,000
// 92.2 -> 4.3, 10^6 x 1,000 0.64 -> 0.3.
//
// The rows must name an item once (the supports' sum is compared with the
// number of ids); other matrices take the tensor-core pass.
#include <algorithm>

#include "fim_common.cuh"

namespace {

constexpr int PR_T = 256;               // threads per CTA
constexpr int PR_W = PR_T / 32;
constexpr int PR_CAP = kRowLong;        // packed elements a warp holds at a time
constexpr int kTop = kRowPairsTop;      // most frequent items: the tensor cores' block

// Rows [r0, r0 + 32) of warp tiles, grid-stride.
__global__ void __launch_bounds__(PR_T)
pairs_rows_kernel(const uint32_t *__restrict__ ptr, const unsigned short *__restrict__ idx, int64_t n,
                  const int32_t *__restrict__ rank, int m, int mf, int a0, int *__restrict__ pair_cnt) {
    extern __shared__ __align__(16) unsigned short pr_smem[];
    unsigned short *const table = pr_smem;                       // [m] internal id, 0xFFFF: infrequent
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned short *const el = pr_smem + ((m + 7) & ~7) + warp * 2 * PR_CAP;  // packed internal ids ...
    unsigned short *const own = el + PR_CAP;                                  // ... and the row of each
    for (int i = threadIdx.x; i < m; i += PR_T) table[i] = (unsigned short)rank[i];  // -1 -> 0xFFFF
    __syncthreads();
    const uint32_t lt = (1u << lane) - 1u;
    const int64_t tiles = (n + 31) / 32;
    for (int64_t t = (int64_t)blockIdx.x * PR_W + warp; t < tiles; t += (int64_t)gridDim.x * PR_W) {
        const int64_t r0 = t * 32;
        const int nr = (int)min64(32, n - r0);
        const uint32_t beg = ptr[r0 + (lane < nr ? lane : nr)];
        const uint32_t last = ptr[r0 + nr];
        int done = 0;  // rows of the tile already paired
        while (done < nr) {
            // as many whole rows as surely fit the buffer (a longer row is
            // paired from the id array itself, below)
            const uint32_t b0 = __shfl_sync(0xffffffffu, beg, done);
            uint32_t nx = __shfl_down_sync(0xffffffffu, beg, 1);
            if (lane >= nr - 1) nx = last;
            const uint32_t fits = __ballot_sync(0xffffffffu, lane >= done && lane < nr && nx - b0 <= (uint32_t)PR_CAP);
            const int end = fits ? 32 - __clz(fits) : done;  // rows [done, end) fit (the row ends ascend)
            if (end == done) {
                // one row of more than PR_CAP ids: its pairs, lane-strided
                const uint32_t e0 = b0, e1 = __shfl_sync(0xffffffffu, nx, done);
                for (uint32_t i = e0; i < e1; i++) {
                    const uint32_t x = table[idx[i]];
                    if (x == 0xFFFFu) continue;
                    for (uint32_t j = i + 1 + lane; j < e1; j += 32) {
                        const uint32_t y = table[idx[j]];
                        if (y == 0xFFFFu) continue;
                        const uint32_t a = min(x, y), b = max(x, y);
                        if ((int)a < a0) atomicAdd(pair_cnt + (int64_t)a * mf + b, 1);
                    }
                }
                done++;
                continue;
            }
            // pack the frequent items of rows [done, end); lane r learns where
            // row r's elements begin
            const uint32_t b1 = end < nr ? __shfl_sync(0xffffffffu, beg, end) : last;
            uint32_t k = 0, start = 0;
            for (uint32_t e0 = b0; e0 < b1; e0 += 32) {
                const uint32_t e = e0 + lane;
                uint32_t x = 0xFFFFu;
                if (e < b1) x = table[idx[e]];
                // the row of element e: the last one that begins at or before it
                int r = done;
#pragma unroll
                for (int st = 16; st > 0; st >>= 1) {
                    const uint32_t c = __shfl_sync(0xffffffffu, beg, min(r + st, 31));
                    if (r + st < end && c <= e) r += st;
                }
                const bool f = x != 0xFFFFu;
                const uint32_t bal = __ballot_sync(0xffffffffu, f);
                if (f) {
                    const uint32_t at = k + __popc(bal & lt);
                    el[at] = (unsigned short)x;
                    own[at] = (unsigned short)r;
                }
                // lane r's row begins after the packed elements of earlier ids
                if (beg >= e0 && beg < e0 + 32) start = k + __popc(bal & ((1u << (beg - e0)) - 1u));
                k += __popc(bal);
            }
            if (beg >= b1) start = k;  // empty rows at the end (and rows past the last)
            uint32_t stop = __shfl_down_sync(0xffffffffu, start, 1);
            if (lane >= end - 1) stop = k;
            __syncwarp();
            for (uint32_t e0 = 0; e0 < k; e0 += 32) {
                const uint32_t e = e0 + lane;
                const int r = e < k ? own[e] : 0;
                const uint32_t s = __shfl_sync(0xffffffffu, start, r), L = __shfl_sync(0xffffffffu, stop, r) - s;
                if (e < k) {
                    const uint32_t x = el[e], p = e - s;
                    const uint32_t nd = (L & 1u) ? L >> 1 : (L >> 1) - (p < (L >> 1) ? 0u : 1u);
                    for (uint32_t d = 1, q = p; d <= nd; d++) {
                        q = q + 1 == L ? 0 : q + 1;
                        const uint32_t y = el[s + q];
                        const uint32_t a = min(x, y), b = max(x, y);
                        if ((int)a < a0) atomicAdd(pair_cnt + (int64_t)a * mf + b, 1);
                    }
                }
            }
            __syncwarp();
            done = end;
        }
    }
}

// Counts that the top block may run beside (2 million rows of ten items, block
// beside the rows against block first: 4 MB 591 against 693 us, 16 MB 614 and
// 695, 25 MB 750 and 676, 36 MB 622 and 633, 49 MB 729 and 635).
constexpr size_t kBesideBytes = 16u << 20;
constexpr double kStageUs = 0.59;       // a 128-transaction stage of one tensor-core tile

// The row pass: its REDs, or one warp's where a few rows hold most of the pairs.
// A RED costs the chip 4.5 ps while the counts fit L2 (100 MB), then more:
// 9.6 ps at 196 MB, 24 at 400 MB, 35 at 1 GB (2 million rows of ten items over
// 7,001 to 16,001).  A warp counts 600 to 700 pairs a us of the rows it packs
// and half as many of longer ones: one row of 1,024 ids among 100,000 short
// ones takes 0.8 ms, one of 1,500 3.5 and one of 5,000 36, where the tensor
// cores take 1.35 ms whatever the rows are.
double rows_us(const fim_ctx *ctx) {
    const double mb = 4e-6 * (double)ctx->mfreq * (double)ctx->mfreq;
    const double ps = 4.5 + std::min(30.0, 0.065 * std::max(0.0, mb - 100.0));
    return std::max((double)ctx->row_pairs * ps * 1e-6, (double)ctx->tile_pairs / 600.0) + 15.0;
}

}  // namespace

// The row pass pays where it takes less than the tensor cores' tiles outside
// the top block (0.59 us per 128-transaction stage and SM,
// measured on 10^6 x 1,000 and 10^7 x 5,000).
bool pairs_rows_pays(const fim_ctx *ctx) {
    const int mf = ctx->mfreq;
    // an item repeated in a row would be counted twice: the supports (set
    // semantics) then sum to less than the ids
    if (!ctx->rows_kept || ctx->host_ctr.sup_sum != (unsigned long long)ctx->row_nnz || mf <= kTop || ctx->pairs_split > 0 || ctx->pairs_kdrain > 0) return false;
    if (ctx->pairs_rows >= 0) return ctx->pairs_rows != 0;
    const int nta = (mf + 127) / 128, ntb = (mf + 255) / 256;
    double tiles = 0;
    for (int ta = 0; ta < nta; ta++) tiles += ntb - (ta >> 1);
    const double stages = (double)((ctx->nw + 3) / 4);
    const double tc_us = (tiles - 2.0) * stages / ctx->num_sms * kStageUs;
    return rows_us(ctx) < tc_us;
}

int launch_pairs_rows(fim_ctx *ctx) {
    const int mf = ctx->mfreq, a0 = mf - kTop;
    cudaStream_t st = ctx->stream;
    FIM_TRY(fim_aux_stream(ctx));
    for (auto &e : ctx->pair_ev)
        if (!e) FIM_CUDA_TRY(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    FIM_CUDA_TRY(cudaMemsetAsync(ctx->pair_cnt.p, 0, sizeof(int) * (size_t)mf * mf, st));
    FIM_CUDA_TRY(cudaEventRecord(ctx->pair_ev[0], st));
    FIM_CUDA_TRY(cudaStreamWaitEvent(ctx->aux_stream, ctx->pair_ev[0], 0));
    // A tensor-core CTA fills an SM's shared memory, so on all SMs the top
    // block's two tiles hold the row pass back, which fewer SMs keep bound by its
    // REDs.  So the block gets half as many SMs again as would let it end with
    // the rows (it runs slower beside them): 10^6 x 1,000 0.355 -> 0.28 to
    // 0.32 ms for both (1x: 0.308, 2x: 0.328), 333,333 x 701 0.148 -> 0.113.  Where the
    // counts are a large part of L2 the block's reads evict them, and it goes
    // first on all SMs: 10^7 x 5,000 (73 MB) 4.33 ms, beside the rows 4.95.
    const bool beside = sizeof(int) * (size_t)mf * mf <= kBesideBytes;
    const double block_us = 2.0 * (double)((ctx->nw + 3) / 4) * kStageUs;
    int tc = ctx->num_sms;
    if (beside) tc = (int)std::min(1.5 * block_us / rows_us(ctx) + 1.0, ctx->num_sms / 2.0);
    if (tc < 1) tc = 1;
    FIM_TRY(launch_pairs_tc(ctx, a0, false, ctx->aux_stream, tc));
    FIM_CUDA_TRY(cudaEventRecord(ctx->pair_ev[1], ctx->aux_stream));
    const size_t smem = sizeof(unsigned short) * ((((size_t)ctx->m + 7) & ~(size_t)7) + PR_W * 2 * PR_CAP);
    FIM_CUDA_TRY(fim_allow_smem(pairs_rows_kernel, sizeof(unsigned short) * (((FIM_MAX_ITEMS + 7) & ~7) + PR_W * 2 * PR_CAP)));
    int64_t grid = ceil_div64(ceil_div64(ctx->n, 32), PR_W);
    // beside the block, resident CTAs only: a grid-stride share that waited for
    // an SM would end late
    int64_t room = (int64_t)ctx->num_sms * 8;
    if (beside) room = (int64_t)std::max(1, ctx->num_sms - tc) * std::min(8, (int)(227 * 1024 / (smem + 1024)));
    if (grid > room) grid = room;
    ctx->launches++;
    pairs_rows_kernel<<<(unsigned)grid, PR_T, smem, st>>>(ctx->row_ptr.as<uint32_t>(),
                                                          ctx->row_idx.as<unsigned short>(), ctx->n,
                                                          ctx->rank.as<int32_t>(), ctx->m, mf, a0,
                                                          ctx->pair_cnt.as<int>());
    FIM_CUDA_TRY(cudaGetLastError());
    FIM_CUDA_TRY(cudaStreamWaitEvent(st, ctx->pair_ev[1], 0));
    return FIM_OK;
}
