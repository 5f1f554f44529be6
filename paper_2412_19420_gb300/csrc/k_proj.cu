// k_proj.cu -- prefix extension on projected columns, one warp per worker.
//
// The search is dfs_kernel's (Section III: the column AND "in sequence",
// Eq. 3's threshold pruning every infrequent extension), but a root item a's
// subtree only ever looks at the S(a) transactions that hold a.  So before
// the search those transactions are projected out once per item:
//   T(a)    the rows of a's bit column, listed (tid_list_kernel);
//   C(a)    the items b > a whose pair {a, b} is frequent, ascending;
//   M_a     |C(a)| bit columns of W_a = ceil(S(a) / 128) * 4 words: bit i of
//           column b says whether the i-th transaction of T(a) holds b
//           (proj_gather_kernel).
// Every class {a, b, ...} below a is then counted on W_a words instead of
// ceil(n / 32): S(a) is at most a few percent of n on basket data.  A class
// pass that took a 256-thread CTA 25 us on whole columns is one warp's work on
// a column of one or a few 128-word chunks, with no block barrier at all.
// Databases whose whole matrix is small skip the projection: the workers then
// run on the bit columns themselves (`direct`).  Long columns of dense items, or
// with few sets, take the CTA workers of k_dfs.cu instead (projection_pays in
// fim_api.cu).
// The first level, S({a, b, c}), is one flat pass over all items
// (proj_triple_kernel); its frequent triples are the search's roots.
//
// dfs_proj_kernel: every warp is a depth-first worker.  It takes roots
// (triples; pairs when `direct`, in a split mine or when the triple table
// would be too large) from a ticket counter and, once those are gone, prefix
// classes that busy workers hand to the device queue.  A worker's stack and
// sibling lists sit in its slice of shared memory and spill to global memory.
// Every wait is bounded (FIM_E_TIMEOUT), and no worker waits for one that has
// not started.  A search deeper than a worker's stack reports FIM_E_STACK and
// is mined again by the CTA workers of k_dfs.cu, which also serve traces and
// the no-split option.  With FIM_LEARNED or FIM_DIFFSET_RULE a worker asks the
// network, or the size rule, for each class's representation (a build of the
// kernel of its own: the choice costs registers).
//
// Prefix extension, ms (one GB300; CTA workers -> this file, projection and
// triple pass included): 100,000 x 2,000 planted 47.3 -> 5.6 (14 bytes of
// every column in 15 are gone, and 4.2 million sets come from 24 warps an SM
// instead of 4 CTAs); 10^7 x 5,000 49 (twice, when its stack had to grow) ->
// 4.6; 10^6 x 1,000 0.97 -> 0.37; 50,001 x 60 dense 0.73 -> 0.25; 20,000 x 800
// planted with the network 4.1 -> 1.3.  What bounds
// it now: each class's chain of dependent steps (12 cycles from one of a
// worker's instructions to its next, 0.48 of the issue slots used on 100,000 x
// 2,000, ncu), and for the triple pass popc.
#include "fim_common.cuh"

namespace {

// Six warps a CTA, four CTAs an SM: 24 workers at 80 registers.  (32 workers at
// 64 registers spill and crowd the queue: 100,000 x 2,000 6.2 ms against 5.5.)
constexpr int PW = 6;            // warps (workers) per CTA
constexpr int PLV = 48;          // levels a worker tracks
constexpr int PFR = 256;         // sibling entries in shared memory per worker
constexpr int PST = 832;         // stack words in shared memory per worker
// Classes a worker hands over at a time, from its shallowest levels: handing
// over only the class at hand left most workers waiting (utilisation 0.19).
constexpr int PGIVE = 8;

template <bool REP>
struct __align__(16) PWork {
    uint32_t stack[PST];         // stored prefixes, bottom up
    uint32_t frames[PFR];        // sibling lists, bottom up
    uint32_t path[PLV + FIM_TASK_MAXR];      // the prefix, packed (column << 16 | internal id)
    int nF[PLV], cur[PLV];       // siblings of a level, next one to expand
    int fpos[PLV], spos[PLV];    // where its list / stored prefix lies (< 0: global)
    int ftopS[PLV], ftopG[PLV];  // first free list entry above it, shared / global
    int stopS[PLV], stopG[PLV];  // first free stack word above it
    unsigned long long rec_next, rec_end, it_next, it_end;  // reserved output slots
    unsigned long long n_sup, n_words, n_bytes, n_classes, n_diff, emitted, emitted_items;
    int max_len;
    // representation choice (network, diffset rule): supports of the list
    // entries and of the levels' classes, the network's input and output
    uint32_t fsup[REP ? PFR : 1], supY[REP ? PLV : 1];
    float feat[REP ? FIM_MLP_FEATURES : 1], out[2];
};

__device__ __forceinline__ void perr(const DfsParams &p, int code) { atomicCAS(&p.ctr->err, 0, code); }

// k, W and S of every item with at least two candidates: one warp per item.
__global__ void __launch_bounds__(256)
proj_count_kernel(const uint32_t *__restrict__ pairbits, int mf, int mpw, const int32_t *__restrict__ perm,
                  const uint32_t *__restrict__ sup, ProjItem *__restrict__ items) {
    const int a = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (a >= mf) return;
    uint32_t k = 0;
    for (int w = lane; w < mpw; w += 32) k += __popc(pairbits[(int64_t)a * mpw + w]);
    k = warp_sum_u32(k);
    if (lane == 0) {
        const uint32_t s = sup[perm[a]];
        items[a].k = k >= 2 ? k : 0u;  // one frequent pair {a, b} has no third item to try
        items[a].s = s;
        items[a].W = (uint32_t)(((uint64_t)s + 127) / 128 * 4);
    }
}

// The triple pass's units of an item: TB x TC blocks of its candidate pairs.
constexpr int TB = 4, TC = 8;
__host__ __device__ __forceinline__ unsigned long long triple_units(uint32_t k) {
    return (unsigned long long)((k + TB - 1) / TB) * ((k + TC - 1) / TC);
}

// What an item adds to each of the plan's six totals: projected words, row
// list, candidates, gather tiles, triple supports, triple units.
constexpr int NP = 6;
__device__ __forceinline__ void proj_sizes(const ProjItem &it, unsigned long long v[NP]) {
    v[0] = (unsigned long long)it.k * it.W;
    v[1] = it.s;
    v[2] = it.k;
    v[3] = (it.W + 31) / 32;
    v[4] = (unsigned long long)it.k * it.k;
    v[5] = triple_units(it.k);
}
__device__ __forceinline__ void proj_offsets(ProjItem &it, const unsigned long long run[NP],
                                             unsigned long long *tile0, unsigned long long *trip0) {
    it.moff = run[0];
    it.loff = run[1];
    it.coff = (uint32_t)run[2];
    it.toff = run[4];
    it.cursor = 0;
    *tile0 = run[3];
    *trip0 = run[5];
}
__device__ __forceinline__ void proj_totals(ProjTotals *tot, const unsigned long long v[NP]) {
    tot->words = v[0];
    tot->rows = v[1];
    tot->cands = v[2];
    tot->tiles = v[3];
    tot->triples = v[4];
    tot->units = v[5];
}

// Offsets of everything the plan sizes, and the totals (one CTA).
__global__ void __launch_bounds__(1024)
proj_scan_kernel(ProjItem *__restrict__ items, int mf, unsigned long long *__restrict__ tile0,
                 unsigned long long *__restrict__ trip0, ProjTotals *__restrict__ tot) {
    __shared__ unsigned long long sc[NP][1024];
    const int seg = (mf + 1023) / 1024;
    const int b = threadIdx.x * seg, e = min(b + seg, mf);
    unsigned long long v[NP] = {}, own[NP];
    uint32_t wmax = 0;
    for (int i = b; i < e; i++) {
        const ProjItem it = items[i];
        if (!it.k) continue;
        unsigned long long x[NP];
        proj_sizes(it, x);
        for (int q = 0; q < NP; q++) v[q] += x[q];
        wmax = max(wmax, it.W);
    }
    for (int q = 0; q < NP; q++) sc[q][threadIdx.x] = own[q] = v[q];
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
        unsigned long long x[NP];
        for (int q = 0; q < NP; q++) x[q] = threadIdx.x >= (unsigned)o ? sc[q][threadIdx.x - o] : 0ull;
        __syncthreads();
        for (int q = 0; q < NP; q++) sc[q][threadIdx.x] += x[q];
        __syncthreads();
    }
    unsigned long long run[NP], all[NP];
    for (int q = 0; q < NP; q++) run[q] = sc[q][threadIdx.x] - own[q], all[q] = sc[q][1023];
    for (int i = b; i < e; i++) {
        ProjItem &it = items[i];
        proj_offsets(it, run, tile0 + i, trip0 + i);
        if (!it.k) continue;
        unsigned long long x[NP];
        proj_sizes(it, x);
        for (int q = 0; q < NP; q++) run[q] += x[q];
    }
    if (wmax) atomicMax(&tot->wmax, wmax);
    if (threadIdx.x == 1023) {
        proj_totals(tot, all);
        tile0[mf] = all[3];
        trip0[mf] = all[5];
    }
}

// Everything between the pair counts and the search of a mine with at most
// SP_MAX frequent items, in one CTA: the threshold on the pairs (Eq. 3), the
// pair bitset, the pair records, the root classes with at least one candidate,
// most candidates first, and the projection's plan.  On such a mine each of
// these steps is a few microseconds of launch and latency, so one launch takes
// the place of nine.
constexpr int SP_MAX = 256, SP_T = 1024;
__global__ void __launch_bounds__(SP_T)
proj_small_plan_kernel(const int *__restrict__ pair_cnt, int m, uint32_t thr, const int32_t *__restrict__ perm,
                       const uint32_t *__restrict__ sup, uint32_t *__restrict__ pairbits, MineCounters *ctr,
                       uint32_t *epoch, unsigned long long *__restrict__ rec_off, uint32_t *__restrict__ rec_len,
                       uint32_t *__restrict__ rec_sup, uint32_t *__restrict__ rec_items, unsigned long long rec_cap,
                       unsigned long long items_cap, uint32_t *__restrict__ root_a, uint32_t *__restrict__ root_b,
                       uint32_t *__restrict__ root_sup, uint32_t *__restrict__ root_order,
                       ProjItem *__restrict__ items, unsigned long long *__restrict__ tile0,
                       unsigned long long *__restrict__ trip0, uint32_t *__restrict__ cands,
                       ProjTotals *__restrict__ tot, int triples, int ask) {
    constexpr int MW = SP_MAX / 32, NW = SP_T / 32, KB = SP_MAX;  // bucket = candidates, 0 .. SP_MAX - 1
    __shared__ uint32_t bits[SP_MAX][MW];
    __shared__ uint32_t rowpos[SP_MAX + 1];
    __shared__ uint32_t hist[KB];
    __shared__ ProjItem s_it[SP_MAX];
    __shared__ unsigned long long s_base[2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int mf = *(volatile const int *)&ctr->m_freq;  // <= m, the host's bound
    const int mpw = (mf + 31) / 32;
    for (int i = threadIdx.x; i < KB; i += SP_T) hist[i] = 0;
    if (ask && threadIdx.x == 0) tot->pair_sum = 0;
    if (ask) __syncthreads();
    unsigned long long pair_sum = 0;
    for (int a = warp; a < mf; a += NW) {
        uint32_t c = 0, sum = 0;
        int v[MW];
#pragma unroll
        for (int w = 0; w < MW; w++) {
            const int b = w * 32 + lane;
            v[w] = b > a && b < mf ? pair_cnt[(int64_t)a * mf + b] : 0;
        }
#pragma unroll
        for (int w = 0; w < MW; w++) {
            const int b = w * 32 + lane;
            const uint32_t bal = __ballot_sync(0xffffffffu, b > a && b < mf && (uint32_t)v[w] >= thr);
            if (lane == 0) {
                bits[a][w] = bal;
                if (w < mpw) pairbits[a * mpw + w] = bal;
            }
            c += __popc(bal);
            if (ask && ((bal >> lane) & 1u)) sum += (uint32_t)v[w];
        }
        if (c >= 2) pair_sum += sum;
        if (lane == 0) {
            const uint32_t S = sup[perm[a]];
            rowpos[a] = c;
            s_it[a].k = c >= 2 ? c : 0u;
            s_it[a].s = S;
            s_it[a].W = (uint32_t)(((uint64_t)S + 127) / 128 * 4);
        }
    }
    if (ask && pair_sum) atomicAdd(&tot->pair_sum, pair_sum);
    __syncthreads();
    if (warp == 0) {  // prefix sums over the rows, four to a lane
        constexpr int PER = SP_MAX / 32;
        uint32_t n = 0, wmax = 0;
        unsigned long long v[NP] = {}, x[NP];
        for (int i = 0; i < PER; i++) {
            const int a = lane * PER + i;
            if (a >= mf) break;
            n += rowpos[a];
            if (!s_it[a].k) continue;
            proj_sizes(s_it[a], x);
#pragma unroll
            for (int q = 0; q < NP; q++) v[q] += x[q];
            wmax = max(wmax, s_it[a].W);
        }
        uint32_t xn = n;
        unsigned long long run[NP];
#pragma unroll
        for (int q = 0; q < NP; q++) run[q] = v[q];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t yn = __shfl_up_sync(0xffffffffu, xn, o);
            if (lane >= o) xn += yn;
#pragma unroll
            for (int q = 0; q < NP; q++) {
                const unsigned long long y = __shfl_up_sync(0xffffffffu, run[q], o);
                if (lane >= o) run[q] += y;
            }
        }
        for (int o = 16; o > 0; o >>= 1) wmax = max(wmax, __shfl_xor_sync(0xffffffffu, wmax, o));
        if (lane == 31) {  // the totals
            proj_totals(tot, run);
            tot->wmax = wmax;
            for (int a = mf; a <= m; a++) {  // (the later kernels search m entries)
                tile0[a] = run[3];
                trip0[a] = run[5];
            }
        }
        uint32_t rn = xn - n;
#pragma unroll
        for (int q = 0; q < NP; q++) run[q] -= v[q];
        for (int i = 0; i < PER; i++) {
            const int a = lane * PER + i;
            if (a >= mf) break;
            const uint32_t c = rowpos[a];
            rowpos[a] = rn;
            rn += c;
            proj_offsets(s_it[a], run, tile0 + a, trip0 + a);
            if (!s_it[a].k) continue;
            proj_sizes(s_it[a], x);
#pragma unroll
            for (int q = 0; q < NP; q++) run[q] += x[q];
        }
        if (lane == 31) {
            rowpos[mf] = xn;
            s_base[0] = ctr->n_records;
            s_base[1] = ctr->n_rec_items;
            ctr->n_records = s_base[0] + xn;
            ctr->n_rec_items = s_base[1] + 2ull * xn;
            if (s_base[0] + xn > rec_cap) atomicOr(&ctr->overflow, 1);
            else if (s_base[1] + 2ull * xn > items_cap) atomicOr(&ctr->overflow, 2);
            const uint32_t e = *epoch + 1u;
            *epoch = e ? e : 1u;  // 0 marks a slot that was never published
        }
    }
    __syncthreads();
    for (int a = threadIdx.x; a < m; a += SP_T) {
        if (a >= mf) s_it[a].k = 0;
        items[a] = s_it[a];
    }
    // pair records and root classes, in (a, b) order; roots counted by their
    // number of candidates
    for (int pass = 0; pass < 2; pass++) {
        for (int a = warp; a < mf; a += NW) {
            uint32_t pos = rowpos[a];
            for (int w = (a + 1) >> 5; w < mpw; w++) {
                const uint32_t bal = bits[a][w];
                if ((bal >> lane) & 1u) {
                    const int b = w * 32 + lane;
                    const uint32_t at = pos + __popc(bal & ((1u << lane) - 1u));
                    int k = 0;
#pragma unroll
                    for (int x = 0; x < MW; x++) {
                        uint32_t m = bits[a][x] & bits[b][x];
                        if (x < w) m = 0;
                        else if (x == w) m &= 0xFFFFFFFEu << lane;
                        k += __popc(m);
                    }
                    if (pass == 0) {
                        const uint32_t S = (uint32_t)pair_cnt[(int64_t)a * mf + b];
                        const unsigned long long r = s_base[0] + at, it = s_base[1] + 2ull * at;
                        if (r < rec_cap && it + 2 <= items_cap) {
                            rec_off[r] = it;
                            rec_len[r] = 2;
                            rec_sup[r] = S;
                            rec_items[it] = (uint32_t)a;
                            rec_items[it + 1] = (uint32_t)b;
                        }
                        root_a[at] = (uint32_t)a;
                        root_b[at] = (uint32_t)b;
                        root_sup[at] = S;
                        if (s_it[a].k) cands[s_it[a].coff + at - rowpos[a]] = (uint32_t)b;
                        atomicAdd(&hist[k], 1u);
                    } else if (k > 0) {
                        root_order[atomicAdd(&hist[k], 1u)] = at;
                    }
                }
                pos += __popc(bal);
            }
        }
        __syncthreads();
        if (pass == 0 && warp == 0) {  // bucket starts: most candidates first, none dropped
            constexpr int PER = KB / 32;
            uint32_t c[PER], n = 0;
            for (int i = 0; i < PER; i++) {
                const int q = KB - 1 - (lane * PER + i);
                c[i] = q > 0 ? hist[q] : 0u;
                n += c[i];
            }
            uint32_t x = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            uint32_t run = x - n;
            for (int i = 0; i < PER; i++) {
                const int q = KB - 1 - (lane * PER + i);
                if (q > 0) hist[q] = run;
                run += c[i];
            }
            if (lane == 31) {  // (the triple pass brings its own roots)
                ctr->n_roots = x;
                ctr->pending = triples ? 0ll : (long long)x;
            }
        }
        __syncthreads();
    }
}

// C(a): one warp per item lists its pair bits, ascending.
__global__ void __launch_bounds__(256)
proj_cands_kernel(const uint32_t *__restrict__ pairbits, int mf, int mpw, const ProjItem *__restrict__ items,
                  uint32_t *__restrict__ cands, MineCounters *ctr, int triples) {
    if (triples && blockIdx.x == 0 && threadIdx.x == 0) ctr->pending = 0;  // the triple pass brings its own roots
    const int a = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (a >= mf || !items[a].k) return;
    uint32_t at = items[a].coff;
    for (int w0 = 0; w0 < mpw; w0 += 32) {
        const int w = w0 + lane;
        uint32_t bits = w < mpw ? pairbits[(int64_t)a * mpw + w] : 0u;
        const uint32_t c = __popc(bits);
        uint32_t x = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        uint32_t pos = at + x - c;
        while (bits) {
            cands[pos++] = (uint32_t)(w * 32 + __ffs(bits) - 1);
            bits &= bits - 1;
        }
        at += __shfl_sync(0xffffffffu, x, 31);
    }
}

// T(a), in any order: a CTA takes one 8,192-word segment of one column, 32
// words a thread in registers; one block scan and one global atomic place its
// rows.  (The order only names the bits of M_a; every column of M_a uses the
// same one.)
// NV 16-byte loads a thread: eight on long columns, one where the matrix is
// small and its columns dense (a thread then lists at most 128 rows, and the
// list is spread over eight times the threads).
constexpr int TL_T = 256;
template <int NV>
__global__ void __launch_bounds__(TL_T)
tid_list_kernel(const uint32_t *__restrict__ bm, const int32_t *__restrict__ perm, int64_t nwp,
                ProjItem *__restrict__ items, uint32_t *__restrict__ list) {
    __shared__ uint32_t wsum[TL_T / 32];
    __shared__ uint32_t base;
    const int a = blockIdx.y;
    ProjItem &it = items[a];
    if (!it.k) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t *col = bm + (int64_t)perm[a] * nwp;
    // a warp's NV * 128 words are contiguous: NV loads of 512 bytes
    const int64_t w0 = ((int64_t)blockIdx.x * (TL_T / 32) + warp) * (NV * 128) + lane * 4;
    uint4 v[NV];
    uint32_t c = 0;
#pragma unroll
    for (int i = 0; i < NV; i++) {
        const int64_t w = w0 + i * 128;
        v[i] = w < nwp ? ldg_u4(col + w) : make_uint4(0, 0, 0, 0);  // nwp % 128 == 0
        c += __popc(v[i].x) + __popc(v[i].y) + __popc(v[i].z) + __popc(v[i].w);
    }
    uint32_t x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t acc = 0;
        for (int w = 0; w < TL_T / 32; w++) {
            const uint32_t t = wsum[w];
            wsum[w] = acc;
            acc += t;
        }
        base = acc ? atomicAdd(&it.cursor, acc) : 0u;
    }
    __syncthreads();
    uint32_t *out = list + it.loff + base + wsum[warp] + x - c;
    const uint32_t r0 = (uint32_t)(w0 * 32);
#pragma unroll
    for (int i = 0; i < NV; i++) {
        const uint32_t w[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
#pragma unroll
        for (int q = 0; q < 4; q++) {
            uint32_t b = w[q];
            while (b) {
                *out++ = r0 + (uint32_t)(i * 4096 + q * 32 + __ffs(b) - 1);
                b &= b - 1;
            }
        }
    }
}

// M_a from the bit columns: a warp takes 1,024 rows of T(a) (32 words of every
// projected column) and, candidate by candidate, gathers the word of each of
// its rows, 32 loads in flight per lane; a ballot per 32 rows makes one output
// word.  Neighbouring rows of T(a) share sectors of the candidate's column
// (256 rows to a sector), so the gather's traffic is close to the columns'.
__global__ void __launch_bounds__(256)
proj_gather_kernel(const uint32_t *__restrict__ bm, const int32_t *__restrict__ perm, int64_t nwp, int mf,
                   const ProjItem *__restrict__ items, const unsigned long long *__restrict__ tile0,
                   const uint32_t *__restrict__ list, const uint32_t *__restrict__ cands,
                   uint32_t *__restrict__ mat, int csplit) {
    const int lane = threadIdx.x & 31;
    const unsigned long long nu = tile0[mf] * (unsigned)csplit;
    for (unsigned long long u = (unsigned long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); u < nu;
         u += (unsigned long long)gridDim.x * (blockDim.x >> 5)) {
    const unsigned long long t = u / (unsigned)csplit;
    const uint32_t part = (uint32_t)(u % (unsigned)csplit);
    int lo = 0, hi = mf;  // tile0[lo] <= t < tile0[hi]; the last such item is the tile's
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (tile0[mid] <= t) lo = mid; else hi = mid;
    }
    const ProjItem it = items[lo];
    const uint32_t w0 = (uint32_t)(t - tile0[lo]) * 32u;
    const int nq = (int)min(32u, it.W - w0);
    uint32_t pos[32];
#pragma unroll
    for (int q = 0; q < 32; q++) {
        const uint32_t i = (w0 + q) * 32u + lane;
        pos[q] = (q < nq && i < it.s) ? __ldg(list + it.loff + i) : 0xFFFFFFFFu;
    }
    for (uint32_t c = part; c < it.k; c += (uint32_t)csplit) {
        const uint32_t *col = bm + (int64_t)perm[cands[it.coff + c]] * nwp;
        uint32_t g[32];
#pragma unroll
        for (int q = 0; q < 32; q++)
            g[q] = (q < nq && pos[q] != 0xFFFFFFFFu) ? __ldg(col + (pos[q] >> 5)) : 0u;
        uint32_t mine = 0;
#pragma unroll
        for (int q = 0; q < 32; q++) {
            const uint32_t b = __ballot_sync(0xffffffffu, (g[q] >> (pos[q] & 31u)) & 1u);
            if (lane == q) mine = b;
        }
        if (lane < nq) mat[it.moff + (unsigned long long)c * it.W + w0 + lane] = mine;
    }
    }
}

// S({a, b, c}) for every a and b < c in C(a) with {b, c} frequent: the first
// level of the search as one flat pass, M_a's columns against each other (a
// bit-matrix product per item).  A warp takes a block of TB x TC pairs: lanes
// over the columns' words, 12 columns loaded for 32 supports, one reduction
// each at the end.  Frequent triples become records and the search's roots; the
// counts stay in triple[] (row b of item a: k entries), from which a root reads
// its candidates.  As tasks of single workers these classes were few and wide:
// 1,770 of them, up to 58 candidates each, took most of a 50,001 x 60 mine.
// (Two CTAs an SM: left to itself the compiler may take 164 registers, one CTA,
// and half as long again.)
__global__ void __launch_bounds__(256, 2)
proj_triple_kernel(const ProjItem *__restrict__ items, int mf, const unsigned long long *__restrict__ trip0,
                   const uint32_t *__restrict__ cands, const uint32_t *__restrict__ mat,
                   const uint32_t *__restrict__ pairbits, const DbDesc *__restrict__ dbs, uint32_t thr,
                   uint32_t *__restrict__ triple,
                   unsigned long long *__restrict__ roots, MineCounters *ctr, unsigned long long *rec_off,
                   uint32_t *rec_len, uint32_t *rec_sup, uint32_t *rec_items, unsigned long long rec_cap,
                   unsigned long long items_cap) {
    const int lane = threadIdx.x & 31;
    const int mpw = (dbs->mfreq + 31) / 32;
    const unsigned long long nu = trip0[mf];
    unsigned long long n_sup = 0, n_words = 0, n_bytes = 0;
    bool any = false;
    for (unsigned long long u = (unsigned long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); u < nu;
         u += (unsigned long long)gridDim.x * (blockDim.x >> 5)) {
        int lo = 0, hi = mf;  // trip0[lo] <= u < trip0[hi]; the last such item is the unit's
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (trip0[mid] <= u) lo = mid; else hi = mid;
        }
        const ProjItem it = items[lo];
        const uint32_t r = (uint32_t)(u - trip0[lo]), nc = (it.k + TC - 1) / TC;
        const uint32_t b0 = r / nc * TB, c0 = r % nc * TC;
        if (c0 + TC - 1 <= b0) continue;  // no pair b < c in this block
        // lane = pair (b0 + lane / TC, c0 + lane % TC)
        const uint32_t bi = b0 + lane / TC, ci = c0 + lane % TC;
        const bool in = bi < ci && ci < it.k;
        const uint32_t ib = in ? cands[it.coff + bi] : 0u, ic = in ? cands[it.coff + ci] : 0u;
        const bool want = in && ((pairbits[(int64_t)ib * mpw + (ic >> 5)] >> (ic & 31)) & 1u);
        const uint32_t wanted = __ballot_sync(0xffffffffu, want);
        uint32_t mine = 0;
        if (wanted) {
            const uint32_t *col = mat + it.moff;
            uint32_t acc[TB * TC];
#pragma unroll
            for (int x = 0; x < TB * TC; x++) acc[x] = 0u;
            for (uint32_t w = lane * 4; w < it.W; w += 128) {
                uint4 vb[TB], vc[TC];
#pragma unroll
                for (int x = 0; x < TB; x++) vb[x] = ldg_u4(col + (int64_t)min(b0 + x, it.k - 1) * it.W + w);
#pragma unroll
                for (int x = 0; x < TC; x++) vc[x] = ldg_u4(col + (int64_t)min(c0 + x, it.k - 1) * it.W + w);
#pragma unroll
                for (int x = 0; x < TB * TC; x++) acc[x] += popc_and4(vb[x / TC], vc[x % TC]);
            }
#pragma unroll
            for (int x = 0; x < TB * TC; x++) {
                const uint32_t t = __reduce_add_sync(0xffffffffu, acc[x]);
                if (lane == x) mine = t;
            }
        }
        const bool f = want && mine >= thr;
        if (in) triple[it.toff + (unsigned long long)bi * it.k + ci] = f ? mine : 0u;
        const uint32_t bal = __ballot_sync(0xffffffffu, f), more = __ballot_sync(0xffffffffu, f && ci + 1 < it.k);
        const unsigned tot = __popc(bal);
        if (lane == 0) {
            n_sup += __popc(wanted);
            n_words += (unsigned long long)__popc(wanted) * it.W;
            n_bytes += wanted ? 4ull * it.W * (TB + TC) : 0ull;
        }
        if (!tot) continue;
        any = true;
        unsigned long long rb = 0, ib3 = 0, q = 0;
        if (lane == 0) {
            rb = atomicAdd(&ctr->n_records, (unsigned long long)tot);
            ib3 = atomicAdd(&ctr->n_rec_items, 3ull * tot);
            if (more) {
                // only the roots that fit are stored and searched, so only they
                // are pending (the others are beyond the records, whose overflow
                // repeats the mine)
                const unsigned long long n = (unsigned long long)__popc(more);
                q = atomicAdd(&ctr->n_triples, n);
                if (q < rec_cap)
                    atomicAdd((unsigned long long *)&ctr->pending, q + n <= rec_cap ? n : rec_cap - q);
            }
        }
        rb = __shfl_sync(0xffffffffu, rb, 0);
        ib3 = __shfl_sync(0xffffffffu, ib3, 0);
        q = __shfl_sync(0xffffffffu, q, 0);
        const uint32_t lt = (1u << lane) - 1u;
        if (f) {
            const unsigned pos = __popc(bal & lt);
            const unsigned long long rr = rb + pos, i3 = ib3 + 3ull * pos;
            if (rr < rec_cap && i3 + 3 <= items_cap) {
                rec_off[rr] = i3;
                rec_len[rr] = 3;
                rec_sup[rr] = mine;
                rec_items[i3] = (uint32_t)lo;
                rec_items[i3 + 1] = ib;
                rec_items[i3 + 2] = ic;
            } else {
                atomicOr(&ctr->overflow, rr < rec_cap ? 2 : 1);
            }
            if (ci + 1 < it.k) {
                const unsigned long long at = q + __popc(more & lt);
                if (at < rec_cap) roots[at] = (unsigned long long)lo << 32 | bi << 16 | ci;
            }
        }
    }
    if (lane == 0) {
        if (n_sup) {
            atomicAdd(&ctr->supports_dfs, n_sup);
            atomicAdd(&ctr->dfs_words, n_words);
            atomicAdd(&ctr->dfs_bytes, n_bytes);
            atomicAdd(&ctr->dfs_touched, n_bytes);
        }
        if (any) atomicMax(&ctr->max_len, 3);
    }
}

// Where a worker's lists and stored prefixes lie.
struct Space {
    uint32_t *gfr, *gst;     // this worker's global list / stack
    uint32_t *gfs;           // its list entries' supports (REP)
    int gfr_cap, gst_cap;
};

template <bool REP>
__device__ __forceinline__ uint32_t *frame_at(PWork<REP> &s, const Space &sp, int pos) {
    return pos >= 0 ? s.frames + pos : sp.gfr + ~pos;
}
template <bool REP>
__device__ __forceinline__ uint32_t *fsup_at(PWork<REP> &s, const Space &sp, int pos) {
    if (!REP) return nullptr;
    return pos >= 0 ? s.fsup + pos : sp.gfs + ~pos;
}
template <bool REP>
__device__ __forceinline__ uint32_t *stack_at(PWork<REP> &s, const Space &sp, int pos) {
    return pos >= 0 ? s.stack + pos : sp.gst + ~pos;
}
// Room for `need` entries above (topS, topG): a position, or INT_MIN.
__device__ __forceinline__ int place(int need, int topS, int capS, int topG, int capG) {
    if (topS + need <= capS) return topS;
    return (long long)topG + need <= capG ? ~topG : INT32_MIN;
}

// Lane 0: output slots for tot itemsets of nitems items.  A worker that has
// emitted much reserves ahead (an eighth of what it has emitted, at most 64
// sets), so that a returning global atomic is paid every few classes; slots
// left over at its end are holes, which the compactor leaves out.
template <bool REP>
__device__ __forceinline__ void take_slots(const DfsParams &p, PWork<REP> &s, unsigned tot, unsigned nitems,
                                           unsigned long long *rb, unsigned long long *ib) {
    if (s.rec_next + tot > s.rec_end) {
        for (unsigned long long r = s.rec_next; r < s.rec_end; r++)
            if (r < p.rec_cap) p.rec_len[r] = 0u;
        if (s.rec_end > s.rec_next) atomicAdd(&p.ctr->rec_holes, s.rec_end - s.rec_next);
        const unsigned long long ahead = s.emitted >> 3 < 64 ? s.emitted >> 3 : 64;
        const unsigned long long want = tot > ahead ? tot : ahead;
        s.rec_next = atomicAdd(&p.ctr->n_records, want);
        s.rec_end = s.rec_next + want;
    }
    if (s.it_next + nitems > s.it_end) {
        if (s.it_end > s.it_next) atomicAdd(&p.ctr->item_holes, s.it_end - s.it_next);
        const unsigned long long ahead = s.emitted_items >> 3 < 512 ? s.emitted_items >> 3 : 512;
        const unsigned long long want = nitems > ahead ? nitems : ahead;
        s.it_next = atomicAdd(&p.ctr->n_rec_items, want);
        s.it_end = s.it_next + want;
    }
    *rb = s.rec_next;
    *ib = s.it_next;
    s.rec_next += tot;
    s.it_next += nitems;
    s.emitted += tot;
    s.emitted_items += nitems;
}

// One class: prefix b_Y = src0 AND src1 (W words), candidates cand[0 .. k),
// packed (column << 16 | id).  Frequent ones are compacted in order into fout
// (which may be cand: a sweep reads its entries before any write reaches them)
// and emitted with the prefix s.path[0 .. plen).  2^lg lanes cover 128 words
// of the prefix at a time, so short columns count 32 >> lg candidates side by
// side; PG candidates per lane are loaded together.  Returns |F|.
// REP: diff counts through the diffset, S(X u e) - popc((src0 AND NOT src1) AND
// col(e)), with the parent supports psup (which also receives the children's).
template <int PG, bool REP>
__device__ __forceinline__ int proj_class_pass(const DfsParams &p, PWork<REP> &s, uint32_t thr, const uint32_t *src0,
                                               const uint32_t *src1, const uint32_t *__restrict__ cols,
                                               int64_t stride, int W, int lg, const uint32_t *cand, int k, int plen,
                                               uint32_t *store, uint32_t *fout, uint32_t *psup, bool diff) {
    const int lane = threadIdx.x & 31;
    const int NS = 32 >> lg, sub = lane >> lg;
    const int wl = (lane & ((1 << lg) - 1)) * 4, step = 4 << lg;
    int nF = 0;
    for (int g0 = 0; g0 < k; g0 += PG * NS) {
        const int gn = min(PG * NS, k - g0);
        const uint32_t my = lane < gn ? cand[g0 + lane] : 0u;
        const uint32_t ps = REP && diff && lane < gn ? psup[g0 + lane] : 0u;
        const int nu = (gn + NS - 1) >> (5 - lg);
        uint32_t ci[PG], acc[PG];
#pragma unroll
        for (int u = 0; u < PG; u++) {
            ci[u] = __shfl_sync(0xffffffffu, my, min(u * NS + sub, gn - 1)) >> 16;
            acc[u] = 0u;
        }
        for (int w0 = 0; w0 < W; w0 += step) {
            const int w = w0 + wl;
            if (w < W) {
                const uint4 a = *reinterpret_cast<const uint4 *>(src0 + w), b = *reinterpret_cast<const uint4 *>(src1 + w);
                uint4 y = and4(a, b);
                uint4 cv[PG];
#pragma unroll
                for (int u = 0; u < PG; u++)
                    if (u < nu) cv[u] = ldg_u4(cols + (int64_t)ci[u] * stride + w);
                if (g0 == 0 && store && sub == 0) *reinterpret_cast<uint4 *>(store + w) = y;
                if (REP && diff) y = make_uint4(a.x & ~b.x, a.y & ~b.y, a.z & ~b.z, a.w & ~b.w);
#pragma unroll
                for (int u = 0; u < PG; u++)
                    if (u < nu) acc[u] += popc_and4(y, cv[u]);
            }
        }
        uint32_t mine = 0;
        if (lg == 5) {
#pragma unroll
            for (int u = 0; u < PG; u++)
                if (u < nu) {
                    const uint32_t t = __reduce_add_sync(0xffffffffu, acc[u]);
                    if (lane == u) mine = t;
                }
        } else {
#pragma unroll
            for (int u = 0; u < PG; u++)
                if (u < nu) {
                    uint32_t t = acc[u];
                    for (int o = (1 << lg) >> 1; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                    // candidate u * NS + g sits in lane group g: to lane u * NS + g
                    t = __shfl_sync(0xffffffffu, t, (lane & (NS - 1)) << lg);
                    if (lane >> (5 - lg) == u) mine = t;
                }
        }
        if (REP && diff) mine = ps - mine;
        const bool f = lane < gn && mine >= thr;
        const uint32_t bal = __ballot_sync(0xffffffffu, f);
        const int tot = __popc(bal);
        if (tot) {
            const unsigned len = (unsigned)plen + 1u;
            unsigned long long rb = 0, ib = 0;
            if (lane == 0) take_slots(p, s, (unsigned)tot, (unsigned)tot * len, &rb, &ib);
            rb = __shfl_sync(0xffffffffu, rb, 0);
            ib = __shfl_sync(0xffffffffu, ib, 0);
            const bool fits = rb + tot <= p.rec_cap && ib + (unsigned long long)tot * len <= p.rec_items_cap;
            if (f) {
                const int pos = __popc(bal & ((1u << lane) - 1u));
                fout[nF + pos] = my;
                if (REP) psup[nF + pos] = mine;
                if (fits) {
                    const unsigned long long r = rb + pos;
                    p.rec_off[r] = ib + (unsigned long long)pos * len;
                    p.rec_len[r] = len;
                    p.rec_sup[r] = mine;
                }
            }
            __syncwarp();
            if (fits) {  // the sets' items are one contiguous run: a word per lane
                for (unsigned t = lane; t < (unsigned)tot * len; t += 32) {
                    const unsigned r = t / len, q = t - r * len;
                    p.rec_items[ib + t] = (q < (unsigned)plen ? s.path[q] : fout[nF + r]) & 0xFFFFu;
                }
            } else if (lane == 0) {
                atomicOr(&p.ctr->overflow, rb + tot <= p.rec_cap ? 2 : 1);
            }
            nF += tot;
        }
        __syncwarp();
    }
    return nF;
}

// Child candidates of sibling j of a list of nF: the later siblings whose pair
// with it is frequent, in order.  Returns their number; *cit = sibling j.
template <bool REP>
__device__ __forceinline__ int siblings(const DfsParams &p, int mpw, const uint32_t *fr, const uint32_t *fs, int j,
                                        int nF, uint32_t *out, uint32_t *outs, uint32_t *cit) {
    const int lane = threadIdx.x & 31;
    const uint32_t c = fr[j];
    const uint32_t *rb = p.pairbits + (int64_t)(c & 0xFFFFu) * mpw;
    int k = 0;
    for (int l0 = j + 1; l0 < nF; l0 += 32) {
        const int l = l0 + lane;
        const uint32_t d = l < nF ? fr[l] : 0u;
        const uint32_t id = d & 0xFFFFu;
        const bool f = l < nF && ((__ldg(rb + (id >> 5)) >> (id & 31)) & 1u);
        const uint32_t bal = __ballot_sync(0xffffffffu, f);
        if (f) {
            const int at = k + __popc(bal & ((1u << lane) - 1u));
            out[at] = d;
            if (REP) outs[at] = fs[l];
        }
        k += __popc(bal);
    }
    *cit = c;
    return k;
}

// Publish the class s.path[0 .. plen) + cit with candidates cand[0 .. k) as a
// queue slot.  False when the queue or the candidate pool is full.
template <bool REP>
__device__ __noinline__ bool give(const DfsParams &p, PWork<REP> &s, uint32_t epoch, int plen, uint32_t cit,
                                  uint32_t sup, const uint32_t *cand, int k) {
    const int lane = threadIdx.x & 31;
    unsigned long long off = 0, slot = ~0ull;
    __syncwarp();
    if (lane == 0) {
        off = atomicAdd(&p.ctr->w_pool, (unsigned long long)k);
        if (off + k <= p.cand_pool_cap) {
            atomicAdd((unsigned long long *)&p.ctr->pending, 1ull);
            slot = atomicAdd(&p.ctr->w_tail, 1ull);
            if (slot >= p.task_cap) {
                slot = ~0ull;
                atomicAdd((unsigned long long *)&p.ctr->pending, (unsigned long long)(-1ll));
            } else {
                atomicAdd(&p.ctr->pushed, 1ull);
            }
        }
    }
    off = __shfl_sync(0xffffffffu, off, 0);
    slot = __shfl_sync(0xffffffffu, slot, 0);
    if (slot == ~0ull) return false;
    for (int c = lane; c < k; c += 32) p.cand_pool[off + c] = cand[c];
    Task *tk = p.tasks + slot;
    if (lane < plen) tk->items[lane] = s.path[lane];
    if (lane == 0) {
        tk->items[plen] = cit;
        tk->support = sup;
        tk->len = (uint32_t)(plen + 1);
        tk->n_cand = (uint32_t)k;
        tk->cand_off = off;
    }
    __threadfence();
    __syncwarp();
    // (the fault-injection hook withholds one publish)
    if (lane == 0 && (long long)slot != p.withhold_slot) atomicExch(&tk->ready, epoch);
    __syncwarp();
    return true;
}

// The scheduling network on one class, by one warp: the arithmetic of
// dfs_kernel's inference (bf16 weights and activations, float32 sums in the
// same order); w: the CTA's copy, W1 and W2 transposed to [in][out].
__device__ void proj_mlp(const __nv_bfloat16 *w, const float *x, float *y) {
    const __nv_bfloat16 *W1t = w, *b1 = W1t + 64 * 8, *W2t = b1 + 64, *b2 = W2t + 64 * 64, *W3 = b2 + 64,
                        *b3 = W3 + 2 * 64;
    const int l = threadIdx.x & 31;
    auto f = [](__nv_bfloat16 v) { return __bfloat162float(v); };
    auto rb = [](float v) { return __bfloat162float(__float2bfloat16_rn(v)); };
    float a0 = f(b1[l]), a1 = f(b1[l + 32]);
#pragma unroll
    for (int i = 0; i < 8; i++) {
        const float xi = rb(x[i]);
        a0 = fmaf(f(W1t[i * 64 + l]), xi, a0);
        a1 = fmaf(f(W1t[i * 64 + l + 32]), xi, a1);
    }
    const float ha = rb(fmaxf(a0, 0.f)), hb = rb(fmaxf(a1, 0.f));
    float c0 = f(b2[l]), c1 = f(b2[l + 32]);
#pragma unroll 4
    for (int i = 0; i < 64; i++) {
        const float hi = __shfl_sync(0xffffffffu, i < 32 ? ha : hb, i & 31);
        c0 = fmaf(f(W2t[i * 64 + l]), hi, c0);
        c1 = fmaf(f(W2t[i * 64 + l + 32]), hi, c1);
    }
    const float g0 = rb(fmaxf(c0, 0.f)), g1 = rb(fmaxf(c1, 0.f));
    float y0 = f(W3[l]) * g0 + f(W3[l + 32]) * g1;
    float y1 = f(W3[64 + l]) * g0 + f(W3[64 + l + 32]) * g1;
    for (int d = 16; d > 0; d >>= 1) {
        y0 += __shfl_xor_sync(0xffffffffu, y0, d);
        y1 += __shfl_xor_sync(0xffffffffu, y1, d);
    }
    if (l == 0) {
        y[0] = y0 + f(b3[0]);
        y[1] = y1 + f(b3[1]);
    }
    __syncwarp();
}

// Whether a class Y = X u {c} (support supY, parent supX, k candidates with
// parent supports psup) is counted through its diffset: as the network says
// where the choice can pay for asking it (learned_kmin candidates), or by the
// size rule.  The choice never changes a count.
__device__ __noinline__ bool proj_choose_diff(const DfsParams &p, PWork<true> &s, const DbDesc &D, const __nv_bfloat16 *w,
                                              int ylen, uint32_t supY, uint32_t supX, const uint32_t *psup, int k) {
    if (p.diffset_rule && !p.learned) return supX - supY < supY;
    if (!p.learned || k < p.learned_kmin) return false;
    const int lane = threadIdx.x & 31;
    float acc = 0.f;
    for (int c = lane; c < k; c += 32) acc += (float)psup[c];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) {
        const float sx = supX > 0 ? (float)supX : 1.f, sy = supY > 0 ? (float)supY : 1.f;
        s.feat[0] = (float)ylen / 16.f;
        s.feat[1] = log2f(1.f + (float)supY) / 32.f;
        s.feat[2] = (float)supY / (float)(D.n > 0 ? D.n : 1);
        s.feat[3] = log2f(1.f + (float)k) / 16.f;
        s.feat[4] = (float)supY / sx;
        s.feat[5] = k > 0 ? acc / ((float)k * sx) : 0.f;
        s.feat[6] = log2f(1.f + (float)D.nw) / 32.f;
        s.feat[7] = (float)D.thr / sy;
    }
    __syncwarp();
    proj_mlp(w, s.feat, s.out);
    return s.out[1] > 0.f;
}

// REP: classes choose their representation (FIM_LEARNED, FIM_DIFFSET_RULE).
template <int MB, int PG, bool REP>
__global__ void __launch_bounds__(PW * 32, MB)
dfs_proj_kernel(const DfsParams p, const ProjParams q) {
    extern __shared__ __align__(16) uint8_t proj_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    PWork<REP> &s = reinterpret_cast<PWork<REP> *>(proj_smem)[warp];
    __nv_bfloat16 *const mlp = reinterpret_cast<__nv_bfloat16 *>(proj_smem + sizeof(PWork<REP>) * PW);
    if (REP && p.learned) {
        for (int i = threadIdx.x; i < FIM_MLP_PARAMS; i += PW * 32) {
            int d = i;  // W1 [64][8] and W2 [64][64] are stored [out][in]; kept [in][out]
            if (i < 64 * 8) d = (i % 8) * 64 + i / 8;
            else if (i >= 64 * 8 + 64 && i < 64 * 8 + 64 + 64 * 64) {
                const int k = i - (64 * 8 + 64);
                d = 64 * 8 + 64 + (k % 64) * 64 + k / 64;
            }
            mlp[d] = p.mlp_w[i];
        }
        __syncthreads();
    }
    // workers are numbered across the CTAs, so that few roots spread over the SMs
    const int64_t wid = (int64_t)warp * gridDim.x + blockIdx.x;
    const unsigned long long n_workers = (unsigned long long)gridDim.x * PW;
    const unsigned long long nr = q.triple ? min(*(volatile const unsigned long long *)&p.ctr->n_triples, p.rec_cap)
                                           : *(volatile const unsigned long long *)&p.ctr->n_roots;
    // a few roots can feed only so many workers: the others leave at once
    // rather than crowd the queue's counters
    if ((unsigned long long)wid >= 8 * nr) return;
    Space sp;
    sp.gfr = p.frame_items + wid * p.frame_pool;
    sp.gfs = REP ? p.frame_sups + wid * p.frame_pool : nullptr;
    sp.gst = p.stack_bits + wid * q.gstack;
    sp.gfr_cap = (int)p.frame_pool;
    sp.gst_cap = (int)q.gstack;
    const uint32_t epoch = *(volatile const uint32_t *)p.epoch;
    const DbDesc &D = p.dbs[0];
    const int mf = D.mfreq, mpw = (mf + 31) / 32;
    const uint32_t thr = D.thr, maxlen = D.maxlen;
    unsigned long long busy = 0, t_task = 0, done = 0;
    if (lane == 0) {
        atomicCAS(&p.ctr->t_first, 0ull, globaltimer_ns());
        s.rec_next = s.rec_end = s.it_next = s.it_end = 0ull;
        s.n_sup = s.n_words = s.n_bytes = s.n_classes = s.n_diff = s.emitted = s.emitted_items = 0ull;
        s.max_len = 0;
    }
    bool roots_left = true;
    // lane 0: a ticket taken ahead (roots are only ever taken by a worker that
    // runs: the mine does not depend on every CTA being resident)
    unsigned long long next = ~0ull;
    int err = 0;
    while (true) {
        // ---- the next task: a root pair, or a class from the queue ----------
        unsigned long long t = 0;
        int kind = 0;  // 1: root t, 2: queue slot t
        if (lane == 0) {
            err = *(volatile int *)&p.ctr->err;
            if (err == 0 && roots_left) {
                t = next != ~0ull ? next : atomicAdd(&p.ctr->ticket, 1ull);
                next = ~0ull;
                if (t < nr) {
                    kind = 1;
                    // far from the end the next ticket is fetched behind this task
                    if (t + 8 * n_workers < nr) next = atomicAdd(&p.ctr->ticket, 1ull);
                }
            }
            if (err == 0 && kind == 0) {
                if (done) {  // the finished roots leave the count that ends the mine
                    __threadfence();
                    atomicAdd((unsigned long long *)&p.ctr->pending, 0ull - done);
                    done = 0;
                }
                t = atomicAdd(&p.ctr->w_head, 1ull);
                unsigned long long spins = 0;
                const unsigned long long t_wait = globaltimer_ns();
                while (true) {
                    // a waiting worker polls its own slot; the shared end and
                    // error words only every 8th time
                    if (t < p.task_cap && *(volatile uint32_t *)&p.tasks[t].ready == epoch) {
                        __threadfence();
                        kind = 2;
                        break;
                    }
                    if ((spins++ & 7) == 0) {
                        if (*(volatile long long *)&p.ctr->pending == 0) break;
                        if (*(volatile int *)&p.ctr->err != 0) break;
                        if ((spins & 255) == 1 && globaltimer_ns() - t_wait > p.spin_limit) {
                            perr(p, FIM_E_TIMEOUT);
                            break;
                        }
                    }
                    __nanosleep(400);
                }
            }
            t_task = globaltimer_ns();
        }
        kind = __shfl_sync(0xffffffffu, kind, 0);
        if (kind == 0) break;
        t = __shfl_sync(0xffffffffu, t, 0);
        if (kind == 2) roots_left = false;
        // ---- its columns and candidates --------------------------------------
        uint32_t a = 0, b = 0, bc = 0;
        uint32_t supY = 0, supX = 0;  // REP: the class's support and its parent's
        int tlen = 2, kq = 0;
        unsigned long long coff_q = 0;
        if (kind == 1 && q.triple) {
            const unsigned long long r = q.roots[t];  // a << 32 | column of b << 16 | column of c
            a = (uint32_t)(r >> 32);
            bc = (uint32_t)r;
            tlen = 3;
        } else if (kind == 1) {
            const unsigned long long tt = p.root_reverse ? nr - 1 - t : t;
            const unsigned long long rt = p.root_order ? p.root_order[tt] : tt;
            a = p.root_a[rt];
            b = p.root_b[rt];
            if (REP) {
                supY = p.root_sup[rt];
                supX = __ldg(p.item_sup + __ldg(p.perm + a));
            }
        } else {
            const Task *tk = p.tasks + t;
            if (REP) supY = __ldcg(&tk->support);
            tlen = (int)__ldcg(&tk->len);
            kq = (int)__ldcg(&tk->n_cand);
            coff_q = __ldcg(&tk->cand_off);
            const uint32_t x = lane < tlen ? __ldcg(&tk->items[lane]) : 0u;
            if (lane < tlen) s.path[lane] = x;
            a = __shfl_sync(0xffffffffu, x, 0) & 0xFFFFu;
        }
        const uint32_t *cols;
        int64_t stride;
        int W;
        const uint32_t *acand = nullptr;
        uint32_t ak = 0;
        if (q.direct) {
            cols = p.bm;
            stride = D.nwp;
            W = q.direct_words;
        } else {
            const ProjItem it = q.items[a];
            cols = q.mat + it.moff;
            stride = it.W;
            W = (int)it.W;
            acand = q.cands + it.coff;
            ak = it.k;
        }
        // lanes per 128-byte run of a column: all 32 from 65 words on
        const int lg = W > 64 ? 5 : (W > 32 ? 4 : 3);
        int topS = 0, topG = 0;  // stack above the task's own prefix, if stored
        const uint32_t *src0, *src1;
        int k = 0;
        bool ok = true;
        int f0 = 0;
        if (kind == 1 && q.triple) {
            // candidates of {a, b, c}: d > c with {a, b, d} and {c, d} frequent
            const uint32_t bi = bc >> 16, ci = bc & 0xFFFFu;
            const uint32_t *row = q.triple + q.items[a].toff + (unsigned long long)bi * ak;
            const uint32_t idb = __ldg(acand + bi), idc = __ldg(acand + ci);
            const uint32_t *rc = p.pairbits + (int64_t)idc * mpw;
            f0 = place((int)(ak - ci), 0, PFR, 0, sp.gfr_cap);
            ok = f0 != INT32_MIN;
            if (ok) {
                uint32_t *fr = frame_at(s, sp, f0);
                for (uint32_t i0 = ci + 1; i0 < ak; i0 += 32) {
                    const uint32_t i = i0 + lane;
                    const uint32_t id = i < ak ? __ldg(acand + i) : 0u;
                    const uint32_t v = i < ak ? __ldg(row + i) : 0u;
                    const bool f = v != 0u && ((__ldg(rc + (id >> 5)) >> (id & 31)) & 1u);
                    const uint32_t bal = __ballot_sync(0xffffffffu, f);
                    if (f) {
                        const int at = k + __popc(bal & ((1u << lane) - 1u));
                        fr[at] = (i << 16) | id;
                        if (REP) fsup_at(s, sp, f0)[at] = v;
                    }
                    k += __popc(bal);
                }
                if (REP) {
                    supY = __ldg(row + ci);
                    supX = (uint32_t)__ldg(p.pair_cnt + (int64_t)a * mf + idb);
                }
            }
            if (lane == 0) {
                s.path[0] = a;
                s.path[1] = (bi << 16) | idb;
                s.path[2] = (ci << 16) | idc;
            }
            src0 = cols + (int64_t)bi * stride;
            src1 = cols + (int64_t)ci * stride;
        } else if (kind == 1) {
            // candidates of {a, b}: c > b with {a, c} and {b, c} frequent
            const int bound = q.direct ? mf - 1 - (int)b : (int)ak;
            f0 = place(bound, 0, PFR, 0, sp.gfr_cap);
            ok = f0 != INT32_MIN;
            uint32_t *fr = ok ? frame_at(s, sp, f0) : nullptr;
            const uint32_t *rb = p.pairbits + (int64_t)b * mpw;
            uint32_t bcol = 0;
            if (ok && q.direct) {
                const uint32_t *ra = p.pairbits + (int64_t)a * mpw;
                const int wb0 = (int)(b >> 5);
                for (int w0 = wb0; w0 < mpw; w0 += 32) {
                    const int w = w0 + lane;
                    uint32_t bits = 0;
                    if (w < mpw) {
                        bits = __ldg(ra + w) & __ldg(rb + w);
                        if (w == wb0) bits &= 0xFFFFFFFEu << (b & 31);
                    }
                    const uint32_t c = __popc(bits);
                    uint32_t x = c;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                        if (lane >= o) x += y;
                    }
                    uint32_t at = (uint32_t)k + x - c;
                    while (bits) {
                        const uint32_t id = (uint32_t)(w * 32 + __ffs(bits) - 1);
                        bits &= bits - 1;
                        if (REP) fsup_at(s, sp, f0)[at] = (uint32_t)__ldg(p.pair_cnt + (int64_t)a * mf + id);
                        fr[at++] = ((uint32_t)__ldg(p.perm + id) << 16) | id;
                    }
                    k += (int)__shfl_sync(0xffffffffu, x, 31);
                }
                bcol = (uint32_t)__ldg(p.perm + b);
            } else if (ok) {
                for (uint32_t i0 = 0; i0 < ak; i0 += 32) {
                    const uint32_t i = i0 + lane;
                    const uint32_t id = i < ak ? __ldg(acand + i) : 0u;
                    const uint32_t isb = __ballot_sync(0xffffffffu, i < ak && id == b);
                    if (isb) bcol = i0 + (uint32_t)__ffs(isb) - 1u;
                    const bool f = i < ak && id > b && ((__ldg(rb + (id >> 5)) >> (id & 31)) & 1u);
                    const uint32_t bal = __ballot_sync(0xffffffffu, f);
                    if (f) {
                        const int at = k + __popc(bal & ((1u << lane) - 1u));
                        fr[at] = (i << 16) | id;
                        if (REP) fsup_at(s, sp, f0)[at] = (uint32_t)__ldg(p.pair_cnt + (int64_t)a * mf + id);
                    }
                    k += __popc(bal);
                }
            }
            if (lane == 0) {
                s.path[0] = ((q.direct ? (uint32_t)__ldg(p.perm + a) : 0u) << 16) | a;
                s.path[1] = (bcol << 16) | b;
            }
            src1 = cols + (int64_t)bcol * stride;
            src0 = q.direct ? cols + (int64_t)__ldg(p.perm + a) * stride : src1;
        } else {
            k = kq;
            f0 = place(k, 0, PFR, 0, sp.gfr_cap);
            const int pp = place(W, 0, PST, 0, sp.gst_cap);
            ok = f0 != INT32_MIN && pp != INT32_MIN;
            src0 = src1 = nullptr;
            if (ok) {
                uint32_t *fr = frame_at(s, sp, f0);
                for (int c = lane; c < k; c += 32) fr[c] = __ldcg(p.cand_pool + coff_q + c);
                // the class's prefix: the AND of its columns (a's own column is
                // all ones in its projection)
                uint32_t *pre = stack_at(s, sp, pp);
                __syncwarp();
                for (int w = lane * 4; w < W; w += 128) {
                    uint4 y = make_uint4(~0u, ~0u, ~0u, ~0u);
                    for (int x = q.direct ? 0 : 1; x < tlen; x++)
                        y = and4(y, ldg_u4(cols + (int64_t)(s.path[x] >> 16) * stride + w));
                    *reinterpret_cast<uint4 *>(pre + w) = y;
                }
                src0 = src1 = pre;
                if (pp >= 0) topS = pp + W; else topG = ~pp + W;
            }
        }
        __syncwarp();
        const bool len_ok = maxlen == 0 || (uint32_t)tlen + 1 <= maxlen;
        // the class to count next: prefix src0 AND src1, kc candidates at cf,
        // child level L + 1
        int L = -1, kc = k, fc = f0, sc = 0, plen = tlen;
        if (ok && k >= 2) {
            sc = place(W, topS, PST, topG, sp.gst_cap);
            ok = sc != INT32_MIN;
        }
        if (!ok && lane == 0) perr(p, FIM_E_STACK);
        bool go = ok && k > 0 && len_ok;
        // this task's classes, supports and longest set
        uint32_t t_cls = 0, t_sup = 0, t_diff = 0;
        int t_len = 0;
        while (go) {
            // the error flag and how many workers wait for the queue: loaded
            // here, used after the class has been counted
            int q_err = 0;
            uint32_t q_head = 0, q_tail = 0;
            if (lane == 0) {
                q_err = *(volatile int *)&p.ctr->err;
                q_head = *(volatile uint32_t *)&p.ctr->w_head;
                q_tail = *(volatile uint32_t *)&p.ctr->w_tail;
            }
            bool polled = false;
            {
                uint32_t *cf = frame_at(s, sp, fc), *cs = fsup_at(s, sp, fc);
                // (a queued class's prefix comes whole, and a projected pair's
                // parent is all of T(a): no parent's bitmap to differ from)
                bool diff = false;
                if constexpr (REP)
                    if (L >= 0 || (kind == 1 && (q.triple || q.direct))) diff = proj_choose_diff(p, s, D, mlp, plen, supY, supX, cs, kc);
                const int nF = proj_class_pass<PG, REP>(p, s, thr, src0, src1, cols, stride, W, lg, cf, kc, plen,
                                                        kc >= 2 ? stack_at(s, sp, sc) : nullptr, cf, cs, diff);
                t_cls++;
                t_sup += (uint32_t)kc;
                t_diff += diff;
                if (nF > 0 && plen + 1 > t_len) t_len = plen + 1;
                // sets of plen + 1 items: their classes give sets of plen + 2
                if (nF >= 2 && (maxlen == 0 || (uint32_t)plen + 2 <= maxlen)) {
                    L++;
                    if (lane == 0) {
                        const int bS = L > 0 ? s.ftopS[L - 1] : 0, bG = L > 0 ? s.ftopG[L - 1] : 0;
                        if (REP) s.supY[L] = supY;
                        s.nF[L] = nF;
                        s.cur[L] = 0;
                        s.fpos[L] = fc;
                        s.ftopS[L] = fc >= 0 ? fc + nF : bS;
                        s.ftopG[L] = fc >= 0 ? bG : ~fc + nF;
                        s.spos[L] = sc;
                        s.stopS[L] = sc >= 0 ? sc + W : (L > 0 ? s.stopS[L - 1] : topS);
                        s.stopG[L] = sc >= 0 ? (L > 0 ? s.stopG[L - 1] : topG) : ~sc + W;
                    }
                }
                __syncwarp();
            }
            // ---- the next class, depth first --------------------------------
            go = false;
            while (L >= 0) {
                if (!polled) {
                    polled = true;
                    if (__shfl_sync(0xffffffffu, q_err, 0)) break;
                    const int want = __shfl_sync(0xffffffffu, (int)(q_head - q_tail), 0);
                    if (want > 0 && p.split_depth) {
                        // hand over the next siblings of the shallowest levels
                        // (the largest subtrees this worker still holds)
                        const int most = want < PGIVE ? want : PGIVE;
                        for (int l = 0, given = 0; l <= L && given < most; l++) {
                            if (tlen + l + 1 > p.split_depth || tlen + l + 1 > FIM_TASK_MAXR) break;
                            while (given < most && s.cur[l] + 1 < s.nF[l]) {
                                const int at = place(s.nF[l], s.ftopS[L], PFR, s.ftopG[L], sp.gfr_cap);
                                if (at == INT32_MIN) break;
                                uint32_t *tmp = frame_at(s, sp, at), cit = 0;
                                const uint32_t *ls = fsup_at(s, sp, s.fpos[l]);
                                const int kd = siblings<REP>(p, mpw, frame_at(s, sp, s.fpos[l]), ls, s.cur[l], s.nF[l],
                                                             tmp, fsup_at(s, sp, at), &cit);
                                if (kd == 1) break;  // too small to move
                                if (kd > 1 && !give(p, s, epoch, tlen + l, cit, REP ? ls[s.cur[l]] : 0u, tmp, kd)) break;
                                given += kd > 1;
                                __syncwarp();
                                if (lane == 0) s.cur[l]++;
                                __syncwarp();
                            }
                        }
                    }
                }
                const int nFL = s.nF[L], j = s.cur[L];
                if (j + 1 >= nFL) {  // the last sibling has no later ones to combine with
                    L--;
                    continue;
                }
                plen = tlen + L;
                fc = place(nFL - j - 1, s.ftopS[L], PFR, s.ftopG[L], sp.gfr_cap);
                if (fc == INT32_MIN) {
                    if (lane == 0) perr(p, FIM_E_STACK);
                    break;
                }
                uint32_t cit = 0;
                kc = siblings<REP>(p, mpw, frame_at(s, sp, s.fpos[L]), fsup_at(s, sp, s.fpos[L]), j, nFL,
                                   frame_at(s, sp, fc), fsup_at(s, sp, fc), &cit);
                if (REP) {
                    supX = s.supY[L];
                    supY = fsup_at(s, sp, s.fpos[L])[j];
                }
                __syncwarp();  // cur[L] and the path have been read
                if (lane == 0) {
                    s.cur[L] = j + 1;
                    s.path[plen] = cit;
                }
                __syncwarp();
                if (kc == 0) continue;
                sc = kc >= 2 ? place(W, s.stopS[L], PST, s.stopG[L], sp.gst_cap) : 0;
                if (sc == INT32_MIN || L + 2 >= PLV) {
                    if (lane == 0) perr(p, FIM_E_STACK);
                    break;
                }
                src0 = stack_at(s, sp, s.spos[L]);
                src1 = cols + (int64_t)(cit >> 16) * stride;
                plen++;
                go = true;
                break;
            }
        }
        __syncwarp();
        if (lane == 0) {
            s.n_sup += t_sup;
            s.n_classes += t_cls;
            s.n_diff += t_diff;
            s.n_words += (unsigned long long)t_sup * (unsigned long long)W;
            s.n_bytes += 4ull * (unsigned long long)W * ((unsigned long long)t_sup + 3ull * t_cls);
            if (t_len > s.max_len) s.max_len = t_len;
            busy += globaltimer_ns() - t_task;
            if (kind == 1) {
                done++;
            } else {
                __threadfence();
                atomicAdd((unsigned long long *)&p.ctr->pending, (unsigned long long)(-1ll));
            }
        }
    }
    if (lane == 0) {
        if (done) atomicAdd((unsigned long long *)&p.ctr->pending, 0ull - done);
        // the worker's unused slots become holes
        for (unsigned long long r = s.rec_next; r < s.rec_end; r++)
            if (r < p.rec_cap) p.rec_len[r] = 0u;
        if (s.rec_end > s.rec_next) atomicAdd(&p.ctr->rec_holes, s.rec_end - s.rec_next);
        if (s.it_end > s.it_next) atomicAdd(&p.ctr->item_holes, s.it_end - s.it_next);
        if (s.n_classes) {
            atomicAdd(&p.ctr->supports_dfs, s.n_sup);
            atomicAdd(&p.ctr->dfs_words, s.n_words);
            atomicAdd(&p.ctr->dfs_bytes, s.n_bytes);
            atomicAdd(&p.ctr->dfs_touched, s.n_bytes);
            atomicAdd(&p.ctr->classes, s.n_classes);
            if (s.n_diff) atomicAdd(&p.ctr->diffset, s.n_diff);
        }
        if (s.max_len) atomicMax(&p.ctr->max_len, s.max_len);
        atomicAdd(&p.ctr->busy_ns, busy);
        atomicMax(&p.ctr->t_last, globaltimer_ns());
    }
}

}  // namespace

int proj_workers_per_cta() { return PW; }

// Sizes of the projection, on the device; the totals come back to the host.
int launch_proj_plan(fim_ctx *ctx, ProjTotals *host) {
    const int mf = ctx->mfreq, mpw = (int)ceil_div64(mf, 32);
    cudaStream_t st = ctx->stream;
    FIM_TRY(fim_reserve(ctx, ctx->proj_items, sizeof(ProjItem) * (size_t)mf));
    FIM_TRY(fim_reserve(ctx, ctx->proj_tiles, 2 * sizeof(unsigned long long) * (size_t)(mf + 1)));
    FIM_TRY(fim_reserve(ctx, ctx->proj_totals, sizeof(ProjTotals)));
    FIM_CUDA_TRY(cudaMemsetAsync(ctx->proj_totals.p, 0, sizeof(ProjTotals), st));
    ctx->launches += 2;
    proj_count_kernel<<<(unsigned)ceil_div64((int64_t)mf * 32, 256), 256, 0, st>>>(
        ctx->pairbits.as<uint32_t>(), mf, mpw, ctx->perm.as<int32_t>(), ctx->item_sup.as<uint32_t>(),
        ctx->proj_items.as<ProjItem>());
    unsigned long long *tile0 = ctx->proj_tiles.as<unsigned long long>();
    proj_scan_kernel<<<1, 1024, 0, st>>>(ctx->proj_items.as<ProjItem>(), mf, tile0, tile0 + (mf + 1),
                                         ctx->proj_totals.as<ProjTotals>());
    FIM_CUDA_TRY(cudaGetLastError());
    FIM_CUDA_TRY(cudaMemcpyAsync(host, ctx->proj_totals.p, sizeof(ProjTotals), cudaMemcpyDeviceToHost, st));
    FIM_CUDA_TRY(cudaStreamSynchronize(st));
    return FIM_OK;
}

// The projected columns of every item of the plan, which has candidates.
int launch_projection(fim_ctx *ctx, int mf, const ProjTotals &t, bool cands_listed, bool triples, uint32_t thr) {
    MineCounters *d_ctr = ctx->counters.as<MineCounters>();
    const int mpw = (int)ceil_div64(mf, 32);
    cudaStream_t st = ctx->stream;
    FIM_TRY(fim_reserve(ctx, ctx->proj_mat, sizeof(uint32_t) * (size_t)t.words));
    FIM_TRY(fim_reserve(ctx, ctx->proj_list, sizeof(uint32_t) * (size_t)t.rows));
    FIM_TRY(fim_reserve(ctx, ctx->proj_cands, sizeof(uint32_t) * (size_t)t.cands));
    if (!cands_listed) {
        ctx->launches++;
        proj_cands_kernel<<<(unsigned)ceil_div64((int64_t)mf * 32, 256), 256, 0, st>>>(
            ctx->pairbits.as<uint32_t>(), mf, mpw, ctx->proj_items.as<ProjItem>(), ctx->proj_cands.as<uint32_t>(),
            d_ctr, triples ? 1 : 0);
    }
    ctx->launches += 2;
    const bool wide = (int64_t)mf * ctx->nwp > (4ll << 20);
    const dim3 grid((unsigned)ceil_div64(ctx->nwp, TL_T * 4 * (wide ? 8 : 1)), (unsigned)mf);
    (wide ? tid_list_kernel<8> : tid_list_kernel<1>)<<<grid, TL_T, 0, st>>>(
        ctx->bm.as<uint32_t>(), ctx->perm.as<int32_t>(), ctx->nwp, ctx->proj_items.as<ProjItem>(),
        ctx->proj_list.as<uint32_t>());
    // few tiles: several warps share a tile's candidates (a small plan's
    // totals are its worst case, many times its tiles)
    const int64_t want = (int64_t)ctx->num_sms * 64;
    int csplit = (int)(want / (int64_t)(t.tiles ? t.tiles : 1));
    csplit = csplit < 1 ? 1 : (csplit > 8 ? 8 : csplit);
    if (cands_listed) csplit = 12;
    const int64_t units = ceil_div64((int64_t)t.tiles * csplit, 8);
    proj_gather_kernel<<<(unsigned)min64(units, 1 << 20), 256, 0, st>>>(
        ctx->bm.as<uint32_t>(), ctx->perm.as<int32_t>(), ctx->nwp, mf, ctx->proj_items.as<ProjItem>(),
        ctx->proj_tiles.as<unsigned long long>(), ctx->proj_list.as<uint32_t>(), ctx->proj_cands.as<uint32_t>(),
        ctx->proj_mat.as<uint32_t>(), csplit);
    if (triples) {
        FIM_TRY(fim_reserve(ctx, ctx->proj_triple, sizeof(uint32_t) * (size_t)t.triples));
        FIM_TRY(fim_reserve(ctx, ctx->proj_roots, sizeof(unsigned long long) * (size_t)ctx->rec_cap));
        const int64_t blocks = min64(ceil_div64((int64_t)t.units, 8), (int64_t)ctx->num_sms * 16);
        ctx->launches++;
        proj_triple_kernel<<<(unsigned)blocks, 256, 0, st>>>(
            ctx->proj_items.as<ProjItem>(), mf, ctx->proj_tiles.as<unsigned long long>() + (mf + 1),
            ctx->proj_cands.as<uint32_t>(), ctx->proj_mat.as<uint32_t>(), ctx->pairbits.as<uint32_t>(), ctx->dbdesc.as<DbDesc>(), thr,
            ctx->proj_triple.as<uint32_t>(), ctx->proj_roots.as<unsigned long long>(), d_ctr,
            ctx->rec_off.as<unsigned long long>(), ctx->rec_len.as<uint32_t>(), ctx->rec_sup.as<uint32_t>(),
            ctx->rec_items.as<uint32_t>(), ctx->rec_cap, ctx->rec_items_cap);
    }
    FIM_CUDA_TRY(cudaGetLastError());
    return FIM_OK;
}

unsigned long long proj_triple_units(int mf) { return triple_units((uint32_t)(mf > 0 ? mf : 0)); }

bool proj_small_plan_fits(int mf) { return mf <= SP_MAX; }

// Pair threshold, records, roots and the projection's plan of a small mine
// (in place of launch_pairs_finalize, the root plan and launch_proj_plan).
// mf: m', or a bound of it.
int launch_proj_small_plan(fim_ctx *ctx, int mf, uint32_t thr, MineCounters *d_ctr, bool triples, bool ask) {
    const size_t npairs = (size_t)mf * (mf - 1) / 2;
    FIM_TRY(fim_reserve(ctx, ctx->proj_items, sizeof(ProjItem) * (size_t)mf));
    FIM_TRY(fim_reserve(ctx, ctx->proj_tiles, 2 * sizeof(unsigned long long) * (size_t)(mf + 1)));
    FIM_TRY(fim_reserve(ctx, ctx->proj_totals, sizeof(ProjTotals)));
    FIM_TRY(fim_reserve(ctx, ctx->proj_cands, sizeof(uint32_t) * npairs));
    uint32_t *roots = ctx->roots.as<uint32_t>();
    ctx->launches++;
    proj_small_plan_kernel<<<1, SP_T, 0, ctx->stream>>>(
        ctx->pair_cnt.as<int>(), mf, thr, ctx->perm.as<int32_t>(), ctx->item_sup.as<uint32_t>(),
        ctx->pairbits.as<uint32_t>(), d_ctr, ctx->epoch.as<uint32_t>(), ctx->rec_off.as<unsigned long long>(),
        ctx->rec_len.as<uint32_t>(), ctx->rec_sup.as<uint32_t>(), ctx->rec_items.as<uint32_t>(), ctx->rec_cap,
        ctx->rec_items_cap, roots, roots + npairs, roots + 2 * npairs, ctx->root_order.as<uint32_t>(),
        ctx->proj_items.as<ProjItem>(), ctx->proj_tiles.as<unsigned long long>(),
        ctx->proj_tiles.as<unsigned long long>() + (mf + 1), ctx->proj_cands.as<uint32_t>(),
        ctx->proj_totals.as<ProjTotals>(), triples ? 1 : 0, ask ? 1 : 0);
    FIM_CUDA_TRY(cudaGetLastError());
    return FIM_OK;
}

int launch_dfs_proj(fim_ctx *ctx, const DfsParams &p, const ProjParams &q, int ctas_per_sm) {
    const bool rep = p.learned || p.diffset_rule;
    const size_t smem = rep ? sizeof(PWork<true>) * PW + sizeof(__nv_bfloat16) * (FIM_MLP_PARAMS + 6)
                            : sizeof(PWork<false>) * PW;
    const unsigned grid = (unsigned)(ctx->num_sms * ctas_per_sm);
    auto kern = rep ? (ctas_per_sm >= 4 ? dfs_proj_kernel<4, 4, true> : dfs_proj_kernel<2, 8, true>)
                    : (ctas_per_sm >= 4   ? dfs_proj_kernel<4, 4, false>
                       : ctas_per_sm == 3 ? dfs_proj_kernel<3, 8, false>
                                          : dfs_proj_kernel<2, 8, false>);
    FIM_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    ctx->launches++;
    kern<<<grid, PW * 32, smem, ctx->stream>>>(p, q);
    FIM_CUDA_TRY(cudaGetLastError());
    return FIM_OK;
}
