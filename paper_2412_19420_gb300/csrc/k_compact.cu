// k_compact.cu -- frequent-itemset extraction into canonical order.
//
// Records come out of the miner in discovery order with internal item ids.
// The compactor
//   1. maps items to the caller's ids and sorts each set's items (in place);
//   2. packs a big-endian key  [len : 8 bits][item_0 : b]...[item_{L-1} : b]
//      (b = bits per item id), so that numeric key order is the canonical
//      order: size first, then lexicographic;
//   3. sorts the records by that key with a stable LSD radix sort of
//      (key word, record) pairs, 64-bit key words from the least significant
//      one: each word is gathered once into record order, then sorted by its
//      8-bit digits, one launch a digit (small outputs: one CTA, or the cluster
//      of k_csort.cu);
//   4. writes offsets (exclusive scan of the sizes), items and supports.
#include <utility>
#include <vector>

#include "fim_common.cuh"

namespace {

constexpr int RI = 8;            // keys per thread of a radix tile

// Items a set's key is made of in a local copy (longer sets: in place, a chain
// of round trips to global memory).
constexpr int PK_LOCAL = 16;

// Big-endian bit packing into 64-bit words (word 0 most significant), handed
// to emit(word index, word) as they fill.
template <class Emit>
struct KeyPack {
    Emit emit;
    unsigned long long w = 0;
    int used = 0, wi = 0;
    __device__ __forceinline__ explicit KeyPack(Emit e) : emit(e) {}
    __device__ __forceinline__ void put(unsigned long long v, int nb) {
        while (nb > 0) {
            const int room = 64 - used;
            const int take = nb < room ? nb : room;
            const unsigned long long part = (v >> (nb - take)) & ((take == 64) ? ~0ull : ((1ull << take) - 1));
            w |= part << (room - take);
            used += take;
            nb -= take;
            if (used == 64) { emit(wi, w); wi++; w = 0; used = 0; }
        }
    }
    __device__ __forceinline__ void end(int kw) {  // the last word, then zeros
        if (used > 0) { emit(wi, w); wi++; }
        for (; wi < kw; wi++) emit(wi, 0ull);
    }
};

// (With the sort in place this pass took 450 us of 4.2 million records, now 189.)
// dbs/rec_db/db_bits: with several databases the key starts with the record's
// database (db_bits wide) and items map back through that database's perm.
__global__ void prep_keys_kernel(unsigned long long R, const unsigned long long *__restrict__ rec_off,
                                 const uint32_t *__restrict__ rec_len, uint32_t *__restrict__ items,
                                 const int32_t *__restrict__ perm_base, const DbDesc *__restrict__ dbs,
                                 const uint32_t *__restrict__ rec_db, int db_bits, int bits, int kw,
                                 unsigned long long *__restrict__ keys, uint32_t *__restrict__ idx) {
    const unsigned long long r = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= R) return;
    idx[r] = (uint32_t)r;
    const int len = (int)rec_len[r];
    if (len == 0) {  // a hole: the largest key, after every itemset
        for (int w = 0; w < kw; w++) keys[(unsigned long long)w * R + r] = ~0ull;
        return;
    }
    const unsigned long long off = rec_off[r];
    const uint32_t db = db_bits ? rec_db[r] : 0u;
    uint32_t *const it = items + off;
    const int32_t *const perm = perm_base ? perm_base + dbs[db].item_off : nullptr;  // null: already the caller's ids
    // an insertion sort (sets are short), on a local copy where it fits
    uint32_t loc[PK_LOCAL];
    uint32_t *const v = len <= PK_LOCAL ? loc : it;
    for (int q = 0; q < len; q++) {
        const uint32_t raw = it[q];
        const uint32_t x = perm ? (uint32_t)__ldg(perm + raw) : raw;
        int z = q - 1;
        while (z >= 0 && v[z] > x) { v[z + 1] = v[z]; z--; }
        v[z + 1] = x;
    }
    auto emit = [&](int q, unsigned long long v) { keys[(unsigned long long)q * R + r] = v; };
    KeyPack<decltype(emit)> pk(emit);
    if (db_bits) pk.put((unsigned long long)db, db_bits);
    pk.put((unsigned long long)len, 8);
    for (int q = 0; q < len; q++) {
        pk.put(v[q], bits);
        if (v != it) it[q] = v[q];
    }
    pk.end(kw);
}

// The whole compaction of a small output (one database, at most OC_MAX
// records) in one CTA: keys as above in shared memory, a bitonic sort of
// record numbers by key, a scan of the sizes, the canonical output.  These
// mines return a few hundred sets, and five launches with their gaps took
// 36 us of a 10,000 x 169 mine where this takes 10.  Past OC_MAX records the
// sort's log^2 steps in one CTA cost more than the cluster's launches (1,500
// sets: 10 us slower).
constexpr int OC_T = 512, OC_MAX = 1024, OC_KW = 4;
size_t oc_smem(int kw) { return sizeof(unsigned long long) * (size_t)kw * OC_MAX; }
__global__ void __launch_bounds__(OC_T)
one_cta_compact_kernel(int R, int R_valid, const unsigned long long *__restrict__ rec_off,
                       const uint32_t *__restrict__ rec_len, const uint32_t *__restrict__ rec_sup,
                       uint32_t *__restrict__ items, const int32_t *__restrict__ perm, int bits, int kw,
                       unsigned long long *__restrict__ out_off, uint32_t *__restrict__ out_items,
                       uint32_t *__restrict__ out_sup, unsigned long long total_items) {
    extern __shared__ __align__(16) unsigned long long oc_key[];  // [kw][OC_MAX]
    __shared__ unsigned short idx[OC_MAX];
    __shared__ uint32_t lens[OC_MAX], wsum[OC_T / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int n2 = 64;  // slots of the sort: a power of two
    while (n2 < R) n2 <<= 1;
    for (int r = tid; r < n2; r += OC_T) {
        idx[r] = (unsigned short)r;
        const int len = r < R ? (int)rec_len[r] : 0;
        lens[r] = (uint32_t)len;
        if (len == 0) {  // a hole or an empty slot: after every itemset
            for (int w = 0; w < kw; w++) oc_key[w * OC_MAX + r] = ~0ull;
            continue;
        }
        uint32_t *const it = items + rec_off[r];
        // an insertion sort (sets are short), on a local copy where it fits: in
        // place it is a chain of round trips to global memory
        uint32_t loc[PK_LOCAL];
        uint32_t *const v = len <= PK_LOCAL ? loc : it;
        for (int q = 0; q < len; q++) {
            const uint32_t raw = it[q];
            const uint32_t x = perm ? (uint32_t)__ldg(perm + raw) : raw;
            int z = q - 1;
            while (z >= 0 && v[z] > x) { v[z + 1] = v[z]; z--; }
            v[z + 1] = x;
        }
        auto emit = [&](int q, unsigned long long w) { oc_key[q * OC_MAX + r] = w; };
        KeyPack<decltype(emit)> pk(emit);
        pk.put((unsigned long long)len, 8);
        for (int q = 0; q < len; q++) {
            pk.put(v[q], bits);
            if (v != it) it[q] = v[q];
        }
        pk.end(kw);
    }
    __syncthreads();
    for (int k = 2; k <= n2; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int t = tid; t < n2 / 2; t += OC_T) {
                const int i = 2 * t - (t & (j - 1)), l = i + j;  // the pair (i, i ^ j)
                const int a = idx[i], b = idx[l];
                bool gt = false;  // key a > key b
                for (int w = 0; w < kw; w++) {
                    const unsigned long long x = oc_key[w * OC_MAX + a], y = oc_key[w * OC_MAX + b];
                    if (x != y) { gt = x > y; break; }
                }
                if (gt == ((i & k) == 0)) {
                    idx[i] = (unsigned short)b;
                    idx[l] = (unsigned short)a;
                }
            }
            __syncthreads();
        }
    // offsets: a scan of the sizes in sorted order, two positions a thread
    const uint32_t l0 = 2 * tid < n2 ? lens[idx[2 * tid]] : 0u, l1 = 2 * tid + 1 < n2 ? lens[idx[2 * tid + 1]] : 0u;
    uint32_t x = l0 + l1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    uint32_t before = x - l0 - l1;
    for (int w = 0; w < warp; w++) before += wsum[w];
    for (int h = 0; h < 2; h++) {
        const int q = 2 * tid + h;
        if (q < R_valid) {
            const int r = idx[q];
            const uint32_t len = h ? l1 : l0;
            const uint32_t *it = items + rec_off[r];
            out_off[q] = before;
            out_sup[q] = rec_sup[r];
            for (uint32_t z = 0; z < len; z++) out_items[before + z] = it[z];
            before += len;
        } else if (q == R_valid) {
            out_off[q] = total_items;
        }
    }
    if (tid == 0 && R_valid == OC_MAX) out_off[OC_MAX] = total_items;
}

// out[i] = word[idx[i]]: one key word in the records' current order.
__global__ void gather_word_kernel(const unsigned long long *__restrict__ word, const uint32_t *__restrict__ idx,
                                   unsigned long long n, unsigned long long *__restrict__ out,
                                   const int *__restrict__ err) {
    const unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && *err == 0) out[i] = word[idx[i]];
}

// ---- the radix sort of a large output ------------------------------------
// One pass over the keys counts every digit of every word; one launch turns the
// counts into bases; then each digit is one launch: a tile ranks its keys
// (warp match, per-warp counts), publishes its digit counts, adds up its
// predecessors' (decoupled look-back) and scatters.  (A histogram, three scan
// launches and a scatter per digit took 55 us of 4.2 million records and 25 of
// 190,000; a digit is now 44 and 7 us and the count 9 and 1 a digit.  With the
// keys' local sort, whole compactions: 4.2 million sets 2.0 -> 1.66 ms, 640,000
// sets 0.82 -> 0.40, 190,000 sets 0.85 -> 0.31.)
constexpr int RS_MAXPASS = 64;   // digits counted in one launch

struct RsPasses {
    int n;
    signed char word[RS_MAXPASS];
    signed char shift[RS_MAXPASS];
};

__global__ void __launch_bounds__(512)
rs_count_kernel(const unsigned long long *__restrict__ keys, unsigned long long n, RsPasses ps,
                unsigned long long *__restrict__ hist) {
    extern __shared__ uint32_t rs_h[];  // [ps.n][256]
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < ps.n * 256; i += blockDim.x) rs_h[i] = 0;
    __syncthreads();
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long b = (unsigned long long)blockIdx.x * blockDim.x; b < n; b += stride) {  // block-uniform
        const unsigned long long r = b + threadIdx.x;
        int w = -1;
        unsigned long long k = 0;
        for (int p = 0; p < ps.n; p++) {
            if (ps.word[p] != w) {
                w = ps.word[p];
                k = r < n ? keys[(unsigned long long)w * n + r] : 0ull;
            }
            const uint32_t d = r < n ? (uint32_t)((k >> ps.shift[p]) & 255u) : 256u;
            // the keys that share lane 0's digit count as one add (sizes, and
            // the zeros behind short sets, are shared by nearly all), the
            // others one by one; a match over the warp took 20 cycles a digit
            const uint32_t d0 = __shfl_sync(0xffffffffu, d, 0);
            const uint32_t same = __ballot_sync(0xffffffffu, d == d0);
            if (lane == 0) {
                if (d < 256u) atomicAdd(&rs_h[p * 256 + d], (uint32_t)__popc(same));
            } else if (d != d0 && d < 256u) {
                atomicAdd(&rs_h[p * 256 + d], 1u);
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < ps.n * 256; i += blockDim.x)
        if (rs_h[i]) atomicAdd(&hist[i], (unsigned long long)rs_h[i]);
}

// Exclusive scan of each digit's 256 counts: one CTA per digit.
__global__ void __launch_bounds__(256)
rs_base_kernel(unsigned long long *__restrict__ hist) {
    __shared__ unsigned long long ws[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long *h = hist + (size_t)blockIdx.x * 256;
    const unsigned long long v = h[threadIdx.x];
    unsigned long long x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[warp] = x;
    __syncthreads();
    unsigned long long before = x - v;
    for (int w = 0; w < warp; w++) before += ws[w];
    h[threadIdx.x] = before;
}

// A tile's published word of one digit: flag in the top two bits (1: its own
// count, 2: the count up to and including it), the count below.
constexpr unsigned long long RS_OWN = 1ull << 62, RS_ALL = 2ull << 62, RS_VAL = RS_OWN - 1;
// A look-back waits 2 s at most (far above any legitimate wait), or the ctx's
// spin limit.  On expiry the tile sets the error word and scatters nothing, so
// record numbers are missing from then on: later launches look at the word
// first and leave them alone, and the output pass writes the records as they
// lie.  The call that reads the output reports FIM_E_TIMEOUT.
constexpr unsigned long long RS_WAIT_NS = 2000000000ull;

template <int NT>
__global__ void __launch_bounds__(NT)
rs_digit_kernel(const unsigned long long *__restrict__ key_in, const uint32_t *__restrict__ idx_in,
                unsigned long long *__restrict__ key_out, uint32_t *__restrict__ idx_out, unsigned long long n,
                int shift, const unsigned long long *__restrict__ base, unsigned long long *status,
                unsigned long long *__restrict__ next_status, uint32_t *__restrict__ ticket, int *err,
                unsigned long long wait_ns, long long withhold) {
    constexpr int NW = NT / 32;
    __shared__ uint32_t wc[NW][256];            // per-warp digit counts, then offsets
    __shared__ unsigned long long dst[256];     // where the tile's keys of a digit go
    __shared__ uint32_t s_tile;
    __shared__ int s_bad;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        // tiles in the order CTAs start: a tile only waits for tiles that run
        s_tile = atomicAdd(ticket, 1u);
        s_bad = *(volatile int *)err;
    }
    for (int i = threadIdx.x; i < NW * 256; i += NT) (&wc[0][0])[i] = 0;
    __syncthreads();
    if (s_bad) return;  // (a running tile that needs this one's counts sees the word too)
    const unsigned long long tile = s_tile;
    if (threadIdx.x < 256) next_status[tile * 256 + threadIdx.x] = 0ull;  // the next digit's words
    const unsigned long long t0 = tile * (NT * RI) + (unsigned long long)warp * (32 * RI);
    unsigned long long k[RI];
    uint32_t v[RI], rank[RI];
#pragma unroll
    for (int i = 0; i < RI; i++) {
        const unsigned long long e = t0 + i * 32 + lane;
        k[i] = e < n ? key_in[e] : 0ull;
        v[i] = e < n ? idx_in[e] : 0u;
    }
#pragma unroll
    for (int i = 0; i < RI; i++) {  // stable within the warp: its keys in order
        const unsigned long long e = t0 + i * 32 + lane;
        const uint32_t d = e < n ? (uint32_t)((k[i] >> shift) & 255u) : 256u;
        const uint32_t peers = __match_any_sync(0xffffffffu, d);
        const uint32_t below = __popc(peers & ((1u << lane) - 1u));
        uint32_t c = 0;
        if (d < 256u) c = wc[warp][d];
        __syncwarp();
        rank[i] = c + below;
        if (d < 256u && below == 0) wc[warp][d] = c + (uint32_t)__popc(peers);
        __syncwarp();
    }
    __syncthreads();
    if (threadIdx.x < 256) {
        const int d = threadIdx.x;
        uint32_t cnt = 0;
        for (int w = 0; w < NW; w++) {
            const uint32_t c = wc[w][d];
            wc[w][d] = cnt;
            cnt += c;
        }
        volatile unsigned long long *st = status + d;
        unsigned long long pre = 0;
        const bool publish = (long long)tile != withhold;  // (the fault-injection hook withholds one tile's)
        if (tile == 0) {
            if (publish) st[0] = RS_ALL | cnt;
        } else {
            if (publish) st[tile * 256] = RS_OWN | cnt;
            // predecessors LB at a time, their words loaded together: hundreds
            // of tiles start at once, and one word after another is a round
            // trip to L2 each
            constexpr int LB = 8;
            const unsigned long long t_wait = globaltimer_ns();
            long long q = (long long)tile - 1;
            bool more = true;
            while (more) {
                unsigned long long x[LB];
#pragma unroll
                for (int i = 0; i < LB; i++) x[i] = q - i >= 0 ? (unsigned long long)st[(q - i) * 256] : (2ull << 62);
#pragma unroll
                for (int i = 0; i < LB; i++) {
                    if (!more) break;
                    while (!(x[i] >> 62)) {
                        if (globaltimer_ns() - t_wait > wait_ns || *(volatile int *)err) {
                            s_bad = 1;
                            break;
                        }
                        x[i] = st[(q - i) * 256];
                    }
                    pre += x[i] & RS_VAL;
                    more = (x[i] >> 62) == 1;  // else everything before is in it (or the wait ran out)
                }
                q -= LB;
            }
            if (publish) st[tile * 256] = RS_ALL | (pre + cnt);
        }
        dst[d] = base[d] + pre;
    }
    __syncthreads();
    if (s_bad) {  // reported, nothing scattered
        if (threadIdx.x == 0) atomicExch(err, 1);
        return;
    }
#pragma unroll
    for (int i = 0; i < RI; i++) {
        const unsigned long long e = t0 + i * 32 + lane;
        if (e >= n) continue;
        const uint32_t d = (uint32_t)((k[i] >> shift) & 255u);
        const unsigned long long o = dst[d] + wc[warp][d] + rank[i];
        key_out[o] = k[i];
        idx_out[o] = v[i];
    }
}

// The record at position q of the sorted order; record q itself after a sort
// whose look-back ran out (err), which left record numbers unwritten.
__device__ __forceinline__ uint32_t sorted_record(const uint32_t *idx, unsigned long long q, const int *err) {
    return err && *err ? (uint32_t)q : idx[q];
}

// Sizes in sorted order, block sums for the offset scan.
constexpr int ST = 1024;
__global__ void __launch_bounds__(ST)
len_block_sums_kernel(const uint32_t *__restrict__ idx, const uint32_t *__restrict__ rec_len,
                      unsigned long long R, unsigned long long *__restrict__ bsum, const int *__restrict__ err) {
    __shared__ unsigned long long s[ST / 32];
    const unsigned long long q = (unsigned long long)blockIdx.x * ST + threadIdx.x;
    unsigned long long v = q < R ? rec_len[sorted_record(idx, q, err)] : 0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long t = 0;
        for (int w = 0; w < ST / 32; w++) t += s[w];
        bsum[blockIdx.x] = t;
    }
}

__global__ void __launch_bounds__(1024)
scan_u64_single_kernel(unsigned long long *__restrict__ a, unsigned long long n) {
    __shared__ unsigned long long s[1024];
    const unsigned long long seg = (n + 1023) / 1024;
    const unsigned long long b = threadIdx.x * seg, e = b + seg < n ? b + seg : n;
    unsigned long long sum = 0;
    for (unsigned long long i = b; i < e; i++) sum += a[i];
    s[threadIdx.x] = sum;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
        unsigned long long v = threadIdx.x >= (unsigned)o ? s[threadIdx.x - o] : 0;
        __syncthreads();
        s[threadIdx.x] += v;
        __syncthreads();
    }
    unsigned long long run = s[threadIdx.x] - sum;
    for (unsigned long long i = b; i < e; i++) {
        const unsigned long long v = a[i];
        a[i] = run;
        run += v;
    }
}

__global__ void __launch_bounds__(ST)
emit_sorted_kernel(const uint32_t *__restrict__ idx, unsigned long long R,
                   const unsigned long long *__restrict__ rec_off, const uint32_t *__restrict__ rec_len,
                   const uint32_t *__restrict__ rec_sup, const uint32_t *__restrict__ items,
                   const unsigned long long *__restrict__ bsum, unsigned long long *__restrict__ out_off,
                   uint32_t *__restrict__ out_items, uint32_t *__restrict__ out_sup,
                   unsigned long long total_items, const int *__restrict__ err) {
    __shared__ unsigned long long s[ST / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned long long q = (unsigned long long)blockIdx.x * ST + threadIdx.x;
    uint32_t r = 0;
    unsigned long long len = 0;
    if (q < R) { r = sorted_record(idx, q, err); len = rec_len[r]; }
    unsigned long long x = len;
    for (int o = 1; o < 32; o <<= 1) {
        unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s[warp] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long acc = 0;
        for (int w = 0; w < ST / 32; w++) { unsigned long long t = s[w]; s[w] = acc; acc += t; }
    }
    __syncthreads();
    const unsigned long long off = bsum[blockIdx.x] + s[warp] + x - len;
    if (q < R) {
        out_off[q] = off;
        out_sup[q] = rec_sup[r];
        const unsigned long long src = rec_off[r];
        for (unsigned long long z = 0; z < len; z++) out_items[off + z] = items[src + z];
        if (q == R - 1) out_off[R] = total_items;
    }
}

int bits_for(int m) {
    int b = 1;
    while ((1LL << b) < (long long)m) b++;
    return b;
}

}  // namespace

int launch_compact(fim_ctx *ctx, uint64_t R, uint64_t R_valid, int n_db, int m_max, bool identity_items) {
    cudaStream_t st = ctx->stream;
    const int db_bits = n_db > 1 ? bits_for(n_db) : 0;
    // items of the itemsets (the record pool's holes excluded)
    const unsigned long long total_items = ctx->host_ctr.n_rec_items - ctx->host_ctr.item_holes;
    FIM_TRY(fim_reserve(ctx, ctx->out_off, sizeof(unsigned long long) * (R + 1)));
    FIM_TRY(fim_reserve(ctx, ctx->out_items, sizeof(uint32_t) * (total_items ? total_items : 1)));
    FIM_TRY(fim_reserve(ctx, ctx->out_sup, sizeof(uint32_t) * (R ? R : 1)));
    ctx->out_sets = R_valid;  // the holes sort after every itemset: emitted last, never fetched
    ctx->out_items_total = total_items;
    ctx->compact_waits = false;  // until a sort with look-backs is queued
    if (R == 0) {
        FIM_CUDA_TRY(cudaMemsetAsync(ctx->out_off.p, 0, sizeof(unsigned long long), st));
        return FIM_OK;
    }
    const int lmax = ctx->host_ctr.max_len;  // longest set (the host folds in 1- and 2-sets)
    const int bits = bits_for(m_max);
    const int total_bits = db_bits + 8 + bits * lmax;
    const int kw = (int)ceil_div64(total_bits, 64);
    if (n_db == 1 && R <= OC_MAX && kw <= OC_KW && ctx->compact_cluster) {
        FIM_CUDA_TRY(cudaFuncSetAttribute(one_cta_compact_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)oc_smem(OC_KW)));
        ctx->launches++;
        one_cta_compact_kernel<<<1, OC_T, oc_smem(kw), st>>>(
            (int)R, (int)R_valid, ctx->rec_off.as<unsigned long long>(), ctx->rec_len.as<uint32_t>(),
            ctx->rec_sup.as<uint32_t>(), ctx->rec_items.as<uint32_t>(),
            identity_items ? nullptr : ctx->perm.as<int32_t>(), bits, kw, ctx->out_off.as<unsigned long long>(),
            ctx->out_items.as<uint32_t>(), ctx->out_sup.as<uint32_t>(), total_items);
        FIM_CUDA_TRY(cudaGetLastError());
        return FIM_OK;
    }
    FIM_TRY(fim_reserve(ctx, ctx->keys, sizeof(unsigned long long) * R * kw));
    FIM_TRY(fim_reserve(ctx, ctx->idx_a, sizeof(uint32_t) * R));
    FIM_TRY(fim_reserve(ctx, ctx->idx_b, sizeof(uint32_t) * R));
    FIM_TRY(fim_reserve(ctx, ctx->kv_a, sizeof(unsigned long long) * R));
    FIM_TRY(fim_reserve(ctx, ctx->kv_b, sizeof(unsigned long long) * R));
    // radix tiles: 512 threads once they still make two waves
    const bool wide = (int64_t)R >= (int64_t)ctx->num_sms * 2 * 512 * RI;
    const int64_t ntiles = ceil_div64((int64_t)R, (wide ? 512 : 256) * RI);
    const int nblk = (int)ceil_div64((int64_t)R, ST);
    FIM_TRY(fim_reserve(ctx, ctx->scan_tmp, sizeof(unsigned long long) * (size_t)nblk));

    unsigned long long *keys = ctx->keys.as<unsigned long long>();
    // the digit passes, least significant first: (word, shift)
    const int key_pad = kw * 64 - total_bits;  // zero bits at the key's LSB end
    std::vector<std::pair<int, int>> passes;
    for (int w = kw - 1; w >= 0; w--) {
        const int word_lo_bit = (kw - 1 - w) * 64;  // bit index (from the key's LSB) of this word's bit 0
        for (int d = 0; d < 8; d++)
            if (word_lo_bit + d * 8 + 8 > key_pad) passes.push_back({w, d * 8});  // skip pure padding
    }
    const size_t hist_bytes = sizeof(unsigned long long) * 256 * (passes.size() + 2 * (size_t)ntiles) +
                              sizeof(uint32_t) * passes.size();
    // a small output is sorted in one cluster launch (keys in distributed
    // shared memory) instead of a launch triple per digit
    int cs_cl = 0, cs_cap = 0, cs_per = 0;
    const bool csort = cluster_sort_plan(ctx, R, kw, &cs_cl, &cs_cap, &cs_per) != 0;
    if (!csort) {
        FIM_TRY(fim_reserve(ctx, ctx->hist, hist_bytes));
        FIM_CUDA_TRY(cudaMemsetAsync(ctx->dev_flag.as<int>() + kCompactErr, 0, sizeof(int), st));
        if (passes.size() > (size_t)RS_MAXPASS / 2)  // more counters than the default shared memory
            FIM_CUDA_TRY(cudaFuncSetAttribute(rs_count_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)(sizeof(uint32_t) * 256 * RS_MAXPASS)));
    }
    ctx->compact_waits = !csort;
    int *const err = csort ? nullptr : ctx->dev_flag.as<int>() + kCompactErr;
    const unsigned long long spin_ns = (unsigned long long)ctx->spin_limit_ms * 1000000ull;
    const unsigned long long wait_ns = spin_ns < RS_WAIT_NS ? spin_ns : RS_WAIT_NS;
    int enq_rc = FIM_OK;  // a launch that enqueue() could not make
    // The whole pass sequence, enqueued on st.  Returns the kernel count.
    auto enqueue = [&]() -> uint64_t {
        uint64_t nk = 0;
        uint32_t *ia = ctx->idx_a.as<uint32_t>(), *ib = ctx->idx_b.as<uint32_t>();
        prep_keys_kernel<<<(unsigned)ceil_div64((int64_t)R, 256), 256, 0, st>>>(
            R, ctx->rec_off.as<unsigned long long>(), ctx->rec_len.as<uint32_t>(),
            ctx->rec_items.as<uint32_t>(), identity_items ? nullptr : ctx->perm.as<int32_t>(), ctx->dbdesc.as<DbDesc>(),
            ctx->rec_db.as<uint32_t>(), db_bits, bits, kw, keys, ia);
        nk++;
        if (csort) {
            enq_rc = launch_cluster_sort(ctx, keys, R, kw, passes, cs_cl, cs_cap, cs_per, ia, st);
            nk++;
        } else {
            // LSD: least significant word first; within a word, low digits first.
            // (word, record) pairs move together, so each word is gathered into
            // record order once; the least significant word starts in record
            // order and is read straight from the key array.
            unsigned long long *ka = ctx->kv_a.as<unsigned long long>(), *kb = ctx->kv_b.as<unsigned long long>();
            const int np = (int)passes.size();
            // hist: [pass][256] counts, then bases; the look-back words, two
            // digits' in turn; the tickets
            unsigned long long *const hist = ctx->hist.as<unsigned long long>();
            unsigned long long *const status = hist + (size_t)np * 256;
            const size_t words = (size_t)ntiles * 256;
            uint32_t *const ticket = reinterpret_cast<uint32_t *>(status + 2 * words);
            cudaMemsetAsync(hist, 0, hist_bytes, st);
            for (int p0 = 0; p0 < np; p0 += RS_MAXPASS) {
                RsPasses ps{};
                ps.n = np - p0 < RS_MAXPASS ? np - p0 : RS_MAXPASS;
                for (int p = 0; p < ps.n; p++) {
                    ps.word[p] = (signed char)passes[p0 + p].first;
                    ps.shift[p] = (signed char)passes[p0 + p].second;
                }
                const int64_t blocks = min64(ceil_div64((int64_t)R, 512), (int64_t)ctx->num_sms * 2);
                rs_count_kernel<<<(unsigned)blocks, 512, sizeof(uint32_t) * 256 * (size_t)ps.n, st>>>(
                    keys, R, ps, hist + (size_t)p0 * 256);
                nk++;
            }
            rs_base_kernel<<<(unsigned)np, 256, 0, st>>>(hist);
            nk++;
            const unsigned long long *kin = nullptr;
            for (int i = 0; i < np; i++) {
                const int w = passes[i].first, shift = passes[i].second;
                if (i == 0) {
                    kin = keys + (size_t)w * R;  // record order: read the key array itself
                } else if (passes[i - 1].first != w) {
                    gather_word_kernel<<<(unsigned)ceil_div64((int64_t)R, 256), 256, 0, st>>>(keys + (size_t)w * R, ia,
                                                                                            R, ka, err);
                    nk++;
                    kin = ka;
                }
                unsigned long long *kout = (kin == ka) ? kb : ka;
                (wide ? rs_digit_kernel<512> : rs_digit_kernel<256>)<<<(unsigned)ntiles, wide ? 512 : 256, 0, st>>>(
                    kin, ia, kout, ib, R, shift, hist + (size_t)i * 256, status + (i & 1) * words,
                    status + ((i & 1) ^ 1) * words, ticket + i, err, wait_ns, ctx->test_withhold_tile);
                nk++;
                uint32_t *t = ia; ia = ib; ib = t;
                kin = kout;
            }
        }
        unsigned long long *bsum = ctx->scan_tmp.as<unsigned long long>();
        len_block_sums_kernel<<<nblk, ST, 0, st>>>(ia, ctx->rec_len.as<uint32_t>(), R, bsum, err);
        scan_u64_single_kernel<<<1, 1024, 0, st>>>(bsum, (unsigned long long)nblk);
        emit_sorted_kernel<<<nblk, ST, 0, st>>>(ia, R, ctx->rec_off.as<unsigned long long>(),
                                                ctx->rec_len.as<uint32_t>(), ctx->rec_sup.as<uint32_t>(),
                                                ctx->rec_items.as<uint32_t>(), bsum,
                                                ctx->out_off.as<unsigned long long>(),
                                                ctx->out_items.as<uint32_t>(), ctx->out_sup.as<uint32_t>(),
                                                total_items, err);
        return nk + 3;
    };
    // A shape met a second time (same sizes, same buffers) is captured into a
    // CUDA graph and replayed from then on: the pass sequence is dozens of
    // short launches whose launch latency would otherwise dominate.
    uint64_t key = 1469598103934665603ull;
    auto mix = [&key](uint64_t v) { key = (key ^ v) * 1099511628211ull; };
    mix(R); mix((uint64_t)kw); mix((uint64_t)total_bits); mix((uint64_t)db_bits); mix((uint64_t)bits);
    mix(total_items); mix((uint64_t)(uintptr_t)keys); mix((uint64_t)(uintptr_t)ctx->idx_a.p);
    mix((uint64_t)(uintptr_t)ctx->idx_b.p); mix((uint64_t)(uintptr_t)ctx->hist.p);
    mix((uint64_t)(uintptr_t)ctx->scan_tmp.p); mix((uint64_t)(uintptr_t)ctx->rec_off.p);
    mix((uint64_t)(uintptr_t)ctx->rec_items.p); mix((uint64_t)(uintptr_t)ctx->out_off.p);
    mix((uint64_t)(uintptr_t)ctx->out_items.p); mix(identity_items ? 0ull : (uint64_t)(uintptr_t)ctx->perm.p);
    mix((uint64_t)(uintptr_t)ctx->dbdesc.p); mix((uint64_t)(uintptr_t)ctx->rec_db.p);
    mix((uint64_t)(uintptr_t)ctx->kv_a.p); mix((uint64_t)(uintptr_t)ctx->kv_b.p);
    mix(csort ? (uint64_t)(cs_cl * 100000 + cs_per) : 0ull);
    mix(csort ? 0ull : wait_ns); mix(csort ? 0ull : (uint64_t)(int64_t)ctx->test_withhold_tile);
    for (int i = 0; i < 2; i++)
        if (ctx->compact_graph_exec[i] && ctx->compact_key[i] == key) {
            FIM_CUDA_TRY(cudaGraphLaunch((cudaGraphExec_t)ctx->compact_graph_exec[i], st));
            ctx->launches += ctx->compact_graph_launches[i];
            return FIM_OK;
        }
    if (ctx->compact_seen_key[0] != key && ctx->compact_seen_key[1] != key) {  // first time: launch directly
        ctx->compact_seen_key[ctx->compact_seen_next] = key;
        ctx->compact_seen_next ^= 1;
        ctx->launches += enqueue();
        FIM_TRY(enq_rc);
        FIM_CUDA_TRY(cudaGetLastError());
        return FIM_OK;
    }
    const int slot = ctx->compact_next;
    if (ctx->compact_graph_exec[slot]) {
        cudaGraphExecDestroy((cudaGraphExec_t)ctx->compact_graph_exec[slot]);
        ctx->compact_graph_exec[slot] = nullptr;
        ctx->compact_key[slot] = 0;
    }
    cudaGraph_t g = nullptr;
    FIM_CUDA_TRY(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
    const uint64_t nk = enqueue();
    const cudaError_t ce = cudaStreamEndCapture(st, &g);
    if (ce != cudaSuccess) { fim_set_cuda_error(ce, "compact capture", __FILE__, __LINE__); return FIM_E_CUDA; }
    if (enq_rc != FIM_OK) {
        cudaGraphDestroy(g);
        return enq_rc;
    }
    cudaGraphExec_t ex = nullptr;
    const cudaError_t ie = cudaGraphInstantiate(&ex, g, 0);
    cudaGraphDestroy(g);
    if (ie != cudaSuccess) { fim_set_cuda_error(ie, "compact instantiate", __FILE__, __LINE__); return FIM_E_CUDA; }
    ctx->compact_graph_exec[slot] = ex;
    ctx->compact_key[slot] = key;
    ctx->compact_graph_launches[slot] = nk;
    ctx->compact_next ^= 1;
    FIM_CUDA_TRY(cudaGraphLaunch(ex, st));
    ctx->launches += nk;
    return FIM_OK;
}
