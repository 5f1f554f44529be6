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
//      8-bit digits (per pass a tile histogram with warp-aggregated counts, a
//      scan of the [digit][tile] counts, a stable scatter ranked with
//      __match_any_sync that moves the word with its record index);
//   4. writes offsets (exclusive scan of the sizes), items and supports.
#include <utility>
#include <vector>

#include "fim_common.cuh"

namespace {

constexpr int RT = 256;          // threads per radix tile
constexpr int RI = 8;            // keys per thread per tile
constexpr int TILE = RT * RI;    // 2048

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
    uint32_t *it = items + off;
    if (perm_base) {  // null: the items are already the caller's ids
        const int32_t *perm = perm_base + dbs[db].item_off;
        for (int q = 0; q < len; q++) it[q] = (uint32_t)perm[it[q]];
    }
    for (int q = 1; q < len; q++) {  // insertion sort (sets are short)
        const uint32_t v = it[q];
        int z = q - 1;
        while (z >= 0 && it[z] > v) { it[z + 1] = it[z]; z--; }
        it[z + 1] = v;
    }
    auto emit = [&](int q, unsigned long long v) { keys[(unsigned long long)q * R + r] = v; };
    KeyPack<decltype(emit)> pk(emit);
    if (db_bits) pk.put((unsigned long long)db, db_bits);
    pk.put((unsigned long long)len, 8);
    for (int q = 0; q < len; q++) pk.put(it[q], bits);
    pk.end(kw);
}

// The whole compaction of a small output (one database, at most OC_MAX
// records) in one CTA: keys as above in shared memory, a bitonic sort of
// record numbers by key, a scan of the sizes, the canonical output.  These
// mines return a few hundred sets, and five launches with their gaps took
// 36 us of a 10,000 x 169 mine where this takes 10.  Past OC_MAX records the
// sort's log^2 steps in one CTA cost more than the cluster's launches (1,500
// sets: 10 us slower).
constexpr int OC_T = 512, OC_MAX = 1024, OC_KW = 4, OC_LOCAL = 12;
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
        uint32_t loc[OC_LOCAL];
        uint32_t *const v = len <= OC_LOCAL ? loc : it;
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

__global__ void __launch_bounds__(RT)
rs_hist_kernel(const unsigned long long *__restrict__ key, unsigned long long n, int shift,
               uint32_t *__restrict__ hist, int ntiles) {
    __shared__ uint32_t h[256];
    const int lane = threadIdx.x & 31;
    h[threadIdx.x] = 0;
    __syncthreads();
    const unsigned long long t0 = (unsigned long long)blockIdx.x * TILE;
#pragma unroll
    for (int i = 0; i < RI; i++) {
        const unsigned long long e = t0 + i * RT + threadIdx.x;
        const uint32_t d = e < n ? (uint32_t)((key[e] >> shift) & 255u) : 256u;
        // one shared atomic per distinct digit of the warp: a digit that
        // (nearly) every key shares costs 1/32 of the plain count
        const uint32_t peers = __match_any_sync(0xffffffffu, d);
        if (d < 256u && lane == __ffs(peers) - 1) atomicAdd(&h[d], (uint32_t)__popc(peers));
    }
    __syncthreads();
    hist[(size_t)threadIdx.x * ntiles + blockIdx.x] = h[threadIdx.x];
}

// out[i] = word[idx[i]]: one key word in the records' current order.
__global__ void gather_word_kernel(const unsigned long long *__restrict__ word, const uint32_t *__restrict__ idx,
                                   unsigned long long n, unsigned long long *__restrict__ out) {
    const unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = word[idx[i]];
}

// Three-phase exclusive scan for long arrays: per-chunk sums, a scan of the
// sums in one CTA, and a rescan of every chunk from its base.
constexpr int SC_T = 1024, SC_I = 8, SC_CHUNK = SC_T * SC_I;
__global__ void __launch_bounds__(SC_T)
scan_reduce_kernel(const uint32_t *__restrict__ a, unsigned long long n, uint32_t *__restrict__ part) {
    __shared__ uint32_t s[SC_T / 32];
    const unsigned long long b = (unsigned long long)blockIdx.x * SC_CHUNK;
    uint32_t v = 0;
#pragma unroll
    for (int i = 0; i < SC_I; i++) {
        const unsigned long long e = b + (unsigned long long)i * SC_T + threadIdx.x;
        if (e < n) v += a[e];
    }
    v = warp_sum_u32(v);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        uint32_t t = s[threadIdx.x];
        t = warp_sum_u32(t);
        if (threadIdx.x == 0) part[blockIdx.x] = t;
    }
}

__global__ void __launch_bounds__(SC_T)
scan_apply_kernel(uint32_t *__restrict__ a, unsigned long long n, const uint32_t *__restrict__ part) {
    __shared__ uint32_t s[SC_T / 32 + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // thread t owns elements [b + t*SC_I, b + t*SC_I + SC_I) of the chunk
    const unsigned long long b = (unsigned long long)blockIdx.x * SC_CHUNK + (unsigned long long)threadIdx.x * SC_I;
    uint32_t v[SC_I], sum = 0;
#pragma unroll
    for (int i = 0; i < SC_I; i++) {
        v[i] = b + i < n ? a[b + i] : 0u;
        sum += v[i];
    }
    uint32_t x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s[warp] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t acc = part[blockIdx.x];
        for (int w = 0; w < SC_T / 32; w++) { const uint32_t t = s[w]; s[w] = acc; acc += t; }
    }
    __syncthreads();
    uint32_t run = s[warp] + x - sum;
#pragma unroll
    for (int i = 0; i < SC_I; i++) {
        if (b + i < n) a[b + i] = run;
        run += v[i];
    }
}

// Exclusive scan of a uint32 array (length <= a few million) in one CTA.
__global__ void __launch_bounds__(1024)
scan_single_kernel(uint32_t *__restrict__ a, unsigned long long n, uint32_t *__restrict__ zero,
                   unsigned long long nzero) {
    __shared__ uint32_t s[1024];
    for (unsigned long long i = threadIdx.x; i < nzero; i += 1024) zero[i] = 0u;  // next pass's histogram
    const unsigned long long seg = (n + 1023) / 1024;
    const unsigned long long b = threadIdx.x * seg, e = b + seg < n ? b + seg : n;
    uint32_t sum = 0;
    for (unsigned long long i = b; i < e; i++) sum += a[i];
    s[threadIdx.x] = sum;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
        uint32_t v = threadIdx.x >= (unsigned)o ? s[threadIdx.x - o] : 0;
        __syncthreads();
        s[threadIdx.x] += v;
        __syncthreads();
    }
    uint32_t run = s[threadIdx.x] - sum;
    for (unsigned long long i = b; i < e; i++) {
        const uint32_t v = a[i];
        a[i] = run;
        run += v;
    }
}

__global__ void __launch_bounds__(RT)
rs_scatter_kernel(const unsigned long long *__restrict__ key_in, const uint32_t *__restrict__ idx_in,
                  unsigned long long *__restrict__ key_out, uint32_t *__restrict__ idx_out, unsigned long long n,
                  int shift, const uint32_t *__restrict__ hist, int ntiles, uint32_t *__restrict__ next_hist,
                  int next_shift) {
    __shared__ uint32_t base[256];
    __shared__ uint32_t wc[RT / 32][257];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    base[threadIdx.x] = hist[(size_t)threadIdx.x * ntiles + blockIdx.x];
    const unsigned long long t0 = (unsigned long long)blockIdx.x * TILE;
    for (int i = 0; i < RI; i++) {
        const unsigned long long e = t0 + i * RT + threadIdx.x;
        const bool valid = e < n;
        unsigned long long k = 0;
        uint32_t v = 0, d = 256;
        if (valid) { k = key_in[e]; v = idx_in[e]; d = (uint32_t)((k >> shift) & 255u); }
        for (int q = threadIdx.x; q < (RT / 32) * 257; q += RT) (&wc[0][0])[q] = 0;
        __syncthreads();
        const uint32_t peers = __match_any_sync(0xffffffffu, d);
        const uint32_t rank = __popc(peers & ((1u << lane) - 1u));
        if (valid && rank == 0) wc[warp][d] = __popc(peers);
        __syncthreads();
        uint32_t off = 0;
        if (valid) {
            off = base[d] + rank;
            for (int w = 0; w < warp; w++) off += wc[w][d];
            key_out[off] = k;
            idx_out[off] = v;
        }
        if (next_hist) {
            // the next digit's [digit][tile] count, by destination tile: one
            // atomic per distinct (digit, tile) of the warp
            const uint32_t key2 = valid ? ((uint32_t)((k >> next_shift) & 255u) << 20) | (off / TILE) : 0xFFFFFFFFu;
            const uint32_t peers2 = __match_any_sync(0xffffffffu, key2);
            if (valid && lane == __ffs(peers2) - 1)
                atomicAdd(&next_hist[(size_t)(key2 >> 20) * ntiles + (key2 & 0xFFFFFu)], (uint32_t)__popc(peers2));
        }
        __syncthreads();
        uint32_t add = 0;
        for (int w = 0; w < RT / 32; w++) add += wc[w][threadIdx.x];
        base[threadIdx.x] += add;
        __syncthreads();
    }
}

// Sizes in sorted order, block sums for the offset scan.
constexpr int ST = 1024;
__global__ void __launch_bounds__(ST)
len_block_sums_kernel(const uint32_t *__restrict__ idx, const uint32_t *__restrict__ rec_len,
                      unsigned long long R, unsigned long long *__restrict__ bsum) {
    __shared__ unsigned long long s[ST / 32];
    const unsigned long long q = (unsigned long long)blockIdx.x * ST + threadIdx.x;
    unsigned long long v = q < R ? rec_len[idx[q]] : 0;
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
                   unsigned long long total_items) {
    __shared__ unsigned long long s[ST / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned long long q = (unsigned long long)blockIdx.x * ST + threadIdx.x;
    uint32_t r = 0;
    unsigned long long len = 0;
    if (q < R) { r = idx[q]; len = rec_len[r]; }
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
    const int ntiles = (int)ceil_div64((int64_t)R, TILE);
    const unsigned long long nhist = 256ull * (unsigned long long)ntiles;
    const int nchunks = (int)ceil_div64((int64_t)nhist, SC_CHUNK);
    // small sorts (one-CTA scans) fold each digit's histogram into the
    // previous digit's scatter: two histogram buffers, used in turn
    const bool fuse = nchunks <= 1;
    FIM_TRY(fim_reserve(ctx, ctx->hist, sizeof(uint32_t) * nhist * (fuse ? 2 : 1)));
    FIM_TRY(fim_reserve(ctx, ctx->scan_part, sizeof(uint32_t) * (size_t)nchunks));
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
    // a small output is sorted in one cluster launch (keys in distributed
    // shared memory) instead of a launch triple per digit
    int cs_cl = 0, cs_cap = 0, cs_per = 0;
    const bool csort = cluster_sort_plan(ctx, R, kw, &cs_cl, &cs_cap, &cs_per) != 0;
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
        uint32_t *hist = ctx->hist.as<uint32_t>();
        uint32_t *hist_nxt = fuse ? hist + nhist : nullptr;
        const unsigned long long *kin = nullptr;
        for (size_t i = 0; i < passes.size(); i++) {
            const int w = passes[i].first, shift = passes[i].second;
            const bool new_word = i == 0 || passes[i - 1].first != w;
            if (new_word) {
                if (i == 0) {
                    kin = keys + (size_t)w * R;  // record order: read the key array itself
                } else {
                    gather_word_kernel<<<(unsigned)ceil_div64((int64_t)R, 256), 256, 0, st>>>(
                        keys + (size_t)w * R, ia, R, ka);
                    nk++;
                    kin = ka;
                }
            }
            const bool next_fused = fuse && i + 1 < passes.size() && passes[i + 1].first == w;
            if (new_word || !fuse) {
                rs_hist_kernel<<<ntiles, RT, 0, st>>>(kin, R, shift, hist, ntiles);
                nk++;
            }  // else: the previous scatter has counted this digit into hist
            if (nchunks <= 1) {
                scan_single_kernel<<<1, 1024, 0, st>>>(hist, nhist, next_fused ? hist_nxt : nullptr,
                                                       next_fused ? nhist : 0ull);
                nk += 1;
            } else {
                uint32_t *part = ctx->scan_part.as<uint32_t>();
                scan_reduce_kernel<<<nchunks, SC_T, 0, st>>>(hist, nhist, part);
                scan_single_kernel<<<1, 1024, 0, st>>>(part, (unsigned long long)nchunks, nullptr, 0ull);
                scan_apply_kernel<<<nchunks, SC_T, 0, st>>>(hist, nhist, part);
                nk += 3;
            }
            unsigned long long *kout = (kin == ka) ? kb : ka;
            rs_scatter_kernel<<<ntiles, RT, 0, st>>>(kin, ia, kout, ib, R, shift, hist, ntiles,
                                                     next_fused ? hist_nxt : nullptr,
                                                     next_fused ? passes[i + 1].second : 0);
            nk++;
            uint32_t *t = ia; ia = ib; ib = t;
            kin = kout;
            if (fuse) { uint32_t *h = hist; hist = hist_nxt; hist_nxt = h; }
        }
        }
        unsigned long long *bsum = ctx->scan_tmp.as<unsigned long long>();
        len_block_sums_kernel<<<nblk, ST, 0, st>>>(ia, ctx->rec_len.as<uint32_t>(), R, bsum);
        scan_u64_single_kernel<<<1, 1024, 0, st>>>(bsum, (unsigned long long)nblk);
        emit_sorted_kernel<<<nblk, ST, 0, st>>>(ia, R, ctx->rec_off.as<unsigned long long>(),
                                                ctx->rec_len.as<uint32_t>(), ctx->rec_sup.as<uint32_t>(),
                                                ctx->rec_items.as<uint32_t>(), bsum,
                                                ctx->out_off.as<unsigned long long>(),
                                                ctx->out_items.as<uint32_t>(), ctx->out_sup.as<uint32_t>(),
                                                total_items);
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
    mix((uint64_t)(uintptr_t)ctx->scan_part.p);
    mix(csort ? (uint64_t)(cs_cl * 100000 + cs_per) : 0ull);
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
