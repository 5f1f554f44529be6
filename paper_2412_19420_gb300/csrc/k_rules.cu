// k_rules.cu -- association rules from the frequent itemsets: a post-pass over
// the canonical output of the extraction (Eq. 3), for the confidence and lift
// measures the paper names beside support (Section IV.A).
//
// For every frequent Z with 2 <= |Z| <= max_len and every nonempty proper
// subset X of Z (Y = Z \ X), the rule X -> Y has
//     conf = S(Z) / S(X),     lift = S(Z) n / (S(X) S(Y)),
// and is kept when S(Z) * 10^6 >= min_conf_ppm * S(X) (exact integers).
//
// Work layout.  The candidate rules of all sets form one flat space of
// E = sum_Z (2^|Z| - 2) evaluations in (set index, antecedent mask) order, so
// a set of 11 items spreads its 2,046 antecedents over 2,046 threads instead
// of serialising them in one warp.  The output is ordered by size, so the sets
// of one size are a range [first[l], first[l + 1]) and evaluation e names its
// set and mask by a division.
//   1. hash: every set's key, index and support in an open-addressing table,
//      half full at most, and the first set of every size;
//   2. the host reads those, which give the first evaluation of every size
//      and E;
//   3. keep: one thread per evaluation looks S(X) and S(Y) up in the table
//      (every subset of a frequent set is frequent: downward closure), decides
//      the threshold; a CTA of EV evaluations stores its keep words and their
//      sum;
//   4. scan of the CTAs' sums;
//   5. write: the kept evaluations write (set index, mask, conf, lift) at their
//      slot, so the output keeps evaluation order; the keep pass leaves them
//      the two supports (8 bytes a candidate, up to 2^27 candidates; beyond
//      that the write pass repeats the lookups).
// The keep pass is bound by its random loads and the work of naming sets.  So
// a set whose items fit 127 bits at the width of the largest id is its own key
// and a lookup is one 32-byte sector; longer sets have a 127-bit hash and
// compare items.
// Measured on 35,000 sets with 717,000 candidates (a GB300): keep 22 us, from 68
// with binary searches for the set and both subsets and each S(Y) looked up
// again; write 14, from 31; table 8, scan 4 against 45 of two three-launch
// scans; fim_rules with its fetch 192 us, from 357.
#include "fim_common.cuh"

namespace {

constexpr int RMAX = FIM_RULES_MAX_LEN;
constexpr int RT = 512;                    // threads per CTA of the evaluation kernels
constexpr int EV = 1024;                   // evaluations per CTA
constexpr int NSIZE = 32;                  // size table entries (sizes 0 .. 31)
constexpr unsigned long long kRulesAhead = 1ull << 22;   // candidates whose output room is set aside (117 MB)
constexpr unsigned long long kRuleSupsMax = 1ull << 27;  // candidates whose lookups are kept (1 GB)

// First set and first evaluation of every size (entry l: sets of at least l
// items; those longer than NSIZE - 1 have no rules).
struct SizeTable {
    unsigned long long first[NSIZE], eval[NSIZE];
};

// A set in the table, one 32-byte sector.  Key: its items at `bits` bits each,
// plus one so that no digit is 0, where that fits 127 bits; else the top bit
// and a hash.
struct __align__(32) HashEntry {
    unsigned long long lo, hi;
    uint32_t set, sup, unused[2];
};
struct Key {
    unsigned long long lo, hi;
};
constexpr uint32_t EMPTY = 0xFFFFFFFFu;

struct SetsView {
    const unsigned long long *off;         // [R + 1]
    const uint32_t *items;
    const uint32_t *sup;                   // [R]
    const HashEntry *hash;                 // [mask + 1]
    uint32_t mask, bits;
};

// Key of the items picked by pick, out of L at zp.  All lanes of a set load the
// same items, whatever their masks: broadcasts, and none waits for another.
__device__ __forceinline__ Key key_of(const uint32_t *zp, int L, uint32_t pick, uint32_t bits) {
    if ((uint32_t)__popc(pick) * bits <= 127u) {
        Key k{0, 0};
        uint32_t over = 0;
#pragma unroll 4
        for (int j = 0; j < L; j++) {
            const uint32_t it = __ldg(zp + j) + 1u;  // (0 for the largest 32-bit id: over)
            if ((pick >> j) & 1u) {
                over |= (uint32_t)(it == 0u) | (bits < 32u ? it >> bits : 0u);
                k.hi = k.hi << bits | k.lo >> (64u - bits);
                k.lo = k.lo << bits | it;
            }
        }
        if (!over) return k;
    }
    unsigned long long a = 0, b = 0;
    for (uint32_t mm = pick; mm; mm &= mm - 1) {
        const uint32_t it = __ldg(zp + (__ffs(mm) - 1));
        a = (a ^ it) * 0x9E3779B97F4A7C15ull;
        a ^= a >> 29;
        b = (b + a) * 0xC2B2AE3D27D4EB4Full;
    }
    return Key{a, b | 1ull << 63};
}

// First slot of a key and the odd step to its next ones (single steps make
// clusters: 20 probes for the worst of 35,000 keys, and its warp is waited for).
__device__ __forceinline__ uint32_t slot_of(Key k, uint32_t *step) {
    unsigned long long h = (k.lo ^ k.hi * 0xC2B2AE3D27D4EB4Full) * 0x9E3779B97F4A7C15ull;
    h = (h ^ h >> 32) * 0xC2B2AE3D27D4EB4Full;
    *step = (uint32_t)h | 1u;
    return (uint32_t)(h >> 32);
}

// The sets differ, so each takes the first free entry of its slots.  Set
// sizes do not decrease along the canonical order: first[l] is the first set of
// at least l items (R if none).
__global__ void __launch_bounds__(RT)
hash_sets_kernel(const unsigned long long *__restrict__ off, const uint32_t *__restrict__ items,
                 const uint32_t *__restrict__ sup, int64_t R, int max_len, HashEntry *__restrict__ hash,
                 uint32_t mask, uint32_t bits, unsigned long long *__restrict__ first) {
    for (int64_t z = (int64_t)blockIdx.x * RT + threadIdx.x; z < R; z += (int64_t)gridDim.x * RT) {
        const unsigned long long o = off[z], o1 = off[z + 1];
        const unsigned long long before = z ? o - off[z - 1] : 0ull, len = o1 - o;
        if (z == 0) first[0] = 0;
        for (unsigned long long l = before + 1; l <= len && l < NSIZE; l++) first[l] = (unsigned long long)z;
        if (z == R - 1)
            for (unsigned long long l = len + 1; l < NSIZE; l++) first[l] = (unsigned long long)R;
        if (len >= (unsigned long long)max_len) continue;  // never a proper subset of a set with rules
        const int L = (int)len;
        const Key key = key_of(items + o, L, (1u << L) - 1u, bits);
        uint32_t step, at = slot_of(key, &step) & mask;
        while (atomicCAS(&hash[at].set, EMPTY, (uint32_t)z) != EMPTY) at = (at + step) & mask;
        hash[at].lo = key.lo;
        hash[at].hi = key.hi;
        hash[at].sup = sup[z];
    }
}

// Support of the subset of z (L items at zp, ascending) picked by pick.  A
// missing subset (not a mine's output) sets *err; a support of 0 is a support.
__device__ __forceinline__ uint32_t find_subset(const SetsView &v, const uint32_t *zp, int L, uint32_t pick, int *err) {
    const Key key = key_of(zp, L, pick, v.bits);
    uint32_t step;
    for (uint32_t at = slot_of(key, &step) & v.mask;; at = (at + step) & v.mask) {
        const ulonglong2 k = __ldg(reinterpret_cast<const ulonglong2 *>(v.hash + at));
        const uint2 x = __ldg(reinterpret_cast<const uint2 *>(v.hash + at) + 2);
        if (x.x == EMPTY) {
            atomicExch(err, 1);
            return 0;
        }
        if (k.x != key.lo || k.y != key.hi) continue;
        if (!(key.hi >> 63)) return x.y;
        const unsigned long long o = __ldg(v.off + x.x);
        if ((int)(__ldg(v.off + x.x + 1) - o) != __popc(pick)) continue;
        const uint32_t *it = v.items + o;
        bool same = true;
        for (uint32_t mm = pick; mm && same; mm &= mm - 1) same = __ldg(it++) == __ldg(zp + (__ffs(mm) - 1));
        if (same) return x.y;
    }
}

struct Eval {
    int64_t z;
    uint32_t mask;
    uint64_t sz, sx, sy;
};

// The subsets' supports of a kept candidate, carried from the keep pass to the
// write pass when the scratch fits.
struct RuleSups {
    uint32_t x, y;
};

// The set and mask of evaluation e < E, and the set's size; *len comes in as a
// size that it is not below.
__device__ __forceinline__ int64_t set_of_eval(const SizeTable &t, unsigned long long e, uint32_t *mask, int *len) {
    int l = *len;
    while (l + 1 < NSIZE && t.eval[l + 1] <= e) l++;
    *len = l;
    const unsigned long long d = e - t.eval[l];
    const uint32_t per = (1u << l) - 2u;
    const unsigned long long z = d >> 32 ? d / per : (unsigned long long)((uint32_t)d / per);
    *mask = (uint32_t)(d - z * per) + 1u;
    return (int64_t)(t.first[l] + z);
}

__device__ __forceinline__ Eval evaluate(const SetsView &v, const SizeTable &t, unsigned long long e, int len, int *err) {
    Eval r;
    r.z = set_of_eval(t, e, &r.mask, &len);
    const uint32_t *zp = v.items + v.off[r.z];
    r.sx = find_subset(v, zp, len, r.mask, err);
    r.sy = find_subset(v, zp, len, ((1u << len) - 1u) - r.mask, err);
    r.sz = v.sup[r.z];
    return r;
}

// (double)a / (double)b, correctly rounded, in integers: the FP64 pipe issues
// a warp instruction every 16 cycles, and two conversions and a division of
// each rule's two ratios held the write pass to 31 us for 665,000 rules (now
// 14).  a, b > 0 (a zero, which merged sets can bring, takes the FP64 division:
// 0, infinity or NaN) are rounded to 53 bits (as the conversions do) and normalised
// to A, B in [2^52, 2^53); then
// long division with two digits of 28 bits, each the top 32 bits of the rest
// times a 32-bit reciprocal of B's top bits (an FP32 reciprocal and one Newton
// step, lowered so that no digit is too large), and the rest decides the
// rounding (to nearest, ties to even).
__device__ __forceinline__ unsigned long long round53(unsigned long long x) {
    const int s = 11 - __clzll((long long)x);
    if (s <= 0) return x;
    const unsigned long long half = 1ull << (s - 1), rest = x & (2ull * half - 1ull);
    x >>= s;
    x += (rest > half || (rest == half && (x & 1ull))) ? 1ull : 0ull;
    return x << s;  // (2^64 cannot arise: products of two 32-bit supports)
}

__device__ __forceinline__ double ratio(unsigned long long a, unsigned long long b) {
    if (a == 0 || b == 0) return (double)a / (double)b;
    a = round53(a);
    b = round53(b);
    const int la = __clzll((long long)a), lb = __clzll((long long)b);
    const unsigned long long B = (b << lb) >> 11;
    unsigned long long r = (a << la) >> 11, Q = 0;
    const uint32_t top = (uint32_t)(B >> 21);  // [2^31, 2^32)
    const float f = __frcp_rn(__uint2float_rn(top)) * 9223372036854775808.0f;
    const uint32_t x = f >= 4294967040.0f ? 4294967040u : __float2uint_rz(f);
    const long long err = (long long)((1ull << 63) - (unsigned long long)x * top);
    const long long y = (long long)x + (((long long)x * (err >> 12)) >> 51) - 3;
    const uint32_t rcp = y > 0xFFFFFFFFll ? 0xFFFFFFFFu : (uint32_t)y;  // a little under 2^63 / top
#pragma unroll
    for (int i = 0; i < 2; i++) {
        const uint32_t q = (uint32_t)(((unsigned long long)(uint32_t)(r >> 22) * rcp) >> 34);
        r = (r << 28) - (unsigned long long)q * B;
        Q = (Q << 28) + q;
    }
    while (r >= B) {  // once, rarely
        r -= B;
        Q++;
    }
    const int lz = __clzll((long long)Q);  // Q = floor(2^56 A / B) in (2^55, 2^57)
    Q <<= lz;
    const uint32_t low = (uint32_t)Q & 2047u;
    unsigned long long m = Q >> 11;
    m += (low > 1024u || (low == 1024u && (r || (m & 1ull)))) ? 1ull : 0ull;
    return __longlong_as_double((long long)(((unsigned long long)(long long)(lb - la + 1029 - lz) << 52) + m));
}

// Exclusive scan in one CTA of part[0 .. np), part[np] = total.
__global__ void __launch_bounds__(1024)
scan_part_kernel(unsigned long long *__restrict__ part, unsigned long long np) {
    __shared__ unsigned long long s[1024];
    const unsigned long long seg = (np + 1023) / 1024;
    const unsigned long long b = threadIdx.x * seg, e = b + seg < np ? b + seg : np;
    unsigned long long sum = 0;
    for (unsigned long long i = b; i < e; i++) sum += part[i];
    s[threadIdx.x] = sum;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
        const unsigned long long v = threadIdx.x >= (unsigned)o ? s[threadIdx.x - o] : 0ull;
        __syncthreads();
        s[threadIdx.x] += v;
        __syncthreads();
    }
    unsigned long long run = s[threadIdx.x] - sum;
    for (unsigned long long i = b; i < e; i++) {
        const unsigned long long v = part[i];
        part[i] = run;
        run += v;
    }
    if (threadIdx.x == 1023) part[np] = s[1023];
}

// CTA c owns evaluations [c EV, (c + 1) EV), a keep word per 32 of them.  S(Y)
// is the S(X) of the complementary mask, which is the mirrored evaluation of
// the same set: most often one of the same chunk, so it is looked up once.
__global__ void __launch_bounds__(RT)
rule_keep_kernel(SetsView v, const __grid_constant__ SizeTable sizes, unsigned long long E, uint32_t ppm, uint32_t *__restrict__ keep_bits,
                 RuleSups *__restrict__ sups, unsigned long long *__restrict__ part, int *__restrict__ err) {
    __shared__ SizeTable t;
    __shared__ uint32_t kept, ante[EV];
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < (int)(sizeof(SizeTable) / 8); i += RT)
        reinterpret_cast<unsigned long long *>(&t)[i] = reinterpret_cast<const unsigned long long *>(&sizes)[i];
    const unsigned long long chunks = (E + EV - 1) / EV;
    for (unsigned long long c = blockIdx.x; c < chunks; c += gridDim.x) {
        const unsigned long long e0 = c * EV, e1 = e0 + EV < E ? e0 + EV : E;
        __syncthreads();
        if (threadIdx.x == 0) kept = 0;
        int64_t z[EV / RT];
        uint32_t mask[EV / RT], sx[EV / RT];
        int len[EV / RT], len0 = 2;
        set_of_eval(t, e0, &mask[0], &len0);
#pragma unroll
        for (int q = 0; q < EV / RT; q++) {
            const unsigned long long e = e0 + q * RT + threadIdx.x;
            if (e >= e1) continue;
            len[q] = len0;
            z[q] = set_of_eval(t, e, &mask[q], &len[q]);
            sx[q] = find_subset(v, v.items + v.off[z[q]], len[q], mask[q], err);
            ante[e - e0] = sx[q];
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < EV / RT; q++) {
            const unsigned long long e = e0 + q * RT + threadIdx.x;
            bool keep = false;
            if (e < e1) {
                // masks run from 1 to full - 1 along the set's evaluations
                const uint32_t rest = ((1u << len[q]) - 1u) - mask[q];
                const unsigned long long mirror = e - mask[q] + rest;
                const uint32_t sy = mirror >= e0 && mirror < e1
                                        ? ante[mirror - e0]
                                        : find_subset(v, v.items + v.off[z[q]], len[q], rest, err);
                keep = (uint64_t)v.sup[z[q]] * 1000000ull >= (uint64_t)ppm * sx[q];
                if (keep && sups) sups[e] = RuleSups{sx[q], sy};
            }
            const uint32_t bal = __ballot_sync(0xffffffffu, keep);
            if (lane == 0 && e < e1) {
                keep_bits[e >> 5] = bal;
                if (bal) atomicAdd(&kept, (uint32_t)__popc(bal));
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) part[c] = kept;
    }
}

__global__ void __launch_bounds__(RT)
rule_write_kernel(SetsView v, const __grid_constant__ SizeTable sizes, unsigned long long E, uint64_t n, const uint32_t *__restrict__ keep_bits,
                  const unsigned long long *__restrict__ part, const RuleSups *__restrict__ sups,
                  unsigned long long *__restrict__ set_index, uint32_t *__restrict__ ante_mask,
                  double *__restrict__ conf, double *__restrict__ lift, int *__restrict__ err) {
    constexpr int W = EV / 32;  // keep words of a chunk: one per lane of a warp
    static_assert(W == 32, "a warp scans a chunk's keep words");
    __shared__ SizeTable t;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < (int)(sizeof(SizeTable) / 8); i += RT)
        reinterpret_cast<unsigned long long *>(&t)[i] = reinterpret_cast<const unsigned long long *>(&sizes)[i];
    __syncthreads();
    const uint32_t lt = (1u << lane) - 1u;
    const unsigned long long chunks = (E + EV - 1) / EV, nw = (E + 31) / 32;
    for (unsigned long long c = blockIdx.x; c < chunks; c += gridDim.x) {
        // every warp scans the chunk's words for itself
        const unsigned long long w = c * W + lane;
        const uint32_t bits = w < nw ? keep_bits[w] : 0u;
        uint32_t x = __popc(bits);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        const uint32_t before = x - __popc(bits);
        const unsigned long long base = part[c];
        int len0 = 2;
        uint32_t mask0;
        set_of_eval(t, c * EV, &mask0, &len0);
#pragma unroll
        for (int q = 0; q < EV / RT; q++) {
            const int wi = q * (RT / 32) + warp;
            const uint32_t b = __shfl_sync(0xffffffffu, bits, wi), pre = __shfl_sync(0xffffffffu, before, wi);
            if (!((b >> lane) & 1u)) continue;
            const unsigned long long e = c * EV + (unsigned)wi * 32 + lane;
            int64_t z;
            uint32_t mask;
            uint64_t sz, sx, sy;
            if (sups) {  // the keep pass's lookups
                const RuleSups r = sups[e];
                int len = len0;
                z = set_of_eval(t, e, &mask, &len);
                sz = v.sup[z];
                sx = r.x;
                sy = r.y;
            } else {
                const Eval r = evaluate(v, t, e, len0, err);
                z = r.z;
                mask = r.mask;
                sz = r.sz;
                sx = r.sx;
                sy = r.sy;
            }
            const unsigned long long at = base + pre + __popc(b & lt);
            set_index[at] = (unsigned long long)z;
            ante_mask[at] = mask;
            conf[at] = ratio(sz, sx);
            lift[at] = ratio(sz * n, sx * sy);
        }
    }
}

}  // namespace

extern "C" {

int fim_rules(fim_ctx *ctx, uint32_t min_conf_ppm, int max_len, uint64_t *n_rules) {
    FIM_NVTX("fim_rules");
    if (!ctx || !n_rules || min_conf_ppm > 1000000u) return FIM_E_INVAL;
    if (max_len == 0) max_len = RMAX;
    if (max_len < 2 || max_len > RMAX) return FIM_E_INVAL;
    *n_rules = 0;
    if (!ctx->mined) return FIM_E_STATE;
    int dev_prev = -1;
    cudaGetDevice(&dev_prev);
    if (cudaSetDevice(ctx->device) != cudaSuccess) return FIM_E_CUDA;
    struct Restore { int d; ~Restore() { if (d >= 0) cudaSetDevice(d); } } restore{dev_prev};
    cudaStream_t st = ctx->stream;
    const int64_t R = (int64_t)ctx->out_sets;
    ctx->rules_n = 0;
    ctx->rules_of = 0;
    ctx->rules_evaluated = 0;
    if (R > 0) {
        if (R >= (int64_t)0xFFFFFFFFll) return FIM_E_NOMEM;  // set indices are 32-bit in the table
        uint64_t slots = 1024;
        // half full at most, three quarters from 2^28 slots (8 GB) on
        while (slots < 2ull * (uint64_t)R && slots < (1ull << 28)) slots <<= 1;
        while (3ull * slots < 4ull * (uint64_t)R && slots < (1ull << 32)) slots <<= 1;
        uint32_t bits = 1;
        while (bits < 32 && ((uint64_t)ctx->m >> bits)) bits++;
        FIM_TRY(fim_reserve(ctx, ctx->rule_base, sizeof(unsigned long long) * NSIZE));
        // a fuller table where memory is short, with an entry free for a lookup to end at
        int rc_hash = fim_reserve(ctx, ctx->rule_hash, sizeof(HashEntry) * (size_t)slots);
        while (rc_hash == FIM_E_NOMEM && slots / 2 > (uint64_t)R) {
            slots /= 2;
            rc_hash = fim_reserve(ctx, ctx->rule_hash, sizeof(HashEntry) * (size_t)slots);
        }
        FIM_TRY(rc_hash);
        const SetsView v{ctx->out_off.as<unsigned long long>(), ctx->out_items.as<uint32_t>(),
                         ctx->out_sup.as<uint32_t>(), ctx->rule_hash.as<HashEntry>(),
                         (uint32_t)(slots - 1), bits};
        FIM_CUDA_TRY(cudaMemsetAsync(ctx->rule_hash.p, 0xFF, sizeof(HashEntry) * (size_t)slots, st));
        ctx->launches++;
        const int64_t hb = ceil_div64(R, RT);
        hash_sets_kernel<<<(unsigned)min64(hb, (int64_t)ctx->num_sms * (2048 / RT)), RT, 0, st>>>(
            v.off, v.items, v.sup, R, max_len, ctx->rule_hash.as<HashEntry>(), v.mask, bits,
            ctx->rule_base.as<unsigned long long>());
        FIM_CUDA_TRY(cudaGetLastError());
        // read-backs land in page-locked memory: [0] the compaction's error
        // word, from [1] the first set of every size, then the rules' number
        // and this call's error word
        unsigned long long *const pin = static_cast<unsigned long long *>(ctx->pinned);
        static_assert(sizeof(unsigned long long) * (NSIZE + 1) <= kPinnedBytes, "landing place");
        FIM_CUDA_TRY(cudaMemcpyAsync(pin + 1, ctx->rule_base.p, sizeof(unsigned long long) * NSIZE,
                                     cudaMemcpyDeviceToHost, st));
        FIM_TRY(queue_compact_status(ctx));
        FIM_CUDA_TRY(cudaStreamSynchronize(st));
        FIM_TRY(compact_status(ctx));
        SizeTable sizes;
        unsigned long long E = 0;
        for (int l = 0; l < NSIZE; l++) {
            sizes.first[l] = pin[1 + l];
            sizes.eval[l] = E;
            if (l + 1 < NSIZE && l <= max_len && l >= 2) E += (pin[2 + l] - pin[1 + l]) * ((1ull << l) - 2ull);
        }
        ctx->rules_evaluated = E;
        if (E > 0) {
            const unsigned long long nw = (E + 31) / 32, chunks = (E + EV - 1) / EV;
            FIM_TRY(fim_reserve(ctx, ctx->rule_bits, sizeof(uint32_t) * (size_t)nw));
            FIM_TRY(fim_reserve(ctx, ctx->rule_part, sizeof(unsigned long long) * (size_t)(chunks + 1)));
            uint32_t *keep = ctx->rule_bits.as<uint32_t>();
            unsigned long long *part = ctx->rule_part.as<unsigned long long>();
            int *err = ctx->dev_flag.as<int>() + 2;
            FIM_CUDA_TRY(cudaMemsetAsync(err, 0, sizeof(int), st));
            RuleSups *sups = nullptr;
            if (E <= kRuleSupsMax) {
                FIM_TRY(fim_reserve(ctx, ctx->rule_sets, sizeof(RuleSups) * (size_t)E));
                sups = ctx->rule_sets.as<RuleSups>();
            }
            const unsigned long long cap = (unsigned long long)(ctx->num_sms > 0 ? ctx->num_sms : 1) * (2048 / RT);
            const unsigned grid = (unsigned)(chunks < cap ? chunks : cap);
            ctx->launches += 2;
            rule_keep_kernel<<<grid, RT, 0, st>>>(v, sizes, E, min_conf_ppm, keep, sups, part, err);
            scan_part_kernel<<<1, 1024, 0, st>>>(part, chunks);
            FIM_CUDA_TRY(cudaGetLastError());
            FIM_CUDA_TRY(cudaMemcpyAsync(pin + 1, part + chunks, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
            FIM_CUDA_TRY(cudaMemcpyAsync(pin + 2, err, sizeof(int), cudaMemcpyDeviceToHost, st));
            // where room for all candidates is small the write is queued before
            // the kept number is known
            auto write = [&](unsigned long long cap_rules) -> int {
                FIM_TRY(fim_reserve(ctx, ctx->rule_set, sizeof(unsigned long long) * (size_t)cap_rules));
                FIM_TRY(fim_reserve(ctx, ctx->rule_mask, sizeof(uint32_t) * (size_t)cap_rules));
                FIM_TRY(fim_reserve(ctx, ctx->rule_conf, sizeof(double) * (size_t)cap_rules));
                FIM_TRY(fim_reserve(ctx, ctx->rule_lift, sizeof(double) * (size_t)cap_rules));
                ctx->launches++;
                rule_write_kernel<<<grid, RT, 0, st>>>(v, sizes, E, (uint64_t)ctx->out_n, keep, part, sups,
                                                       ctx->rule_set.as<unsigned long long>(),
                                                       ctx->rule_mask.as<uint32_t>(), ctx->rule_conf.as<double>(),
                                                       ctx->rule_lift.as<double>(), err);
                FIM_CUDA_TRY(cudaGetLastError());
                return FIM_OK;
            };
            bool ahead = E <= kRulesAhead;
            if (ahead) {
                const int rc = write(E);
                if (rc == FIM_E_NOMEM) ahead = false;
                else if (rc != FIM_OK) return rc;
            }
            FIM_CUDA_TRY(cudaStreamSynchronize(st));
            const unsigned long long total = pin[1];
            if (static_cast<const int *>(ctx->pinned)[4]) return FIM_E_STATE;  // the held sets are not downward closed
            if (total && !ahead) FIM_TRY(write(total));
            ctx->rules_n = total;
        }
    }
    ctx->rules_of = ctx->mine_serial;
    if (ctx->bytes_held > ctx->stats.peak_device_bytes) ctx->stats.peak_device_bytes = ctx->bytes_held;
    *n_rules = ctx->rules_n;
    return FIM_OK;
}

int fim_rules_evaluated(const fim_ctx *ctx, uint64_t *n_evaluated) {
    FIM_NVTX("fim_rules_evaluated");
    if (!ctx || !n_evaluated) return FIM_E_INVAL;
    if (!ctx->mined || ctx->rules_of != ctx->mine_serial) return FIM_E_STATE;
    *n_evaluated = ctx->rules_evaluated;
    return FIM_OK;
}

int fim_fetch_rules(fim_ctx *ctx, uint64_t *n_rules, uint64_t *set_index, uint32_t *ante_mask, double *conf,
                    double *lift, uint64_t cap, uint32_t flags) {
    FIM_NVTX("fim_fetch_rules");
    if (!ctx || !n_rules) return FIM_E_INVAL;
    if (!ctx->mined || ctx->rules_of != ctx->mine_serial) return FIM_E_STATE;
    *n_rules = ctx->rules_n;
    if (!set_index && !ante_mask && !conf && !lift) return FIM_OK;
    if (!set_index || !ante_mask || !conf || !lift) return FIM_E_INVAL;
    if (cap < ctx->rules_n) return FIM_E_TOO_SMALL;
    if (ctx->rules_n == 0) return FIM_OK;
    int dev_prev = -1;
    cudaGetDevice(&dev_prev);
    if (cudaSetDevice(ctx->device) != cudaSuccess) return FIM_E_CUDA;
    struct Restore { int d; ~Restore() { if (d >= 0) cudaSetDevice(d); } } restore{dev_prev};
    const cudaMemcpyKind k = (flags & FIM_OUTPUT_DEVICE) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    cudaStream_t st = ctx->stream;
    const size_t nr = (size_t)ctx->rules_n;
    FIM_CUDA_TRY(cudaMemcpyAsync(set_index, ctx->rule_set.p, sizeof(uint64_t) * nr, k, st));
    FIM_CUDA_TRY(cudaMemcpyAsync(ante_mask, ctx->rule_mask.p, sizeof(uint32_t) * nr, k, st));
    FIM_CUDA_TRY(cudaMemcpyAsync(conf, ctx->rule_conf.p, sizeof(double) * nr, k, st));
    FIM_CUDA_TRY(cudaMemcpyAsync(lift, ctx->rule_lift.p, sizeof(double) * nr, k, st));
    FIM_CUDA_TRY(cudaStreamSynchronize(st));
    return FIM_OK;
}

}  // extern "C"
