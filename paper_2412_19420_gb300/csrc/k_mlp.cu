// k_mlp.cu -- the scheduling MLP (8 -> 64 -> 64 -> 2): training kernels,
// inference for the root order, weight loading and trace export.
//
// The paper names choosing the Boolean-operation sequence from data
// characteristics and deep models as directions (Section I; Section V); the
// network itself is this miner's design.  It predicts, per prefix class,
// y0 = log2(1 + subtree candidate words) and y1 = logit(store as diffset).  It
// steers the order in which root classes are handed out and the
// representation a class is counted in; supports are always counted exactly.
//
// Arithmetic modes: bf16 = 0 computes in float32; bf16 = 1 rounds weights,
// inputs and hidden activations to bf16 and accumulates in float32 (the
// inference precision).  Parameter layout: W1[64][8] b1[64] W2[64][64] b2[64]
// W3[2][64] b3[2].  Loss: mean_b 0.5 (y0 - t0)^2 + softplus(y1) - t1 y1.
#include "fim_common.cuh"



namespace {

constexpr int P = FIM_MLP_PARAMS;
constexpr int OFF_B1 = 64 * 8, OFF_W2 = OFF_B1 + 64, OFF_B2 = OFF_W2 + 64 * 64, OFF_W3 = OFF_B2 + 64,
              OFF_B3 = OFF_W3 + 2 * 64;
constexpr int CACHE = 256;  // per sample: z1[64] z2[64] dz1[64] dz2[64]

__device__ __forceinline__ float rb(float x, int bf) { return bf ? __bfloat162float(__float2bfloat16_rn(x)) : x; }

// The forward and backward passes take MS samples a CTA: lane = sample, warp
// = eight of a layer's 64 units, so a weight is read once per warp (a
// broadcast) and 4,096 samples fill 128 CTAs of eight warps.  (One thread per
// sample, with its 64 activations in local memory, left 32 CTAs of four warps
// on long dependent chains: 66 us forward and 85 us backward at 4,096 samples
// against 10 and 8.)  Every sum runs in the order it always did -- a unit's
// inputs ascending, a chunk's samples ascending, chunks ascending -- so the
// results are the same to the bit.
constexpr int MS = 32, MT = 256;
constexpr int W2P = 68;  // pitch of the transposed W2: 16-byte rows, few store conflicts

// Eight consecutive floats of the caller's cache: two 16-byte accesses where
// its rows are 16-byte aligned (a cache that starts on such a boundary).
__device__ __forceinline__ bool cache_vec(const float *cache) { return (reinterpret_cast<uintptr_t>(cache) & 15) == 0; }
__device__ __forceinline__ void put8(float *p, const float *v, bool vec) {
    if (vec) {
        reinterpret_cast<float4 *>(p)[0] = make_float4(v[0], v[1], v[2], v[3]);
        reinterpret_cast<float4 *>(p)[1] = make_float4(v[4], v[5], v[6], v[7]);
    } else {
#pragma unroll
        for (int q = 0; q < 8; q++) p[q] = v[q];
    }
}
__device__ __forceinline__ void get8(const float *p, float *v, bool vec) {
    if (vec) {
        const float4 a = reinterpret_cast<const float4 *>(p)[0], b = reinterpret_cast<const float4 *>(p)[1];
        v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w, v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
    } else {
#pragma unroll
        for (int q = 0; q < 8; q++) v[q] = p[q];
    }
}

__global__ void __launch_bounds__(MT)
mlp_forward_kernel(const float *__restrict__ params, const float *__restrict__ x, int64_t B,
                   float *__restrict__ y, float *__restrict__ cache, int bf) {
    __shared__ __align__(16) float w1[64 * 8], w2t[64 * W2P];
    __shared__ float b1[64], b2[64], w3[2 * 64], b3[2], h[2][64][MS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i0 = warp * 8;
    const int64_t b = (int64_t)blockIdx.x * MS + lane;
    float xi[8];
#pragma unroll
    for (int k = 0; k < 8; k++) xi[k] = b < B ? rb(x[b * 8 + k], bf) : 0.f;
    for (int i = threadIdx.x; i < 64 * 8; i += MT) w1[i] = rb(params[i], bf);
    for (int i = threadIdx.x; i < 64 * 64; i += MT) w2t[(i % 64) * W2P + i / 64] = rb(params[OFF_W2 + i], bf);
    if (threadIdx.x < 64) {
        b1[threadIdx.x] = rb(params[OFF_B1 + threadIdx.x], bf);
        b2[threadIdx.x] = rb(params[OFF_B2 + threadIdx.x], bf);
    } else if (threadIdx.x < 192) {
        w3[threadIdx.x - 64] = rb(params[OFF_W3 + threadIdx.x - 64], bf);
    } else if (threadIdx.x < 194) {
        b3[threadIdx.x - 192] = rb(params[OFF_B3 + threadIdx.x - 192], bf);
    }
    __syncthreads();
    auto put = [&](const float *z, int layer) {  // pre-activations to the cache, activations to shared memory
        if (cache && b < B) put8(cache + b * CACHE + 64 * layer + i0, z, cache_vec(cache));
#pragma unroll
        for (int q = 0; q < 8; q++) h[layer][i0 + q][lane] = rb(fmaxf(z[q], 0.f), bf);
    };
    float a[8];
#pragma unroll
    for (int q = 0; q < 8; q++) {
        a[q] = b1[i0 + q];
#pragma unroll
        for (int k = 0; k < 8; k++) a[q] = fmaf(w1[(i0 + q) * 8 + k], xi[k], a[q]);
    }
    put(a, 0);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 8; q++) a[q] = b2[i0 + q];
#pragma unroll 8
    for (int k = 0; k < 64; k++) {
        const float hk = h[0][k][lane];
        const float4 wa = *reinterpret_cast<const float4 *>(w2t + k * W2P + i0);
        const float4 wb = *reinterpret_cast<const float4 *>(w2t + k * W2P + i0 + 4);
        a[0] = fmaf(wa.x, hk, a[0]);
        a[1] = fmaf(wa.y, hk, a[1]);
        a[2] = fmaf(wa.z, hk, a[2]);
        a[3] = fmaf(wa.w, hk, a[3]);
        a[4] = fmaf(wb.x, hk, a[4]);
        a[5] = fmaf(wb.y, hk, a[5]);
        a[6] = fmaf(wb.z, hk, a[6]);
        a[7] = fmaf(wb.w, hk, a[7]);
    }
    put(a, 1);
    __syncthreads();
    if (warp < 2 && b < B) {  // output `warp` of sample b
        float o = b3[warp];
#pragma unroll 16
        for (int i = 0; i < 64; i++) o = fmaf(w3[warp * 64 + i], h[1][i][lane], o);
        y[b * 2 + warp] = o;
    }
}

// Per sample: dz2 = (W3^T dy) * [z2 > 0], dz1 = (W2^T dz2) * [z1 > 0]; loss
// (one part per 32 samples).
__global__ void __launch_bounds__(MT)
mlp_backward_sample_kernel(const float *__restrict__ params, const float *__restrict__ y,
                           const float *__restrict__ t, float *__restrict__ cache, int64_t B,
                           float *__restrict__ loss_parts, int bf) {
    __shared__ __align__(16) float w2[64 * 64];
    __shared__ float w3[2 * 64], d2[64][MS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i0 = warp * 8;
    const int64_t b = (int64_t)blockIdx.x * MS + lane;
    float *const c = cache + (b < B ? b : B - 1) * CACHE + i0;
    const bool vec = cache_vec(cache);
    float z1[8], z2[8];
    get8(c, z1, vec);
    get8(c + 64, z2, vec);
    float y0 = 0.f, y1 = 0.f, t0 = 0.f, t1 = 0.f;
    if (b < B) {
        y0 = y[b * 2];
        y1 = y[b * 2 + 1];
        t0 = t[b * 2];
        t1 = t[b * 2 + 1];
    }
    for (int i = threadIdx.x; i < 64 * 64; i += MT) w2[i] = rb(params[OFF_W2 + i], bf);
    if (threadIdx.x < 128) w3[threadIdx.x] = rb(params[OFF_W3 + threadIdx.x], bf);
    __syncthreads();
    const float e = y0 - t0;
    const float dy0 = e / (float)B, dy1 = (1.f / (1.f + expf(-y1)) - t1) / (float)B;
    float g[8];
#pragma unroll
    for (int q = 0; q < 8; q++) {
        const float v = w3[i0 + q] * dy0 + w3[64 + i0 + q] * dy1;
        g[q] = z2[q] > 0.f ? v : 0.f;
        d2[i0 + q][lane] = g[q];
    }
    if (b < B) put8(c + 192, g, vec);
    __syncthreads();
    float a[8] = {};
#pragma unroll 8
    for (int i = 0; i < 64; i++) {
        const float d = d2[i][lane];
        const float4 wa = *reinterpret_cast<const float4 *>(w2 + i * 64 + i0);
        const float4 wb = *reinterpret_cast<const float4 *>(w2 + i * 64 + i0 + 4);
        a[0] = fmaf(wa.x, d, a[0]);
        a[1] = fmaf(wa.y, d, a[1]);
        a[2] = fmaf(wa.z, d, a[2]);
        a[3] = fmaf(wa.w, d, a[3]);
        a[4] = fmaf(wb.x, d, a[4]);
        a[5] = fmaf(wb.y, d, a[5]);
        a[6] = fmaf(wb.z, d, a[6]);
        a[7] = fmaf(wb.w, d, a[7]);
    }
#pragma unroll
    for (int q = 0; q < 8; q++) a[q] = z1[q] > 0.f ? a[q] : 0.f;
    if (b < B) put8(c + 128, a, vec);
    if (warp == 0) {
        float l = 0.f;
        if (b < B) l = 0.5f * e * e + fmaxf(y1, 0.f) + log1pf(expf(-fabsf(y1))) - t1 * y1;
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (lane == 0) loss_parts[blockIdx.x] = l;
    }
}

// Partial weight gradients over a chunk of samples: every parameter's gradient
// is a sum over the batch of a product of a cached backward term and a forward
// activation, one thread per parameter (two for W2).  A CTA takes one chunk
// and one group of parameters: eight rows of W2, or W1 and b1, or b2, W3 and
// b3 -- ten groups, so that 16 chunks fill the SMs (all parameters of a chunk
// in one CTA: 75 us at 4,096 samples against 15).
constexpr int GCHUNK = 256, GGROUPS = 10;
__global__ void __launch_bounds__(256)
mlp_grad_partial_kernel(const float *__restrict__ x, const float *__restrict__ y, const float *__restrict__ t,
                        const float *__restrict__ cache, int64_t B, float *__restrict__ part, int bf) {
    // 64 samples at a time: a forward activation row and the backward terms
    __shared__ float act[64][64], dz[64][64], sdy[64][2];
    const int grp = blockIdx.y, tid = threadIdx.x;
    const int64_t b0 = (int64_t)blockIdx.x * GCHUNK;
    const int64_t b1 = min64(B, b0 + GCHUNK);
    float *const out = part + (int64_t)blockIdx.x * P;
    float acc[3] = {};
    for (int64_t s0 = b0; s0 < b1; s0 += 64) {
        const int ns = (int)min64(64, b1 - s0);
        __syncthreads();
        if (grp < 8) {  // dz2 of rows 8 grp .., h1
            for (int i = tid; i < ns * 64; i += 256) act[i / 64][i % 64] = rb(fmaxf(cache[(s0 + i / 64) * CACHE + i % 64], 0.f), bf);
            for (int i = tid; i < ns * 8; i += 256) dz[i / 8][i % 8] = cache[(s0 + i / 8) * CACHE + 192 + grp * 8 + i % 8];
        } else if (grp == 8) {  // dz1, x
            for (int i = tid; i < ns * 64; i += 256) dz[i / 64][i % 64] = cache[(s0 + i / 64) * CACHE + 128 + i % 64];
            for (int i = tid; i < ns * 8; i += 256) act[i / 8][i % 8] = rb(x[(s0 + i / 8) * 8 + i % 8], bf);
        } else {  // dz2, h2 (and dy below)
            for (int i = tid; i < ns * 64; i += 256) {
                act[i / 64][i % 64] = rb(fmaxf(cache[(s0 + i / 64) * CACHE + 64 + i % 64], 0.f), bf);
                dz[i / 64][i % 64] = cache[(s0 + i / 64) * CACHE + 192 + i % 64];
            }
        }
        if (grp == 9 && tid < ns) {
            const int64_t bb = s0 + tid;
            sdy[tid][0] = (y[bb * 2] - t[bb * 2]) / (float)B;
            sdy[tid][1] = (1.f / (1.f + expf(-y[bb * 2 + 1])) - t[bb * 2 + 1]) / (float)B;
        }
        __syncthreads();
        if (grp < 8) {  // W2[i][k] += dz2[i] h1[k], i = 8 grp + tid / 32, k = tid % 32 and + 32
            const int i = tid >> 5, k = tid & 31;
#pragma unroll 8
            for (int r = 0; r < ns; r++) {
                const float d = dz[r][i];
                acc[0] = fmaf(d, act[r][k], acc[0]);
                acc[1] = fmaf(d, act[r][k + 32], acc[1]);
            }
        } else if (grp == 8) {  // W1[i][k] += dz1[i] x[k] (two a thread); b1[i] += dz1[i]
            const int i = tid >> 3, k = tid & 7;
#pragma unroll 8
            for (int r = 0; r < ns; r++) {
                const float xk = act[r][k];
                acc[0] = fmaf(dz[r][i], xk, acc[0]);
                acc[1] = fmaf(dz[r][i + 32], xk, acc[1]);
            }
            if (tid < 64)
#pragma unroll 8
                for (int r = 0; r < ns; r++) acc[2] += dz[r][tid];
        } else if (tid < 64) {  // b2[i] += dz2[i]
            for (int r = 0; r < ns; r++) acc[0] += dz[r][tid];
        } else if (tid < 192) {  // W3[o][k] += dy[o] h2[k]
            const int o = (tid - 64) >> 6, k = tid & 63;
#pragma unroll 8
            for (int r = 0; r < ns; r++) acc[0] = fmaf(sdy[r][o], act[r][k], acc[0]);
        } else if (tid < 194) {  // b3[o] += dy[o]
            for (int r = 0; r < ns; r++) acc[0] += sdy[r][tid - 192];
        }
    }
    if (grp < 8) {
        const int i = grp * 8 + (tid >> 5), k = tid & 31;
        out[OFF_W2 + i * 64 + k] = acc[0];
        out[OFF_W2 + i * 64 + k + 32] = acc[1];
    } else if (grp == 8) {
        const int i = tid >> 3, k = tid & 7;
        out[i * 8 + k] = acc[0];
        out[(i + 32) * 8 + k] = acc[1];
        if (tid < 64) out[OFF_B1 + tid] = acc[2];
    } else if (tid < 64) {
        out[OFF_B2 + tid] = acc[0];
    } else if (tid < 194) {
        out[OFF_W3 + tid - 64] = acc[0];  // W3 and, after its 128, b3
    }
}

// grad[j] = sum over chunks of part[c][j] (fixed order: deterministic).
__global__ void mlp_grad_sum_kernel(const float *__restrict__ part, int nchunks, float *__restrict__ grad,
                                    const float *__restrict__ loss_parts, int nloss, float *__restrict__ loss) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < P) {
        float a = 0.f;
#pragma unroll 8
        for (int c = 0; c < nchunks; c++) a += part[(int64_t)c * P + j];
        grad[j] = a;
    }
    if (j == P) {  // four parts (128 samples) at a time
        float a = 0.f;
        for (int c = 0; c < nloss; c += 4) {
            float p[4];
#pragma unroll
            for (int q = 0; q < 4; q++) p[q] = c + q < nloss ? loss_parts[c + q] : 0.f;
            a += p[0] + p[1] + p[2] + p[3];
        }
        *loss = a;
    }
}

__global__ void mlp_adam_kernel(float *__restrict__ w, const float *__restrict__ g, float *__restrict__ m,
                                float *__restrict__ v, float lr, float b1, float b2, float eps, float c1, float c2) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= P) return;
    const float gj = g[j];
    const float mj = b1 * m[j] + (1.f - b1) * gj;
    const float vj = b2 * v[j] + (1.f - b2) * gj * gj;
    m[j] = mj;
    v[j] = vj;
    w[j] -= lr * (mj / c1) / (sqrtf(vj / c2) + eps);
}

__global__ void to_bf16_kernel(const float *__restrict__ w, __nv_bfloat16 *__restrict__ o) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < P) o[j] = __float2bfloat16_rn(w[j]);
}

// ---- root plan: drop the roots without candidates, order the rest ---------
// A root {a, b} roots the prefix class of the sets whose two smallest items
// are a and b; its candidates are the c > b with {a, c} and {b, c} frequent
// (a row AND of the pair bitsets).  A root without candidates has no subtree,
// so it is dropped before the prefix extension starts: no worker spends a
// task fetch on it.  The others are ordered by a bucket sort on a priority,
// largest first: the scheduling network's predicted subtree work (the bf16
// MLP's y0 on the root class's features, as the DFS computes them), or the
// candidate count, or none (bucket 0: about the pair pass's order).
constexpr int NBUCKET = 256;
constexpr uint8_t DROP = NBUCKET - 1;

struct RootView {
    const uint32_t *pairbits;
    const int *pair_cnt;
    const uint32_t *item_sup;
    const int32_t *perm;
    int64_t n, nw;
    int mf, mpw;
    uint32_t thr;
};

__global__ void __launch_bounds__(256)
root_plan_kernel(const uint32_t *__restrict__ root_a, const uint32_t *__restrict__ root_b,
                 const uint32_t *__restrict__ root_sup, const uint32_t *__restrict__ root_db,
                 const MineCounters *ctr, const RootWindow *win, const DbDesc *__restrict__ dbs, RootView single,
                 int mode, const __nv_bfloat16 *__restrict__ wbf, uint8_t *__restrict__ bucket,
                 uint32_t *__restrict__ hist) {
    __shared__ float w[P];
    __shared__ uint32_t h[NBUCKET];
    if (mode == 2)
        for (int i = threadIdx.x; i < P; i += blockDim.x) w[i] = __bfloat162float(wbf[i]);
    for (int i = threadIdx.x; i < NBUCKET; i += blockDim.x) h[i] = 0;
    __syncthreads();
    const unsigned long long r0 = win ? win->base : 0ull, nr = win ? r0 + win->count : ctr->n_roots;
    for (unsigned long long r = r0 + (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; r < nr;
         r += (unsigned long long)gridDim.x * blockDim.x) {
        RootView v = single;
        if (dbs) {  // a batch: the root's database
            const DbDesc &D = dbs[root_db[r]];
            v.mf = *(volatile const int32_t *)&D.mfreq;
            v.mpw = (v.mf + 31) / 32;
            v.pairbits = single.pairbits + D.pb_off;
            v.pair_cnt = single.pair_cnt + D.pair_off;
            v.item_sup = single.item_sup + D.item_off;
            v.perm = single.perm + D.item_off;
            v.n = D.n;
            v.nw = D.nw;
            v.thr = D.thr;
        }
        const uint32_t a = root_a[r], bb = root_b[r];
        const uint32_t *ra = v.pairbits + (int64_t)a * v.mpw, *rbp = v.pairbits + (int64_t)bb * v.mpw;
        int k = 0;
        float ps = 0.f;
        for (int wd = (int)(bb >> 5); wd < v.mpw; wd++) {
            uint32_t bits = ra[wd] & rbp[wd];
            if (wd == (int)(bb >> 5)) bits &= 0xFFFFFFFEu << (bb & 31);
            k += __popc(bits);
            if (mode == 2)
                while (bits) {
                    const int c = wd * 32 + __ffs(bits) - 1;
                    bits &= bits - 1;
                    ps += (float)v.pair_cnt[(int64_t)a * v.mf + c];
                }
        }
        uint8_t bq = DROP;
        if (k > 0 && mode == 1) {
            bq = (uint8_t)(254 - (k < 254 ? k : 254));  // more candidates first
        } else if (k > 0 && mode == 2) {
            const uint32_t sy = root_sup[r], sx = v.item_sup[v.perm[a]];
            const float fx = sx > 0 ? (float)sx : 1.f, fy = sy > 0 ? (float)sy : 1.f;
            // the DFS kernel's feature vector of the root class (same scaling)
            float x[8] = {2.f / 16.f, log2f(1.f + (float)sy) / 32.f, (float)sy / (float)(v.n > 0 ? v.n : 1),
                          log2f(1.f + (float)k) / 16.f, (float)sy / fx, ps / ((float)k * fx),
                          log2f(1.f + (float)v.nw) / 32.f, (float)v.thr / fy};
            float h1[64];
            for (int i = 0; i < 64; i++) {
                float acc = w[OFF_B1 + i];
                for (int q = 0; q < 8; q++) acc = fmaf(w[i * 8 + q], __bfloat162float(__float2bfloat16_rn(x[q])), acc);
                h1[i] = __bfloat162float(__float2bfloat16_rn(fmaxf(acc, 0.f)));
            }
            float y0 = w[OFF_B3];
            for (int i = 0; i < 64; i++) {
                float acc = w[OFF_B2 + i];
                for (int q = 0; q < 64; q++) acc = fmaf(w[OFF_W2 + i * 64 + q], h1[q], acc);
                y0 = fmaf(w[OFF_W3 + i], __bfloat162float(__float2bfloat16_rn(fmaxf(acc, 0.f))), y0);
            }
            int q = (int)lrintf(4.f * y0);  // predicted log2(1 + subtree words), quarter steps
            q = q < 0 ? 0 : (q > 254 ? 254 : q);
            bq = (uint8_t)(254 - q);  // most predicted work first
        } else if (k > 0) {
            bq = 0;
        }
        bucket[r] = bq;
        atomicAdd(&h[bq], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < NBUCKET; i += blockDim.x)
        if (h[i]) atomicAdd(&hist[i], h[i]);
}

// Exclusive scan of the bucket counts; the dropped roots leave the root
// count (a window's kept count instead) and the pending-task count.
// hist[NBUCKET] keeps the count before.
__global__ void __launch_bounds__(NBUCKET)
root_plan_scan_kernel(uint32_t *hist, MineCounters *ctr, RootWindow *win) {
    // one thread per bucket: a serial walk of the 256 counts took 14 us
    __shared__ uint32_t wsum[NBUCKET / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t v = hist[threadIdx.x];
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    uint32_t before = 0;
    for (int w = 0; w < warp; w++) before += wsum[w];
    hist[threadIdx.x] = before + x - v;
    if (threadIdx.x == DROP) {
        const unsigned long long total = win ? win->count : ctr->n_roots;
        const uint32_t dropped = v;
        hist[NBUCKET] = (uint32_t)total;
        if (win)
            win->kept = total - dropped;
        else
            ctr->n_roots = total - dropped;
        ctr->pending -= (long long)dropped;
    }
}

__global__ void root_plan_scatter_kernel(const uint8_t *__restrict__ bucket, uint32_t *__restrict__ hist,
                                         const RootWindow *win, uint32_t *__restrict__ order) {
    const unsigned long long r0 = win ? win->base : 0ull, nr = r0 + hist[NBUCKET];
    for (unsigned long long r = r0 + (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; r < nr;
         r += (unsigned long long)gridDim.x * blockDim.x)
        if (bucket[r] != DROP) order[r0 + atomicAdd(&hist[bucket[r]], 1u)] = (uint32_t)r;
}

}  // namespace

int reserve_root_plan(fim_ctx *ctx, size_t root_cap) {
    FIM_TRY(fim_reserve(ctx, ctx->root_order, sizeof(uint32_t) * (root_cap ? root_cap : 1)));
    FIM_TRY(fim_reserve(ctx, ctx->root_bucket, root_cap ? root_cap : 1));
    FIM_TRY(fim_reserve(ctx, ctx->root_hist, sizeof(uint32_t) * (NBUCKET + 1)));
    return FIM_OK;
}

// (allocates nothing: it may run inside a stream capture once
// reserve_root_plan has sized the buffers)
int launch_root_plan(fim_ctx *ctx, MineCounters *d_ctr, size_t root_cap, const DbDesc *d_dbs, int mode,
                     RootWindow *win, cudaStream_t st) {
    if (mode == 2 && !ctx->has_weights) return FIM_E_STATE;
    FIM_CUDA_TRY(cudaMemsetAsync(ctx->root_hist.p, 0, sizeof(uint32_t) * (NBUCKET + 1), st));
    const uint32_t *roots = ctx->roots.as<uint32_t>();
    RootView v{};
    v.pairbits = ctx->pairbits.as<uint32_t>();
    v.pair_cnt = ctx->pair_cnt.as<int>();
    v.item_sup = ctx->item_sup.as<uint32_t>();
    v.perm = ctx->perm.as<int32_t>();
    if (!d_dbs) {
        v.mf = ctx->mfreq;
        v.mpw = (int)ceil_div64(v.mf, 32);
        v.n = ctx->n;
        v.nw = ctx->nw;
        v.thr = ctx->cur_thr;
    }
    // the root count is known only on the device: a grid-stride loop over at
    // most the capacity, with a grid of a few CTAs per SM
    int64_t grid = ceil_div64((int64_t)(root_cap ? root_cap : 1), 256);
    const int64_t resident = (int64_t)(ctx->num_sms > 0 ? ctx->num_sms : 1) * 8;
    if (grid > resident) grid = resident;
    ctx->launches += 3;
    root_plan_kernel<<<(unsigned)grid, 256, 0, st>>>(roots, roots + root_cap, roots + 2 * root_cap,
                                           d_dbs ? roots + 3 * root_cap : nullptr, d_ctr, win, d_dbs, v, mode,
                                           ctx->mlp_wbf.as<__nv_bfloat16>(), ctx->root_bucket.as<uint8_t>(),
                                           ctx->root_hist.as<uint32_t>());
    root_plan_scan_kernel<<<1, NBUCKET, 0, st>>>(ctx->root_hist.as<uint32_t>(), d_ctr, win);
    root_plan_scatter_kernel<<<(unsigned)grid, 256, 0, st>>>(ctx->root_bucket.as<uint8_t>(), ctx->root_hist.as<uint32_t>(),
                                                   win, ctx->root_order.as<uint32_t>());
    FIM_CUDA_TRY(cudaGetLastError());
    return FIM_OK;
}

extern "C" {

int fim_sched_load_weights(fim_ctx *ctx, const float *weights, size_t n_params) {
    FIM_NVTX("fim_sched_load_weights");
    if (!ctx || !weights || n_params != (size_t)P) return FIM_E_INVAL;
    FIM_TRY(fim_reserve(ctx, ctx->mlp_w32, sizeof(float) * P));
    FIM_TRY(fim_reserve(ctx, ctx->mlp_wbf, sizeof(__nv_bfloat16) * P));
    FIM_CUDA_TRY(cudaMemcpyAsync(ctx->mlp_w32.p, weights, sizeof(float) * P, cudaMemcpyHostToDevice, ctx->stream));
    ctx->launches++;
    to_bf16_kernel<<<(P + 255) / 256, 256, 0, ctx->stream>>>(ctx->mlp_w32.as<float>(),
                                                              ctx->mlp_wbf.as<__nv_bfloat16>());
    FIM_CUDA_TRY(cudaGetLastError());
    FIM_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
    ctx->has_weights = true;
    return FIM_OK;
}

int fim_fetch_traces(fim_ctx *ctx, uint64_t *n_rows, float *features, float *targets, uint64_t cap) {
    FIM_NVTX("fim_fetch_traces");
    if (!ctx || !n_rows) return FIM_E_INVAL;
    if (!ctx->mined || !(ctx->mflags & FIM_TRACE)) return FIM_E_STATE;
    unsigned long long n = ctx->host_ctr.n_traces;
    if (n > ctx->trace_cap) n = ctx->trace_cap;
    *n_rows = n;
    if (!features && !targets) return FIM_OK;
    if (!features || !targets) return FIM_E_INVAL;
    if (cap < n) return FIM_E_TOO_SMALL;
    if (n) {
        FIM_CUDA_TRY(cudaMemcpyAsync(features, ctx->trace_x.p, sizeof(float) * FIM_MLP_FEATURES * n,
                                     cudaMemcpyDeviceToHost, ctx->stream));
        FIM_CUDA_TRY(cudaMemcpyAsync(targets, ctx->trace_y.p, sizeof(float) * 2 * n, cudaMemcpyDeviceToHost,
                                     ctx->stream));
        FIM_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
    }
    return FIM_OK;
}

int fim_mlp_forward(fim_ctx *ctx, const float *params, const float *x, int64_t B, float *y, float *cache,
                    int bf16) {
    FIM_NVTX("fim_mlp_forward");
    if (!ctx || !params || !x || !y || B < 0) return FIM_E_INVAL;
    if (B == 0) return FIM_OK;
    ctx->launches++;
    mlp_forward_kernel<<<(unsigned)ceil_div64(B, MS), MT, 0, ctx->stream>>>(params, x, B, y, cache, bf16 ? 1 : 0);
    FIM_CUDA_TRY(cudaGetLastError());
    return FIM_OK;
}

int fim_mlp_backward(fim_ctx *ctx, const float *params, const float *x, const float *y, const float *t,
                     const float *cache, int64_t B, float *grad, float *loss_out, int bf16) {
    FIM_NVTX("fim_mlp_backward");
    if (!ctx || !params || !x || !y || !t || !cache || !grad || B <= 0) return FIM_E_INVAL;
    const int nb = (int)ceil_div64(B, MS);
    const int nchunks = (int)ceil_div64(B, GCHUNK);
    FIM_TRY(fim_reserve(ctx, ctx->mlp_scratch, sizeof(float) * ((size_t)nchunks * P + nb + 1)));
    float *part = ctx->mlp_scratch.as<float>();
    float *loss_parts = part + (size_t)nchunks * P;
    float *loss = loss_parts + nb;
    const int bf = bf16 ? 1 : 0;
    ctx->launches += 3;
    mlp_backward_sample_kernel<<<nb, MT, 0, ctx->stream>>>(params, y, t, const_cast<float *>(cache), B, loss_parts, bf);
    mlp_grad_partial_kernel<<<dim3((unsigned)nchunks, GGROUPS), 256, 0, ctx->stream>>>(x, y, t, cache, B, part, bf);
    mlp_grad_sum_kernel<<<(P + 1 + 255) / 256, 256, 0, ctx->stream>>>(part, nchunks, grad, loss_parts, nb, loss);
    FIM_CUDA_TRY(cudaGetLastError());
    if (loss_out) {
        FIM_CUDA_TRY(cudaMemcpyAsync(loss_out, loss, sizeof(float), cudaMemcpyDeviceToHost, ctx->stream));
        FIM_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
        *loss_out /= (float)B;
    }
    return FIM_OK;
}

int fim_mlp_adam(fim_ctx *ctx, float *params, const float *grad, float *m, float *v, int step, float lr,
                 float beta1, float beta2, float eps) {
    FIM_NVTX("fim_mlp_adam");
    if (!ctx || !params || !grad || !m || !v || step < 1) return FIM_E_INVAL;
    const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
    ctx->launches++;
    mlp_adam_kernel<<<(P + 255) / 256, 256, 0, ctx->stream>>>(params, grad, m, v, lr, beta1, beta2, eps, c1, c2);
    FIM_CUDA_TRY(cudaGetLastError());
    return FIM_OK;
}

}  // extern "C"
