// The ends of the network: im2col of few-channel stems, the 3x3 stride-2 max-pool, and the head (global average pool, linear
// layer, mean softmax cross-entropy and their gradients).  fp32 arithmetic on T = float or bf16 storage; every sum has a fixed order.
#include <algorithm>
#include <cooperative_groups.h>
#include "internal.h"

namespace resist {

template <class T> __device__ __forceinline__ float ldf(const void* p, long long i);
template <> __device__ __forceinline__ float ldf<float>(const void* p, long long i) { return ((const float*)p)[i]; }
template <> __device__ __forceinline__ float ldf<__nv_bfloat16>(const void* p, long long i) { return __bfloat162float(((const __nv_bfloat16*)p)[i]); }
template <class T> __device__ __forceinline__ void stf(void* p, long long i, float v);
template <> __device__ __forceinline__ void stf<float>(void* p, long long i, float v) { ((float*)p)[i] = v; }
template <> __device__ __forceinline__ void stf<__nv_bfloat16>(void* p, long long i, float v) { ((__nv_bfloat16*)p)[i] = __float2bfloat16_rn(v); }
__device__ __forceinline__ void unpack8(const uint4& v, float* f) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) { f[2 * k] = __uint_as_float(w[k] << 16); f[2 * k + 1] = __uint_as_float(w[k] & 0xFFFF0000u); }
}
__device__ __forceinline__ uint4 pack8(const float* f) {
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) { __nv_bfloat162 h = __floats2bfloat162_rn(f[2 * k], f[2 * k + 1]); w[k] = *reinterpret_cast<uint32_t*>(&h); }
    return make_uint4(w[0], w[1], w[2], w[3]);
}
static int ew_grid(long long n) { long long g = (n + 255) / 256; if (g > 148 * 16) g = 148 * 16; if (g < 1) g = 1; return (int)g; }

// ------------------------------------------------------------------------------------------------
// 3x3 stride-2 max-pool (padding 1, padded cells never win; first maximum in row-major window order).  HBM-bound: the winner is
// kept as one byte per output (its tap), and the bf16 path moves 8 channels per thread and access.
// ------------------------------------------------------------------------------------------------
template <class T>
__device__ void maxpool_fwd_scalar(const PoolProb& p) {
    const long long n = (long long)p.N * p.P * p.Q * p.C;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        int c = (int)(i % p.C); long long t = i / p.C; int q = (int)(t % p.Q); t /= p.Q; int pp = (int)(t % p.P); int nn = (int)(t / p.P);
        bool have = false; float best = 0.f; int bi = 0;
        for (int r = 0; r < 3; ++r) { int h = 2 * pp + r - 1; if (h < 0 || h >= p.H) continue;
            for (int s = 0; s < 3; ++s) { int w = 2 * q + s - 1; if (w < 0 || w >= p.W) continue;
                float v = ldf<T>(p.x, (((long long)nn * p.H + h) * p.W + w) * p.C + c);
                if (!have || v > best) { have = true; best = v; bi = r * 3 + s; } } }
        stf<T>(p.y, i, best);
        if (p.arg) p.arg[i] = (uint8_t)bi;
    }
}
template <class T>
__device__ void maxpool_bwd_scalar(const PoolProb& p) {
    const long long n = (long long)p.N * p.H * p.W * p.C;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        int c = (int)(i % p.C); long long t = i / p.C; int w = (int)(t % p.W); t /= p.W; int h = (int)(t % p.H); int nn = (int)(t / p.H);
        float acc = 0.f;
        for (int pp = h / 2; pp <= (h + 1) / 2; ++pp) { if (pp >= p.P) continue;          // windows with 2p-1 <= h <= 2p+1
            for (int q = w / 2; q <= (w + 1) / 2; ++q) { if (q >= p.Q) continue;
                long long o = (((long long)nn * p.P + pp) * p.Q + q) * p.C + c;
                if (p.arg[o] == (h - 2 * pp + 1) * 3 + (w - 2 * q + 1)) acc += ldf<T>(p.dy, o); } }
        stf<T>(p.dx, i, acc);
    }
}
__device__ __forceinline__ bool pool_vec(const PoolProb& p, const void* a, const void* b) {
    return p.C % 8 == 0 && (((uintptr_t)a | (uintptr_t)b) & 15) == 0 && ((uintptr_t)p.arg & 7) == 0 && (long long)p.N * p.H * p.W * (p.C / 8) < (1ll << 31);
}
template <class T>
__global__ void __launch_bounds__(256) maxpool_fwd_kernel(const PoolProb* __restrict__ probs) {
    const PoolProb& p = probs[blockIdx.y];
    if (sizeof(T) != 2 || !pool_vec(p, p.x, p.y)) { maxpool_fwd_scalar<T>(p); return; }
    const int G = p.C >> 3, Q = p.Q, P = p.P, H = p.H, W = p.W;
    const unsigned n = (unsigned)((long long)p.N * P * Q * G);
    const uint4* __restrict__ x = (const uint4*)p.x; uint4* __restrict__ y = (uint4*)p.y; uint2* __restrict__ arg = (uint2*)p.arg;
    for (unsigned i = blockIdx.x * 256u + threadIdx.x; i < n; i += gridDim.x * 256u) {
        unsigned t = i / (unsigned)G; const unsigned g = i - t * G; const unsigned t2 = t / (unsigned)Q; const int q = (int)(t - t2 * Q);
        const unsigned nn = t2 / (unsigned)P; const int pp = (int)(t2 - nn * P);
        uint4 v[9]; bool in[9];                                   // all taps in flight together; a tap outside reads the centre and is ignored
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const int h = 2 * pp + k / 3 - 1, w = 2 * q + k % 3 - 1;
            in[k] = h >= 0 && h < H && w >= 0 && w < W;
            v[k] = __ldg(x + ((long long)(nn * H + (in[k] ? h : 2 * pp)) * W + (in[k] ? w : 2 * q)) * G + g);
        }
        float best[8]; uint32_t bi[8]; bool have = false;
#pragma unroll
        for (int j = 0; j < 8; ++j) { best[j] = 0.f; bi[j] = 0; }
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            if (!in[k]) continue;
            float f[8]; unpack8(v[k], f);
#pragma unroll
            for (int j = 0; j < 8; ++j) if (!have || f[j] > best[j]) { best[j] = f[j]; bi[j] = k; }
            have = true;
        }
        y[i] = pack8(best);
        if (arg) arg[i] = make_uint2(bi[0] | bi[1] << 8 | bi[2] << 16 | bi[3] << 24, bi[4] | bi[5] << 8 | bi[6] << 16 | bi[7] << 24);
    }
}
template <class T>
__global__ void __launch_bounds__(256) maxpool_bwd_kernel(const PoolProb* __restrict__ probs) {
    const PoolProb& p = probs[blockIdx.y];
    if (sizeof(T) != 2 || !pool_vec(p, p.dx, p.dy)) { maxpool_bwd_scalar<T>(p); return; }
    const int G = p.C >> 3, Q = p.Q, P = p.P, H = p.H, W = p.W;
    const unsigned n = (unsigned)((long long)p.N * H * W * G);
    const uint4* __restrict__ dy = (const uint4*)p.dy; uint4* __restrict__ dx = (uint4*)p.dx; const uint2* __restrict__ arg = (const uint2*)p.arg;
    for (unsigned i = blockIdx.x * 256u + threadIdx.x; i < n; i += gridDim.x * 256u) {
        unsigned t = i / (unsigned)G; const unsigned g = i - t * G; const unsigned t2 = t / (unsigned)W; const int w = (int)(t - t2 * W);
        const unsigned nn = t2 / (unsigned)H; const int h = (int)(t2 - nn * H);
        uint4 d[4]; uint2 a[4]; uint32_t tap[4]; bool in[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {                             // an even row (column) lies in one window's row (column), an odd one in two
            const int pp = h / 2 + k / 2, q = w / 2 + k % 2;
            in[k] = (k / 2 == 0 || (h & 1)) && (k % 2 == 0 || (w & 1)) && pp < P && q < Q;
            const long long o = ((long long)(nn * P + (in[k] ? pp : 0)) * Q + (in[k] ? q : 0)) * G + g;
            d[k] = in[k] ? __ldg(dy + o) : make_uint4(0u, 0u, 0u, 0u); a[k] = in[k] ? __ldg(arg + o) : make_uint2(0u, 0u);
            tap[k] = (uint32_t)((h - 2 * pp + 1) * 3 + (w - 2 * q + 1));
        }
        float acc[8] = {};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (!in[k]) continue;
            float f[8]; unpack8(d[k], f);
#pragma unroll
            for (int j = 0; j < 8; ++j) if ((((j < 4 ? a[k].x : a[k].y) >> (8 * (j & 3))) & 255u) == tap[k]) acc[j] += f[j];
        }
        dx[i] = pack8(acc);
    }
}
void launch_maxpool_fwd(const PoolProb* d, int nprob, long long max_elems, bool bf16, cudaStream_t s) {
    if (bf16) maxpool_fwd_kernel<__nv_bfloat16><<<dim3(ew_grid((max_elems + 7) / 8), nprob), 256, 0, s>>>(d);
    else maxpool_fwd_kernel<float><<<dim3(ew_grid(max_elems), nprob), 256, 0, s>>>(d);
}
void launch_maxpool_bwd(const PoolProb* d, int nprob, long long max_elems, bool bf16, cudaStream_t s) {
    if (bf16) maxpool_bwd_kernel<__nv_bfloat16><<<dim3(ew_grid((max_elems + 7) / 8), nprob), 256, 0, s>>>(d);
    else maxpool_bwd_kernel<float><<<dim3(ew_grid(max_elems), nprob), 256, 0, s>>>(d);
}

// ------------------------------------------------------------------------------------------------ head of few classes and channels
// One CTA per sample: average pool, logits, softmax cross-entropy and, in training, the gradient of the pooled features spread
// back over the map.  The last CTA of a problem adds the samples' losses in order.
template <class T>
__global__ void __launch_bounds__(256) head_small_kernel(HeadProb* __restrict__ probs) {
    HeadProb& p = probs[blockIdx.y];
    const int b = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (b >= p.B) return;
    const int C = p.C, HW = p.HW, classes = p.classes;
    __shared__ float part[256], pooled[256], logit[128], dl[128], dp[256];
    __shared__ int last;
    {   // R row lanes per channel, added in order
        const int R = 256 / C, c = tid % C, r = tid / C;
        float s = 0.f;
        if (r < R) {
#pragma unroll 8
            for (int k = r; k < HW; k += R) s += ldf<T>(p.a, ((long long)b * HW + k) * C + c);
        }
        part[tid] = s;
        __syncthreads();
        if (tid < C) {
            float v = 0.f;
            for (int k = 0; k < R; ++k) v += part[k * C + tid];
            v /= (float)HW; pooled[tid] = v; p.pooled[(long long)b * C + tid] = v;
        }
        __syncthreads();
    }
    for (int k = warp; k < classes; k += 8) {
        float s = 0.f;
        for (int c = lane; c < C; c += 32) s = fmaf(p.w[k * C + c], pooled[c], s);
        for (int d = 16; d; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
        if (lane == 0) { s += p.b[k]; logit[k] = s; p.logits[(long long)b * classes + k] = s; if (p.logits_user) p.logits_user[(long long)b * classes + k] = s; }
    }
    __syncthreads();
    if (warp == 0) {
        float mx = -INFINITY; int arg = 0x7fffffff;
        for (int k = lane; k < classes; k += 32) { const float v = logit[k]; if (v > mx) { mx = v; arg = k; } }
        for (int d = 16; d; d >>= 1) {
            const float om = __shfl_xor_sync(0xffffffffu, mx, d); const int oa = __shfl_xor_sync(0xffffffffu, arg, d);
            if (om > mx || (om == mx && oa < arg)) { mx = om; arg = oa; }
        }
        float se = 0.f;
        for (int k = lane; k < classes; k += 32) se += expf(logit[k] - mx);
        for (int d = 16; d; d >>= 1) se += __shfl_xor_sync(0xffffffffu, se, d);
        const float lse = mx + logf(se);
        const int y = p.labels ? p.labels[b] : -1;
        if (p.dlogits)
            for (int k = lane; k < classes; k += 32) {
                const float g = (expf(logit[k] - lse) - (k == y ? 1.f : 0.f)) / (float)p.B;
                dl[k] = g; p.dlogits[(long long)b * classes + k] = g;
            }
        if (lane == 0) { p.sample_loss[b] = y >= 0 ? lse - logit[y] : 0.f; p.sample_loss[p.B + b] = arg == y ? 1.f : 0.f; }
    }
    __syncthreads();
    if (p.da) {
        if (tid < C) {
            float s = 0.f;
            for (int k = 0; k < classes; ++k) s = fmaf(dl[k], p.w[k * C + tid], s);
            dp[tid] = s / (float)HW;
        }
        __syncthreads();
        for (int i = tid; i < HW * C; i += 256) stf<T>(p.da, (long long)b * HW * C + i, dp[i % C]);
    }
    if (tid == 0) { __threadfence(); last = atomicInc(&p.done, (unsigned)p.B - 1u) == (unsigned)p.B - 1u; __threadfence(); }
    __syncthreads();
    if (last && warp == 0) {
        float s = 0.f, hits = 0.f;
        for (int b0 = 0; b0 < p.B; b0 += 32) {                    // 32 samples at a time, added in order
            const float v = b0 + lane < p.B ? __ldcg(p.sample_loss + b0 + lane) : 0.f, h = b0 + lane < p.B ? __ldcg(p.sample_loss + p.B + b0 + lane) : 0.f;
            for (int l = 0; l < 32; ++l) { s += __shfl_sync(0xffffffffu, v, l); hits += __shfl_sync(0xffffffffu, h, l); }
        }
        if (lane == 0) {
            s /= (float)p.B;
            if (p.loss) *p.loss = s;
            if (p.loss_user) *p.loss_user = s;
            if (p.correct) *p.correct = (int)hits;
        }
    }
}

// ------------------------------------------------------------------------------------------------ larger heads
template <class T>
__global__ void __launch_bounds__(256) avgpool_kernel(const HeadProb* __restrict__ probs) {
    const HeadProb& p = probs[blockIdx.y];
    const int C = p.C, HW = p.HW;
    if (sizeof(T) == 2 && C % 8 == 0 && ((uintptr_t)p.a & 15) == 0) {       // 8 channels per thread, eight loads in flight, added in order
        const int G = C >> 3, n = p.B * G;
        const uint4* __restrict__ a = (const uint4*)p.a;
        for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) {
            const int g = i % G, b = i / G;
            const uint4* row = a + (long long)b * HW * G + g;
            float s[8] = {};
            for (int k0 = 0; k0 < HW; k0 += 8) {
                uint4 v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = k0 + u < HW ? __ldg(row + (long long)(k0 + u) * G) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                for (int u = 0; u < 8; ++u) { float f[8]; unpack8(v[u], f);
#pragma unroll
                    for (int j = 0; j < 8; ++j) s[j] += f[j]; }
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) p.pooled[(long long)b * C + g * 8 + j] = s[j] / (float)HW;
        }
        return;
    }
    const int n = p.B * C;
    for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) {
        const int c = i % C, b = i / C;
        float s = 0.f;
#pragma unroll 8
        for (int k = 0; k < HW; ++k) s += ldf<T>(p.a, ((long long)b * HW + k) * C + c);
        p.pooled[i] = s / (float)HW;
    }
}

// The head's three matrix products in fp32 on CUDA cores: tiles of 32 x 64 with a 32-deep slice in shared memory, 4 x 4 results per
// thread, the next slice's loads in flight while one is used; the reduction runs in ascending order.  (One thread or warp per
// result, as before, read both operands from L2 for every result: 220 + 650 us for 4 x 64 samples of 2048 channels and 1000 classes.)
// A slice takes about 1.2 us, most of it the loads' latency, and the logits have few tiles and 64 slices at 2048 channels.  So from 16 slices on a cluster of HEAD_SPLIT
// CTAs shares a tile of logits: each adds its part of the reduction, then each adds its rows of the eight partial tiles, in the order of the parts, out of the others' shared
// memory.  Pooling, logits and loss of 8 x 128 samples and 100 classes 118 -> 68 us, of 50 samples and 1000 classes 109 -> 52, of 16 and 100 98 -> 36.
//   PROD 0: logits[b][k] = pooled[b] . w[k] + bias    1: dw[k][c] = sum_b dlogits[b][k] pooled[b][c], and db    2: dpooled[b][c] = sum_k dlogits[b][k] w[k][c] / HW
template <int PROD, int SPLIT>
__global__ void __launch_bounds__(128) head_gemm_kernel(const HeadProb* __restrict__ probs) {
    static_assert(PROD == 0 || SPLIT == 1, "only the logits' reduction is shared");
    const HeadProb& p = probs[blockIdx.z / SPLIT];
    const int part = blockIdx.z % SPLIT;
    const int C = p.C, classes = p.classes, B = p.B;
    const int M = PROD == 1 ? classes : B, N = PROD == 0 ? classes : C, K = PROD == 0 ? C : PROD == 1 ? B : classes;
    const int m0 = blockIdx.y * 32, n0 = blockIdx.x * 64;
    if (m0 >= M || n0 >= N) return;                               // a cluster leaves as a whole
    const int per = ((K + 31) / 32 + SPLIT - 1) / SPLIT * 32, k_first = part * per, k_end = min(K, k_first + per);
    const float* __restrict__ A = PROD == 0 ? p.pooled : p.dlogits;
    const float* __restrict__ Bm = PROD == 1 ? p.pooled : p.w;
    const int lda = PROD == 0 ? C : classes, ldb = C;
    __shared__ __align__(16) float As[32][36], Bs[32][68];        // [k][m], [k][n]
    const int tid = threadIdx.x, tm = tid >> 4, tn = tid & 15;
    float ra[8], rb[16];
    // a slice's elements of this thread; PROD 1 reads A along m, the others along k; PROD 0 reads B along k, the others along n
    auto load = [&](int k0) {
#pragma unroll
        for (int i = 0; i < 8; ++i) { const int e = tid + i * 128, x = e & 31, y = e >> 5, k = k0 + (PROD == 1 ? y : x), m = m0 + (PROD == 1 ? x : y);
            ra[i] = k < K && m < M ? A[PROD == 1 ? (long long)k * lda + m : (long long)m * lda + k] : 0.f; }
#pragma unroll
        for (int i = 0; i < 16; ++i) { const int e = tid + i * 128, k = k0 + (PROD == 0 ? e & 31 : e >> 6), n = n0 + (PROD == 0 ? e >> 5 : e & 63);
            rb[i] = k < K && n < N ? Bm[PROD == 0 ? (long long)n * ldb + k : (long long)k * ldb + n] : 0.f; }
    };
    float acc[4][4] = {}, bias = 0.f;
    load(k_first);
    for (int k0 = k_first; k0 < k_end; k0 += 32) {
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 8; ++i) { const int e = tid + i * 128; if (PROD == 1) As[e >> 5][e & 31] = ra[i]; else As[e & 31][e >> 5] = ra[i]; }
#pragma unroll
        for (int i = 0; i < 16; ++i) { const int e = tid + i * 128; if (PROD == 0) Bs[e & 31][e >> 5] = rb[i]; else Bs[e >> 6][e & 63] = rb[i]; }
        __syncthreads();
        if (k0 + 32 < k_end) load(k0 + 32);
#pragma unroll 8
        for (int k = 0; k < 32; ++k) {
            const float4 a = *reinterpret_cast<const float4*>(&As[k][tm * 4]), b = *reinterpret_cast<const float4*>(&Bs[k][tn * 4]);
            const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
        }
        if (PROD == 1 && blockIdx.x == 0 && tid < 32)
            for (int k = 0; k < 32; ++k) bias += As[k][tid];
    }
    if (PROD == 1 && blockIdx.x == 0 && tid < 32 && m0 + tid < M) p.db[m0 + tid] = bias;
    auto put = [&](int m, int n, float v) {
        if (m >= M || n >= N) return;
        const long long o = (long long)m * N + n;
        if (PROD == 0) { v += p.b[n]; p.logits[o] = v; if (p.logits_user) p.logits_user[o] = v; }
        else if (PROD == 1) p.dw[o] = v;
        else p.dpooled[o] = v / (float)p.HW;
    };
    if (SPLIT == 1) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) put(m0 + tm * 4 + i, n0 + tn * 4 + j, acc[i][j]);
        return;
    }
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    __syncthreads();
    float* mine = &Bs[0][0];                                      // [32][64]
#pragma unroll
    for (int i = 0; i < 4; ++i) *reinterpret_cast<float4*>(mine + (tm * 4 + i) * 64 + tn * 4) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    cluster.sync();
    constexpr int ROWS = 32 / SPLIT;
    for (int e = tid; e < ROWS * 32; e += 128) {
        const int m = part * ROWS + (e >> 5), n = (e & 31) * 2;
        float2 v[SPLIT];
#pragma unroll
        for (int r = 0; r < SPLIT; ++r) v[r] = *reinterpret_cast<const float2*>(cluster.map_shared_rank(mine, r) + m * 64 + n);
        float2 sum = v[0];
#pragma unroll
        for (int r = 1; r < SPLIT; ++r) { sum.x += v[r].x; sum.y += v[r].y; }
        put(m0 + m, n0 + n, sum.x); put(m0 + m, n0 + n + 1, sum.y);
    }
    cluster.sync();                                               // no CTA leaves while another reads its tile
}
constexpr int HEAD_SPLIT = 8;
// The rule looks at the channels alone, so that a sub-ResNet's results do not depend on how many others share the launch.  (The input gradient, a reduction over the classes
// with a tile per 64 channels, has CTAs enough: 119 -> 124 us for the three backward kernels of 4 x 64 samples and 1000 classes with eight CTAs per tile there too.)
static void launch_head_logits(const HeadProb* d, int nprob, int B, int classes, int C, cudaStream_t s) {
    const dim3 grid((classes + 63) / 64, (B + 31) / 32, nprob);
    if (C < 16 * 32) { head_gemm_kernel<0, 1><<<grid, 128, 0, s>>>(d); return; }
    cudaLaunchConfig_t cfg = {}; cfg.gridDim = dim3(grid.x, grid.y, nprob * HEAD_SPLIT); cfg.blockDim = dim3(128); cfg.stream = s;
    cudaLaunchAttribute at[1]; at[0].id = cudaLaunchAttributeClusterDimension; at[0].val.clusterDim.x = 1; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = HEAD_SPLIT;
    cfg.attrs = at; cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, head_gemm_kernel<0, HEAD_SPLIT>, d);
}
// eight samples per CTA, one warp each; the last CTA of a problem adds the samples' losses in order
__global__ void __launch_bounds__(256) loss_kernel(HeadProb* __restrict__ probs) {
    HeadProb& p = probs[blockIdx.y];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, b = blockIdx.x * 8 + warp;
    const unsigned ctas = (unsigned)(p.B + 7) / 8u;
    if (blockIdx.x >= ctas) return;
    __shared__ int last;
    if (b < p.B) {
        const float* lg = p.logits + (long long)b * p.classes;
        float mx = -INFINITY; int arg = 0x7fffffff;
        for (int k = lane; k < p.classes; k += 32) { float v = lg[k]; if (v > mx) { mx = v; arg = k; } }
        for (int d = 16; d; d >>= 1) {
            float om = __shfl_xor_sync(0xffffffffu, mx, d); int oa = __shfl_xor_sync(0xffffffffu, arg, d);
            if (om > mx || (om == mx && oa < arg)) { mx = om; arg = oa; }
        }
        float se = 0.f;
        for (int k = lane; k < p.classes; k += 32) se += expf(lg[k] - mx);
        for (int d = 16; d; d >>= 1) se += __shfl_xor_sync(0xffffffffu, se, d);
        const float lse = mx + logf(se);
        const int y = p.labels ? p.labels[b] : -1;
        if (p.dlogits)
            for (int k = lane; k < p.classes; k += 32)
                p.dlogits[(long long)b * p.classes + k] = (expf(lg[k] - lse) - (k == y ? 1.f : 0.f)) / (float)p.B;
        if (lane == 0) { p.sample_loss[b] = y >= 0 ? lse - lg[y] : 0.f; p.sample_loss[p.B + b] = arg == y ? 1.f : 0.f; }
    }
    __syncthreads();
    if (threadIdx.x == 0) { __threadfence(); last = atomicInc(&p.done, ctas - 1u) == ctas - 1u; __threadfence(); }
    __syncthreads();
    if (last && warp == 0) {
        float s = 0.f, hits = 0.f;
        for (int b0 = 0; b0 < p.B; b0 += 32) {
            const float v = b0 + lane < p.B ? __ldcg(p.sample_loss + b0 + lane) : 0.f, h = b0 + lane < p.B ? __ldcg(p.sample_loss + p.B + b0 + lane) : 0.f;
            for (int l = 0; l < 32; ++l) { s += __shfl_sync(0xffffffffu, v, l); hits += __shfl_sync(0xffffffffu, h, l); }
        }
        if (lane == 0) {
            s /= (float)p.B;
            if (p.loss) *p.loss = s;
            if (p.loss_user) *p.loss_user = s;
            if (p.correct) *p.correct = (int)hits;
        }
    }
}
template <class T>
__global__ void __launch_bounds__(256) avgpool_bwd_kernel(const HeadProb* __restrict__ probs) {
    const HeadProb& p = probs[blockIdx.y];
    const long long n = (long long)p.B * p.HW * p.C;
    if (sizeof(T) == 2 && p.C % 8 == 0 && (((uintptr_t)p.da | (uintptr_t)p.dpooled) & 15) == 0) {   // 8 channels per thread
        const int G = p.C / 8; const long long nv = n / 8;
        for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < nv; v += (long long)gridDim.x * blockDim.x) {
            const int g = (int)(v % G); const long long b = v / ((long long)p.HW * G);
            const float4 f0 = *reinterpret_cast<const float4*>(p.dpooled + b * p.C + g * 8), f1 = *reinterpret_cast<const float4*>(p.dpooled + b * p.C + g * 8 + 4);
            const float f[8] = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y, f1.z, f1.w};
            reinterpret_cast<uint4*>(p.da)[v] = pack8(f);
        }
        return;
    }
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i % p.C); const long long b = i / ((long long)p.HW * p.C);
        stf<T>(p.da, i, p.dpooled[b * p.C + c]);
    }
}

// All problems of a launch have the network's own head, so max* are every problem's sizes.
int launch_head_fwd(const HeadProb* d, int nprob, int maxB, int maxC, int max_classes, bool bf16, cudaStream_t s) {
    HeadProb* dm = const_cast<HeadProb*>(d);
    if (head_small(maxC, max_classes)) {
        if (bf16) head_small_kernel<__nv_bfloat16><<<dim3(maxB, nprob), 256, 0, s>>>(dm);
        else head_small_kernel<float><<<dim3(maxB, nprob), 256, 0, s>>>(dm);
        return 1;
    }
    if (bf16) avgpool_kernel<__nv_bfloat16><<<dim3(ew_grid((long long)maxB * ((maxC + 7) / 8)), nprob), 256, 0, s>>>(d);
    else avgpool_kernel<float><<<dim3(ew_grid((long long)maxB * maxC), nprob), 256, 0, s>>>(d);
    launch_head_logits(d, nprob, maxB, max_classes, maxC, s);
    loss_kernel<<<dim3((maxB + 7) / 8, nprob), 256, 0, s>>>(dm);
    return 3;
}
int launch_head_bwd(const HeadProb* d, int nprob, int maxB, int maxC, int max_classes, long long max_elems,
                    bool bf16, cudaStream_t s) {
    head_gemm_kernel<1, 1><<<dim3((maxC + 63) / 64, (max_classes + 31) / 32, nprob), 128, 0, s>>>(d);
    if (head_small(maxC, max_classes)) return 1;                  // the forward kernel has made the input gradient
    head_gemm_kernel<2, 1><<<dim3((maxC + 63) / 64, (maxB + 31) / 32, nprob), 128, 0, s>>>(d);
    if (bf16) avgpool_bwd_kernel<__nv_bfloat16><<<dim3(ew_grid((max_elems + 7) / 8), nprob), 256, 0, s>>>(d);
    else avgpool_bwd_kernel<float><<<dim3(ew_grid(max_elems), nprob), 256, 0, s>>>(d);
    return 3;
}

// ------------------------------------------------------------------------------------------------ im2col (few-channel stem)
// dst rows of (tap r, tap s, channel) columns, zero beyond the taps; the weights are packed alike.  The pass is bound by the rows it
// writes (304 bytes per position of a 7x7 stem of 3 channels), so its reads must not cost instructions: a CTA stages the
// zero-padded input rows of a few output rows in shared memory, and a thread keeps ONE group of 8 columns whose offsets sit in
// registers, so an output is eight 2-byte shared loads without a bounds check and one 16-byte store.  (With a bounds-checked global
// load per element: 765 us for 4 x 64 images of 224 x 224 x 3.)
__device__ void pack_stem_weights(const ColProb& p, long long id, long long step) {
    const int G = p.cols >> 3;
    for (; id < (long long)p.K * G; id += step) {
        const int kx = (int)(id / G), g = (int)(id % G);
        __align__(16) __nv_bfloat16 wv[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) { const int j = g * 8 + e; wv[e] = j < p.kk ? ((const __nv_bfloat16*)p.w)[(long long)kx * p.kk + j] : __float2bfloat16(0.f); }
        *reinterpret_cast<uint4*>((__nv_bfloat16*)p.w32 + (long long)kx * p.cols + g * 8) = *reinterpret_cast<const uint4*>(wv);
    }
}
struct ColGeom { int rp, rows_in, margin, pitch; };              // output rows per CTA; input rows staged; elements before column 0; elements per staged row
__host__ __device__ inline ColGeom col_geom(const ColProb& p, int rp) {
    ColGeom g; g.rp = rp; g.rows_in = (rp - 1) * p.stride + p.ksz; g.margin = (p.pad * p.C + 7) / 8 * 8;
    g.pitch = (g.margin + (p.W + p.pad + p.ksz + p.stride) * p.C + 7) / 8 * 8; return g;
}
__global__ void __launch_bounds__(256) im2col_kernel(const ColProb* __restrict__ probs, int rp) {
    const ColProb& p = probs[blockIdx.y];
    extern __shared__ __align__(16) unsigned short rows_s[];
    const ColGeom ge = col_geom(p, rp);
    const int P = p.P, Q = p.Q, H = p.H, W = p.W, C = p.C, cols = p.cols, G = cols >> 3, tid = threadIdx.x, stride = p.stride;
    const int per_img = (P + rp - 1) / rp;
    const int n = blockIdx.x / per_img, p0 = (blockIdx.x - n * per_img) * rp;
    if (n >= p.N) return;
    const int packers = min(8, (int)gridDim.x);                  // a few small images are fewer than eight CTAs
    if ((int)blockIdx.x < packers) pack_stem_weights(p, blockIdx.x * 256 + tid, packers * 256);
    const unsigned short* __restrict__ src = (const unsigned short*)p.src;
    const int WC = W * C, y0 = p0 * stride - p.pad;
    if ((WC & 7) == 0 && ((uintptr_t)src & 15) == 0) {            // rows are whole 16-byte runs
        const int vr = ge.pitch >> 3, m8 = ge.margin >> 3, w8 = WC >> 3;
        for (int i = tid; i < ge.rows_in * vr; i += 256) {
            const int r = i / vr, v = i - r * vr, y = y0 + r, x = v - m8;
            reinterpret_cast<uint4*>(rows_s)[i] = (y >= 0 && y < H && x >= 0 && x < w8) ? __ldg(reinterpret_cast<const uint4*>(src + ((long long)n * H + y) * WC) + x) : make_uint4(0u, 0u, 0u, 0u);
        }
    } else {
        for (int i = tid; i < ge.rows_in * ge.pitch; i += 256) {
            const int r = i / ge.pitch, x = i - r * ge.pitch - ge.margin, y = y0 + r;
            rows_s[i] = (y >= 0 && y < H && x >= 0 && x < WC) ? src[((long long)n * H + y) * WC + x] : (unsigned short)0;
        }
    }
    __syncthreads();
    const int lanes = 256 / G, g = tid % G, pl = tid / G;
    if (pl >= lanes) return;
    int off[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const int j = g * 8 + e, c = j % C, rs = j / C, s = rs % p.ksz, r = rs / p.ksz;
        off[e] = j < p.kk ? r * ge.pitch + ge.margin + (s - p.pad) * C + c : -1;
    }
    const int nrow = min(rp, P - p0), total = nrow * Q;
    uint4* __restrict__ dst = reinterpret_cast<uint4*>((__nv_bfloat16*)p.dst + ((long long)n * P + p0) * Q * cols) + g;
    for (int i = pl; i < total; i += lanes) {
        const int pr = i / Q, q = i - pr * Q, base = pr * stride * ge.pitch + q * stride * C;
        unsigned h[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) h[e] = off[e] >= 0 ? (unsigned)rows_s[base + off[e]] : 0u;
        dst[(long long)i * G] = make_uint4(h[0] | h[1] << 16, h[2] | h[3] << 16, h[4] | h[5] << 16, h[6] | h[7] << 16);
    }
}
// images whose rows do not fit the staging: one thread per (position, 8-column group), every element looked up in global memory
__global__ void __launch_bounds__(256) im2col_direct_kernel(const ColProb* __restrict__ probs) {
    const ColProb& p = probs[blockIdx.y];
    const unsigned short* __restrict__ src = (const unsigned short*)p.src;
    const int cols = p.cols, G = cols >> 3;
    const long long total = (long long)p.N * p.P * p.Q * G;
    pack_stem_weights(p, blockIdx.x * 256 + threadIdx.x, (long long)gridDim.x * 256);
    for (long long id = blockIdx.x * 256ll + threadIdx.x; id < total; id += (long long)gridDim.x * 256) {
        const int g = (int)(id % G); const long long row = id / G;
        const int q = (int)(row % p.Q); const long long t = row / p.Q; const int pr = (int)(t % p.P); const int n = (int)(t / p.P);
        unsigned h[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int j = g * 8 + e, c = j % p.C, rs = j / p.C, y = pr * p.stride + rs / p.ksz - p.pad, x = q * p.stride + rs % p.ksz - p.pad;
            h[e] = j < p.kk && y >= 0 && y < p.H && x >= 0 && x < p.W ? (unsigned)src[(((long long)n * p.H + y) * p.W + x) * p.C + c] : 0u;
        }
        *reinterpret_cast<uint4*>((__nv_bfloat16*)p.dst + row * cols + g * 8) = make_uint4(h[0] | h[1] << 16, h[2] | h[3] << 16, h[4] | h[5] << 16, h[6] | h[7] << 16);
    }
}
// shape: the problems' common geometry.  A CTA takes as many output rows as give it about 8192 outputs of 16 bytes and fit 48 KB.
void launch_im2col(const ColProb* d, int nprob, const ColProb& shape, cudaStream_t s) {
    const int per_row = std::max(1, shape.Q * (shape.cols / 8));
    int rp = std::max(1, std::min(shape.P, 8192 / per_row));
    auto bytes = [&](int r) { const ColGeom g = col_geom(shape, r); return (size_t)g.rows_in * g.pitch * 2; };
    while (rp > 1 && bytes(rp) > 48 * 1024) --rp;
    if (bytes(rp) > 48 * 1024) {
        const long long gx = std::max(1ll, std::min(((long long)shape.N * shape.P * per_row + 255) / 256, 148ll * 16));
        im2col_direct_kernel<<<dim3((unsigned)gx, nprob), 256, 0, s>>>(d);
        return;
    }
    im2col_kernel<<<dim3((unsigned)(shape.N * ((shape.P + rp - 1) / rp)), nprob), 256, bytes(rp), s>>>(d, rp);
}

}  // namespace resist
