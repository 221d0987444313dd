// CUDA-core kernel family: every layer of the sub-ResNet step for storage type T = float or bf16,
// fp32 arithmetic.  It is the whole path of the fp32 mode, and in bf16 mode it runs whatever the
// tensor-core kernels do not take (3-channel stems, odd shapes) and the small head/loss kernels.
// All reductions have a fixed order: results are reproducible run to run.
#include <algorithm>
#include "internal.h"

namespace resist {

template <class T> __device__ __forceinline__ float ldf(const void* p, long long i);
template <> __device__ __forceinline__ float ldf<float>(const void* p, long long i) { return ((const float*)p)[i]; }
template <> __device__ __forceinline__ float ldf<__nv_bfloat16>(const void* p, long long i) {
    return __bfloat162float(((const __nv_bfloat16*)p)[i]);
}
template <class T> __device__ __forceinline__ void stf(void* p, long long i, float v);
template <> __device__ __forceinline__ void stf<float>(void* p, long long i, float v) { ((float*)p)[i] = v; }
template <> __device__ __forceinline__ void stf<__nv_bfloat16>(void* p, long long i, float v) {
    ((__nv_bfloat16*)p)[i] = __float2bfloat16_rn(v);
}

// ------------------------------------------------------------------------------------------------
// Implicit-GEMM convolution on CUDA cores: 64x64 output tile, 16-deep slices, 256 threads, 4x4 per thread.
//   forward: rows = output pixels (n,p,q), cols = output channels, reduction = (r,s,c)
//   dgrad:   rows = input pixels (n,h,w),  cols = input channels,  reduction = (r,s,k)
//   wgrad:   rows = output channels,       cols = (r,s,c),         reduction = output pixels; split over
//            `splits` CTAs along the reduction, partial sums reduced afterwards in a fixed order.
// ------------------------------------------------------------------------------------------------
constexpr int BM = 64, BN = 64, BK = 16;

template <class T, int MODE>
__device__ __forceinline__ float load_a(const ConvProb& p, int row, int kk) {
    if (row >= p.M || kk >= p.Kred) return 0.f;
    if (MODE == CONV_FWD) {
        int q = row % p.Q, t = row / p.Q, pp = t % p.P, n = t / p.P;
        int c = kk % p.C, t2 = kk / p.C, s = t2 % p.ksz, r = t2 / p.ksz;
        int h = pp * p.stride + r - p.pad, x = q * p.stride + s - p.pad;
        if (h < 0 || h >= p.H || x < 0 || x >= p.W) return 0.f;
        return ldf<T>(p.act, (((long long)n * p.H + h) * p.W + x) * p.C + c);
    } else if (MODE == CONV_DGRAD) {
        int x = row % p.W, t = row / p.W, h = t % p.H, n = t / p.H;
        int ko = kk % p.K, t2 = kk / p.K, s = t2 % p.ksz, r = t2 / p.ksz;
        int ph = h + p.pad - r, qx = x + p.pad - s;
        if (ph < 0 || qx < 0 || ph % p.stride || qx % p.stride) return 0.f;
        int pp = ph / p.stride, q = qx / p.stride;
        if (pp >= p.P || q >= p.Q) return 0.f;
        return ldf<T>(p.act, (((long long)n * p.P + pp) * p.Q + q) * p.K + ko);
    } else {   // wgrad: A[ko, t] = dy[t, ko]
        return ldf<T>(p.wgt, (long long)kk * p.K + row);
    }
}
template <class T, int MODE>
__device__ __forceinline__ float load_b(const ConvProb& p, int kk, int col) {
    if (col >= p.Ncol || kk >= p.Kred) return 0.f;
    if (MODE == CONV_FWD) {
        return ldf<T>(p.wgt, (long long)col * p.Kred + kk);
    } else if (MODE == CONV_DGRAD) {
        int ko = kk % p.K, t2 = kk / p.K, s = t2 % p.ksz, r = t2 / p.ksz;
        return ldf<T>(p.wgt, (((long long)ko * p.ksz + r) * p.ksz + s) * p.C + col);
    } else {   // wgrad: B[t, (r,s,c)] = a[n, p*stride+r-pad, q*stride+s-pad, c]
        int q = kk % p.Q, t = kk / p.Q, pp = t % p.P, n = t / p.P;
        int c = col % p.C, t2 = col / p.C, s = t2 % p.ksz, r = t2 / p.ksz;
        int h = pp * p.stride + r - p.pad, x = q * p.stride + s - p.pad;
        if (h < 0 || h >= p.H || x < 0 || x >= p.W) return 0.f;
        return ldf<T>(p.act, (((long long)n * p.H + h) * p.W + x) * p.C + c);
    }
}

template <class T, int MODE>
__global__ void __launch_bounds__(256) conv_ref_kernel(const ConvProb* __restrict__ probs) {
    const ConvProb& p = probs[blockIdx.y];
    const int tiles = p.tiles_m * p.tiles_n;
    int tile = blockIdx.x;
    if (tile >= tiles * p.splits) return;
    const int split = tile / tiles; tile -= split * tiles;
    const int tm = tile / p.tiles_n, tn = tile % p.tiles_n;
    __shared__ float As[BK][BM + 4];
    __shared__ float Bs[BK][BN + 4];
    const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
    float acc[4][4] = {};
    const int kt0 = split * p.ktiles_per_split;
    int kt1 = kt0 + p.ktiles_per_split;
    const int ktiles = (p.Kred + BK - 1) / BK;
    if (kt1 > ktiles) kt1 = ktiles;
    for (int kt = kt0; kt < kt1; ++kt) {
        const int k0 = kt * BK;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            int e = tid + 256 * i;
            if (MODE == CONV_WGRAD) { int r = e % BM, kc = e / BM; As[kc][r] = load_a<T, MODE>(p, tm * BM + r, k0 + kc); }
            else { int kc = e % BK, r = e / BK; As[kc][r] = load_a<T, MODE>(p, tm * BM + r, k0 + kc); }
            if (MODE == CONV_FWD) { int kc = e % BK, c = e / BK; Bs[kc][c] = load_b<T, MODE>(p, k0 + kc, tn * BN + c); }
            else { int c = e % BN, kc = e / BN; Bs[kc][c] = load_b<T, MODE>(p, k0 + kc, tn * BN + c); }
        }
        __syncthreads();
#pragma unroll
        for (int kc = 0; kc < BK; ++kc) {
            float a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) { a[i] = As[kc][ty * 4 + i]; b[i] = Bs[kc][tx * 4 + i]; }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int row = tm * BM + ty * 4 + i;
        if (row >= p.M) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int col = tn * BN + tx * 4 + j;
            if (col >= p.Ncol) continue;
            const long long o = (long long)row * p.Ncol + col;
            if (MODE == CONV_WGRAD) {
                if (p.splits > 1) p.partial[(long long)split * p.M * p.Ncol + o] = acc[i][j];
                else ((float*)p.out)[o] = acc[i][j];
            } else {
                float v = acc[i][j] * p.scale;
                if (p.add) v += ldf<T>(p.add, o);
                stf<T>(p.out, o, v);
            }
        }
    }
}

__global__ void splitk_reduce_kernel(const ConvProb* __restrict__ probs) {
    const ConvProb& p = probs[blockIdx.y];
    if (p.splits <= 1) return;
    const long long n = (long long)p.M * p.Ncol;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        float s = 0.f;
        for (int k = 0; k < p.splits; ++k) s += p.partial[(long long)k * n + i];
        ((float*)p.out)[i] = s;
    }
}

void launch_conv_ref(const ConvProb* d, int nprob, int max_tiles, int mode, bool bf16, cudaStream_t s) {
    dim3 g(max_tiles, nprob);
    if (!bf16) {
        if (mode == CONV_FWD) conv_ref_kernel<float, CONV_FWD><<<g, 256, 0, s>>>(d);
        else if (mode == CONV_DGRAD) conv_ref_kernel<float, CONV_DGRAD><<<g, 256, 0, s>>>(d);
        else conv_ref_kernel<float, CONV_WGRAD><<<g, 256, 0, s>>>(d);
    } else {
        if (mode == CONV_FWD) conv_ref_kernel<__nv_bfloat16, CONV_FWD><<<g, 256, 0, s>>>(d);
        else if (mode == CONV_DGRAD) conv_ref_kernel<__nv_bfloat16, CONV_DGRAD><<<g, 256, 0, s>>>(d);
        else conv_ref_kernel<__nv_bfloat16, CONV_WGRAD><<<g, 256, 0, s>>>(d);
    }
}
void launch_splitk_reduce(const ConvProb* d, int nprob, int max_elems, cudaStream_t s) {
    int gx = (max_elems + 255) / 256; if (gx > 1184) gx = 1184; if (gx < 1) gx = 1;
    splitk_reduce_kernel<<<dim3(gx, nprob), 256, 0, s>>>(d);
}

// ------------------------------------------------------------------------------------------------
// Batch normalisation + ReLU.  Statistics: each CTA reduces `rows_per_chunk` rows of all C channels
// (fp32 per thread, fp64 across threads), a finalise kernel adds the chunk partials in order.
// ------------------------------------------------------------------------------------------------

// ---- bf16 fast path: 16-byte accesses, a thread owns 8 consecutive channels (one group) and every (256/G)-th row
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

template <int MODE>
__device__ void bn_reduce_vec(const BnProb& p) {
    __shared__ float sm[256][17];
    const int C = p.C, G = C >> 3, R = 256 / G;
    const int g = threadIdx.x % G, r = threadIdx.x / G;
    const long long r0 = (long long)blockIdx.x * p.rows_per_chunk;
    long long r1 = r0 + p.rows_per_chunk; if (r1 > p.m) r1 = p.m;
    float s0[8], s1[8], sh[8], mean[8], istd[8], ga[8], be[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) { s0[j] = 0.f; s1[j] = 0.f; }
    if (MODE == 0) { unpack8(*reinterpret_cast<const uint4*>((const __nv_bfloat16*)p.x + g * 8), sh); }
    else {
#pragma unroll
        for (int j = 0; j < 8; ++j) { const int c = g * 8 + j; mean[j] = p.stat[c]; istd[j] = p.stat[C + c]; ga[j] = p.gamma[c]; be[j] = p.beta[c]; }
    }
    const uint4* xv = reinterpret_cast<const uint4*>(p.x);
    const uint4* dv = reinterpret_cast<const uint4*>(p.da);
    // U rows of loads in flight per thread (backward: x and dy, so six rows = twelve 16-byte loads; forward: eight rows); the rows
    // are still added in ascending order
    constexpr int U = MODE == 1 ? 6 : 8;
    for (long long row = r0 + r; row < r1; row += U * R) {
        uint4 xs[U], ds[MODE == 1 ? U : 1];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const long long rr = row + (long long)u * R;
            if (rr < r1) { xs[u] = __ldg(xv + rr * G + g); if (MODE == 1) ds[u] = __ldg(dv + rr * G + g); }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (row + (long long)u * R >= r1) break;
            float x[8]; unpack8(xs[u], x);
            if (MODE == 0) {
#pragma unroll
                for (int j = 0; j < 8; ++j) { const float d = x[j] - sh[j]; s0[j] += d; s1[j] += d * d; }
            } else {
                float d[8]; unpack8(ds[u], d);
#pragma unroll
                for (int j = 0; j < 8; ++j) { const float xh = (x[j] - mean[j]) * istd[j]; const float dz = (xh * ga[j] + be[j] > 0.f) ? d[j] : 0.f; s0[j] += dz; s1[j] += dz * xh; }
            }
        }
    }
    // lanes of a warp that own the same channel group: fixed-order butterfly in fp32
    if (G < 32) {
        for (int off = 16; off >= G; off >>= 1) {
#pragma unroll
            for (int j = 0; j < 8; ++j) { s0[j] += __shfl_down_sync(0xffffffffu, s0[j], off); s1[j] += __shfl_down_sync(0xffffffffu, s1[j], off); }
        }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) { sm[threadIdx.x][j] = s0[j]; sm[threadIdx.x][8 + j] = s1[j]; }
    __syncthreads();
    if ((int)threadIdx.x < C) {
        const int c = threadIdx.x, cg = c >> 3, j = c & 7;
        double a0 = 0.0, a1 = 0.0;
        if (G < 32) { for (int w = 0; w < 8; ++w) { a0 += sm[w * 32 + cg][j]; a1 += sm[w * 32 + cg][8 + j]; } }
        else { for (int k = 0; k < R; ++k) { a0 += sm[cg + G * k][j]; a1 += sm[cg + G * k][8 + j]; } }
        p.partial[((long long)blockIdx.x * 2 + 0) * C + c] = a0;
        p.partial[((long long)blockIdx.x * 2 + 1) * C + c] = a1;
    }
    // more than 256 channels: the remaining ones, 256 at a time
    for (int c = threadIdx.x + 256; c < C; c += 256) {
        const int cg = c >> 3, j = c & 7;
        double a0 = 0.0, a1 = 0.0;
        for (int k = 0; k < R; ++k) { a0 += sm[cg + G * k][j]; a1 += sm[cg + G * k][8 + j]; }
        p.partial[((long long)blockIdx.x * 2 + 0) * C + c] = a0;
        p.partial[((long long)blockIdx.x * 2 + 1) * C + c] = a1;
    }
}

// Streaming form of the elementwise pass (bf16 vector path; stat: [4][C] as BnProb::stat, in global or shared memory): a thread keeps ONE group of 8 channels for all its rows, so the
// per-channel constants are loaded once into registers and the loop is loads, arithmetic and a store; a CTA takes at least 16 passes
// of 256 / G rows (32768 elements), four rows of loads in flight per thread.  MODE 0: a = relu(bn(x)); MODE 1: dx (+ add).
template <int MODE>
__device__ void bn_stream_vec(const BnProb& p, const float* __restrict__ stat) {
    const int C = p.C, G = C >> 3, R = 256 / G;
    const int g = threadIdx.x % G, r = threadIdx.x / G;
    // the grid's CTAs share the rows evenly, in whole passes of 4 * R rows (at least 16 passes of R rows each)
    long long rows_per_cta = (p.m + gridDim.x - 1) / gridDim.x;
    rows_per_cta = (rows_per_cta + 4 * R - 1) / (4 * R) * (4 * R); if (rows_per_cta < 16 * R) rows_per_cta = 16 * R;
    const long long r0 = (long long)blockIdx.x * rows_per_cta;
    if (r0 >= p.m) return;
    const long long r1 = r0 + rows_per_cta < p.m ? r0 + rows_per_cta : p.m;
    float mean[8], istd[8], ga[8], be[8], sb[8], sg[8];
    const float inv_m = 1.f / (float)p.m;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int c = g * 8 + j;
        mean[j] = stat[c]; istd[j] = stat[C + c]; ga[j] = p.gamma[c]; be[j] = p.beta[c];
        if (MODE == 1) { sb[j] = stat[2 * C + c] * inv_m; sg[j] = stat[3 * C + c] * inv_m; }
    }
    const uint4* xv = reinterpret_cast<const uint4*>(p.x);
    const uint4* dv = reinterpret_cast<const uint4*>(p.da);
    const uint4* av = reinterpret_cast<const uint4*>(p.add);
    uint4* ov = reinterpret_cast<uint4*>(MODE == 0 ? p.a : p.dx);
    for (long long row = r0 + r; row < r1; row += 4 * R) {
        uint4 xs[4], ds[4], as[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const long long rr = row + (long long)u * R;
            if (rr < r1) {
                xs[u] = __ldg(xv + rr * G + g);
                if (MODE == 1) { ds[u] = __ldg(dv + rr * G + g); if (av) as[u] = __ldg(av + rr * G + g); }
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const long long rr = row + (long long)u * R;
            if (rr < r1) {
                float x[8], o[8]; unpack8(xs[u], x);
                if (MODE == 0) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) { const float z = (x[j] - mean[j]) * istd[j] * ga[j] + be[j]; o[j] = z > 0.f ? z : 0.f; }
                } else {
                    float d[8]; unpack8(ds[u], d);
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float xh = (x[j] - mean[j]) * istd[j];
                        const float dz = (xh * ga[j] + be[j] > 0.f) ? d[j] : 0.f;
                        o[j] = ga[j] * istd[j] * (dz - sb[j] - xh * sg[j]);
                    }
                    if (av) { float ad[8]; unpack8(as[u], ad);
#pragma unroll
                        for (int j = 0; j < 8; ++j) o[j] += ad[j]; }
                }
                ov[rr * G + g] = pack8(o);
            }
        }
    }
}

// ---- the other types and channel counts: a thread owns V consecutive channels (4 where the channel count and the addresses allow 8- and
// 16-byte accesses, else 1) and every R-th row, with eight rows of loads in flight (four of 16 bytes), added in ascending order
template <class T, int V> struct Lanes { float v; };                         // one thread's channels of a row as loaded
template <> struct Lanes<float, 4> { float4 v; };
template <> struct Lanes<__nv_bfloat16, 4> { uint2 v; };
template <class T, int V> struct LaneRows { static constexpr int U = V == 4 && sizeof(T) == 4 ? 4 : 8; };
template <class T, int V> __device__ __forceinline__ Lanes<T, V> ldl(const void* p, long long i) {
    Lanes<T, V> l;
    if constexpr (V == 1) l.v = ldf<T>(p, i);
    else if constexpr (sizeof(T) == 4) l.v = __ldg(reinterpret_cast<const float4*>((const float*)p + i));
    else l.v = __ldg(reinterpret_cast<const uint2*>((const __nv_bfloat16*)p + i));
    return l;
}
template <class T, int V> __device__ __forceinline__ void unl(const Lanes<T, V>& l, float* f) {
    if constexpr (V == 1) f[0] = l.v;
    else if constexpr (sizeof(T) == 4) { f[0] = l.v.x; f[1] = l.v.y; f[2] = l.v.z; f[3] = l.v.w; }
    else { f[0] = __uint_as_float(l.v.x << 16); f[1] = __uint_as_float(l.v.x & 0xFFFF0000u); f[2] = __uint_as_float(l.v.y << 16); f[3] = __uint_as_float(l.v.y & 0xFFFF0000u); }
}
template <class T, int V> __device__ __forceinline__ void stv(void* p, long long i, const float* f) {
    if constexpr (V == 1) stf<T>(p, i, f[0]);
    else if constexpr (sizeof(T) == 4) *reinterpret_cast<float4*>((float*)p + i) = make_float4(f[0], f[1], f[2], f[3]);
    else {
        __nv_bfloat162 h0 = __floats2bfloat162_rn(f[0], f[1]), h1 = __floats2bfloat162_rn(f[2], f[3]);
        *reinterpret_cast<uint2*>((__nv_bfloat16*)p + i) = make_uint2(*reinterpret_cast<uint32_t*>(&h0), *reinterpret_cast<uint32_t*>(&h1));
    }
}
template <class T> __device__ __forceinline__ bool bn_by_four(const BnProb& p) {
    return (p.C & 3) == 0 && (((uintptr_t)p.x | (uintptr_t)p.a | (uintptr_t)p.da | (uintptr_t)p.dx | (uintptr_t)p.add) & (4 * sizeof(T) - 1)) == 0;
}
template <class T, int MODE, int V>
__device__ void bn_reduce_lanes(const BnProb& p) {
    constexpr int U = LaneRows<T, V>::U;
    __shared__ double part[2][V][256];
    const int C = p.C, NG = C / V, nl = NG < 256 ? NG : 256, R = 256 / nl;
    const int rg = threadIdx.x / nl, lane = threadIdx.x % nl;
    const long long r0 = (long long)blockIdx.x * p.rows_per_chunk;
    long long r1 = r0 + p.rows_per_chunk; if (r1 > p.m) r1 = p.m;
    for (int gb = 0; gb < NG; gb += nl) {
        const int c = (gb + lane) * V;
        float s0[V], s1[V];
#pragma unroll
        for (int j = 0; j < V; ++j) { s0[j] = 0.f; s1[j] = 0.f; }
        if (rg < R && c < C) {
            float mean[V], istd[V], g[V], b[V], shift[V];
            if (MODE == 1) {
#pragma unroll
                for (int j = 0; j < V; ++j) { mean[j] = p.stat[c + j]; istd[j] = p.stat[C + c + j]; g[j] = p.gamma[c + j]; b[j] = p.beta[c + j]; }
            } else unl<T, V>(ldl<T, V>(p.x, c), shift);      // sums of (x - x[0,c]): no cancellation when |mean| >> std
            for (long long r = r0 + rg; r < r1; r += U * R) {
                Lanes<T, V> xs[U], ds[MODE == 1 ? U : 1];
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (r + u * R < r1) { const long long i = (r + u * R) * C + c; xs[u] = ldl<T, V>(p.x, i); if (MODE == 1) ds[u] = ldl<T, V>(p.da, i); }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (r + u * R >= r1) break;
                    float xv[V], dv[V]; unl<T, V>(xs[u], xv); if (MODE == 1) unl<T, V>(ds[u], dv);
#pragma unroll
                    for (int j = 0; j < V; ++j) {
                        if (MODE == 0) { const float x = xv[j] - shift[j]; s0[j] += x; s1[j] += x * x; }
                        else { const float xh = (xv[j] - mean[j]) * istd[j], dz = xh * g[j] + b[j] > 0.f ? dv[j] : 0.f; s0[j] += dz; s1[j] += dz * xh; }
                    }
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < V; ++j) { part[0][j][threadIdx.x] = s0[j]; part[1][j][threadIdx.x] = s1[j]; }
        __syncthreads();
        for (int i = threadIdx.x; i < 2 * nl * V; i += 256) {
            const int which = i / (nl * V), ch = i - which * nl * V, cc = gb * V + ch;
            if (cc >= C) continue;
            double a = 0.0;
            for (int k = 0; k < R; ++k) a += part[which][ch % V][k * nl + ch / V];
            p.partial[((long long)blockIdx.x * 2 + which) * C + cc] = a;
        }
    }
}

// MODE 0: sums of x and x^2.  MODE 1: sums of dz and dz*xhat (backward).
// VEC: every problem of the launch takes the vector path.  Two kernels, because one with both paths has the registers, shared memory and code
// of the larger (forward + backward of 65535 x 64: 108 us against 101).
template <class T, int MODE, bool VEC>
__global__ void __launch_bounds__(256) bn_reduce_kernel(const BnProb* __restrict__ probs) {
    const BnProb& p = probs[blockIdx.y];
    if ((int)blockIdx.x >= p.chunks || p.eval) return;
    if constexpr (VEC) bn_reduce_vec<MODE>(p);
    else if (bn_by_four<T>(p)) bn_reduce_lanes<T, MODE, 4>(p);
    else bn_reduce_lanes<T, MODE, 1>(p);
}

template <class T, int MODE>
__global__ void bn_finalize_kernel(const BnProb* __restrict__ probs) {
    // one warp per channel: lane l adds chunks l, l+32, ... in order, then a fixed butterfly over the lanes
    const BnProb& p = probs[blockIdx.y];
    const int lane = threadIdx.x & 31;
    const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (c >= p.C) return;
    if (p.eval) {
        if (MODE == 0 && lane == 0) { p.stat[c] = p.run_mean[c]; p.stat[p.C + c] = (float)(1.0 / sqrt((double)p.run_var[c] + (double)p.eps)); }
        return;
    }
    double a0 = 0.0, a1 = 0.0;
    for (int k = lane; k < p.chunks; k += 32) { a0 += p.partial[((long long)k * 2 + 0) * p.C + c]; a1 += p.partial[((long long)k * 2 + 1) * p.C + c]; }
    for (int d = 16; d; d >>= 1) { a0 += __shfl_xor_sync(0xffffffffu, a0, d); a1 += __shfl_xor_sync(0xffffffffu, a1, d); }
    if (lane != 0) return;
    if (MODE == 0) {
        const double m = (double)p.m, dm = a0 / m;                 // sums are of x - x[0,c]
        double var = a1 / m - dm * dm; if (var < 0.0) var = 0.0;
        const double mean = dm + (double)ldf<T>(p.x, c);
        p.stat[c] = (float)mean;
        p.stat[p.C + c] = (float)(1.0 / sqrt(var + (double)p.eps));
        if (p.run_mean) {
            const double unb = p.m > 1 ? var * m / (m - 1.0) : var, mo = (double)p.momentum;
            p.run_mean[c] = (float)((1.0 - mo) * (double)p.run_mean[c] + mo * mean);
            p.run_var[c] = (float)((1.0 - mo) * (double)p.run_var[c] + mo * unb);
        }
    } else {
        p.stat[2 * p.C + c] = (float)a0; p.stat[3 * p.C + c] = (float)a1;
        p.dbeta[c] = (float)a0; p.dgamma[c] = (float)a1;
    }
}

// The elementwise pass of the other types and channel counts, laid out like their sums: a thread keeps its channels with their constants in
// registers and walks down its rows; a CTA takes an even share of the rows.  (A thread per element, with a 64-bit division for the channel and
// its constants loaded anew, and sums with one load in flight: forward + backward of 500000 x 100 in bf16 2000 us, 305 now; 1000000 x 64 in fp32
// 2440, 471 now; their eight passes over the tensors take 123 and 313 at the copy rate.)
template <class T, int MODE, int V>
__device__ void bn_stream_lanes(const BnProb& p) {
    constexpr int U = LaneRows<T, V>::U;
    const int C = p.C, NG = C / V, nl = NG < 256 ? NG : 256, R = 256 / nl, rg = threadIdx.x / nl, lane = threadIdx.x % nl;
    long long rows = (p.m + gridDim.x - 1) / gridDim.x; rows = (rows + R - 1) / R * R;
    const long long r0 = blockIdx.x * rows, r1 = r0 + rows < p.m ? r0 + rows : p.m;
    const float inv_m = 1.f / (float)p.m;
    const void* const add = p.add; void* const out = MODE == 0 ? p.a : p.dx;
    if (rg >= R) return;
    for (int c = lane * V; c < C; c += nl * V) {
        float mean[V], istd[V], g[V], b[V], sb[V], sg[V];
#pragma unroll
        for (int j = 0; j < V; ++j) {
            mean[j] = p.stat[c + j]; istd[j] = p.stat[C + c + j]; g[j] = p.gamma[c + j]; b[j] = p.beta[c + j];
            if (MODE == 1) { sb[j] = p.stat[2 * C + c + j] * inv_m; sg[j] = p.stat[3 * C + c + j] * inv_m; }
        }
        for (long long r = r0 + rg; r < r1; r += U * R) {
            Lanes<T, V> xs[U], ds[MODE == 1 ? U : 1], as[MODE == 1 ? U : 1];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (r + u * R < r1) {
                    const long long i = (r + u * R) * C + c;
                    xs[u] = ldl<T, V>(p.x, i);
                    if (MODE == 1) { ds[u] = ldl<T, V>(p.da, i); if (add) as[u] = ldl<T, V>(add, i); }
                }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (r + u * R >= r1) break;
                float o[V], xv[V], dv[V], av[V]; unl<T, V>(xs[u], xv); if (MODE == 1) { unl<T, V>(ds[u], dv); if (add) unl<T, V>(as[u], av); }
#pragma unroll
                for (int j = 0; j < V; ++j) {
                    const float xh = (xv[j] - mean[j]) * istd[j], z = xh * g[j] + b[j];
                    if (MODE == 0) o[j] = z > 0.f ? z : 0.f;
                    else { o[j] = g[j] * istd[j] * ((z > 0.f ? dv[j] : 0.f) - sb[j] - xh * sg[j]); if (add) o[j] += av[j]; }
                }
                stv<T, V>(out, (r + u * R) * C + c, o);
            }
        }
    }
}
template <class T, bool VEC>
__global__ void __launch_bounds__(256) bn_apply_kernel(const BnProb* __restrict__ probs) {
    const BnProb& p = probs[blockIdx.y];
    if constexpr (VEC) bn_stream_vec<0>(p, p.stat); else if (bn_by_four<T>(p)) bn_stream_lanes<T, 0, 4>(p); else bn_stream_lanes<T, 0, 1>(p);
}
template <class T, bool VEC>
__global__ void __launch_bounds__(256, 2) bn_bwd_apply_kernel(const BnProb* __restrict__ probs) {
    const BnProb& p = probs[blockIdx.y];
    if constexpr (VEC) bn_stream_vec<1>(p, p.stat); else if (bn_by_four<T>(p)) bn_stream_lanes<T, 1, 4>(p); else bn_stream_lanes<T, 1, 1>(p);
}

static int ew_grid(long long n) { long long g = (n + 255) / 256; if (g > 148 * 16) g = 148 * 16; if (g < 1) g = 1; return (int)g; }

void launch_bn_stats(const BnProb* d, int nprob, int max_chunks, int max_c, bool bf16, bool vec, cudaStream_t s) {
    const dim3 g(max_chunks, nprob);
    if (vec) bn_reduce_kernel<__nv_bfloat16, 0, true><<<g, 256, 0, s>>>(d);
    else if (bf16) bn_reduce_kernel<__nv_bfloat16, 0, false><<<g, 256, 0, s>>>(d);
    else bn_reduce_kernel<float, 0, false><<<g, 256, 0, s>>>(d);
    if (bf16) bn_finalize_kernel<__nv_bfloat16, 0><<<dim3((max_c + 7) / 8, nprob), 256, 0, s>>>(d);
    else bn_finalize_kernel<float, 0><<<dim3((max_c + 7) / 8, nprob), 256, 0, s>>>(d);
}
void launch_bn_eval_stats(const BnProb* d, int nprob, int max_c, cudaStream_t s) {
    bn_finalize_kernel<float, 0><<<dim3((max_c + 7) / 8, nprob), 256, 0, s>>>(d);
}
// The vector path takes about 32768 elements per CTA (see bn_stream_vec), in whole waves of the CTAs that are resident together: with three
// and a half waves the last one runs half empty.  At most about 16 CTAs per SM: more and shorter ones stream worse (8 x 131072 x 256
// backward: 28 waves of 296 CTAs 370 us, eight waves 322).
template <class K>
static int stream_grid(K kernel, int& slots, long long n, int nprob) {
    if (!slots) {
        int dev = 0, sms = 0, per = 0; cudaGetDevice(&dev); cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, 256, 0);
        slots = std::max(1, sms * per);
    }
    const long long total = std::max(1ll, (n + 32767) / 32768 * nprob);
    if (total <= slots) return (int)std::max(1ll, (n + 32767) / 32768);
    const long long waves = std::min((total + slots / 2) / slots, std::max(1ll, 2368ll / slots));
    return (int)std::max(1ll, waves * slots / nprob);
}
void launch_bn_apply(const BnProb* d, int nprob, long long max_elems, bool bf16, bool vec, cudaStream_t s) {
    static int slots = 0;
    if (vec) bn_apply_kernel<__nv_bfloat16, true><<<dim3(stream_grid(bn_apply_kernel<__nv_bfloat16, true>, slots, max_elems, nprob), nprob), 256, 0, s>>>(d);
    else if (bf16) bn_apply_kernel<__nv_bfloat16, false><<<dim3(ew_grid(max_elems), nprob), 256, 0, s>>>(d);
    else bn_apply_kernel<float, false><<<dim3(ew_grid(max_elems), nprob), 256, 0, s>>>(d);
}
void launch_bn_bwd_reduce(const BnProb* d, int nprob, int max_chunks, int max_c, bool bf16, bool vec, cudaStream_t s) {
    const dim3 g(max_chunks, nprob);
    if (vec) bn_reduce_kernel<__nv_bfloat16, 1, true><<<g, 256, 0, s>>>(d);
    else if (bf16) bn_reduce_kernel<__nv_bfloat16, 1, false><<<g, 256, 0, s>>>(d);
    else bn_reduce_kernel<float, 1, false><<<g, 256, 0, s>>>(d);
    bn_finalize_kernel<float, 1><<<dim3((max_c + 7) / 8, nprob), 256, 0, s>>>(d);
}
void launch_bn_bwd_apply(const BnProb* d, int nprob, long long max_elems, bool bf16, bool vec, cudaStream_t s) {
    static int slots = 0;
    if (vec) bn_bwd_apply_kernel<__nv_bfloat16, true><<<dim3(stream_grid(bn_bwd_apply_kernel<__nv_bfloat16, true>, slots, max_elems, nprob), nprob), 256, 0, s>>>(d);
    else if (bf16) bn_bwd_apply_kernel<__nv_bfloat16, false><<<dim3(ew_grid(max_elems), nprob), 256, 0, s>>>(d);
    else bn_bwd_apply_kernel<float, false><<<dim3(ew_grid(max_elems), nprob), 256, 0, s>>>(d);
}

// dst[r][0..cols) = src[r][0..cols) for rows of different pitch (fp32): the weight gradient of an im2col'ed stem, computed with
// the padded column count, goes to its place in the gradient vector
__global__ void repack_rows_kernel(const ConvProb* __restrict__ probs) {
    const ConvProb& p = probs[blockIdx.y];
    const float* src = (const float*)p.act; float* dst = (float*)p.out;
    const int n = p.M * p.Ncol;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int r = i / p.Ncol, c = i - r * p.Ncol;
        dst[i] = src[(long long)r * p.Kred + c];
    }
}
void launch_repack_rows(const ConvProb* d, int nprob, int max_elems, cudaStream_t s) {
    repack_rows_kernel<<<dim3(std::max(1, std::min((max_elems + 255) / 256, 148)), nprob), 256, 0, s>>>(d);
}

}  // namespace resist
