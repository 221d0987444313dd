// Evaluation (Sec. 2.6) of a run of identity basic blocks of a narrow stage, image by image, in one launch.
//
// With running statistics every image is independent of the others, and a map of 32 x 32 x 16, 16 x 16 x 32 or 8 x 8 x 64 elements fits shared
// memory three times over (the residual stream x and the inputs a1, a2 of the two convolutions of a block).  So a CTA takes one image (two to
// eight small ones) and carries it through ALL blocks of the run: nothing between the run's input and the BN+ReLU of its output goes through L2, and a
// barrier of the CTA stands where a launch per convolution stood.
//
// What bounds it: the rate of mma.sync (m16n8k16).  A task of a warp is a strip of four map rows x 16 columns (or the 8 columns of two images of maps up
// to 8 wide) x 16 output channels, all its accumulators in registers.  A fragment of input row i, shifted by filter column s, serves the three output
// rows i - 1 .. i + 1 it is a tap of: 18 ldmatrix per 72 MMAs of a 16-channel step, where one per tap and row would be 36 and take as long as the
// MMAs.  Filters come from L2 in the fragments' own order (eval_chain_pack_kernel), 16 bytes per lane, filter row by filter row: a row's registers are
// refilled for the next step as soon as the last map row that uses them is through.
//
// Shared memory: [8-channel group][position][8 channels], 16 bytes per position, so that the eight rows of an ldmatrix matrix are 128 consecutive
// bytes without padding or swizzle; positions are a zero-bordered map of W + 1 columns (the column W of a row is the column -1 of the next).
//
// Measured: evaluation of ResNet-110 on 1000 images 3290 -> 1984 us, its 51 identity blocks 1725 us of that (282 TFLOP/s); 115 launches -> 15.
#include <algorithm>
#include "internal.h"

namespace resist {

namespace {
__device__ __forceinline__ uint32_t sm_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t* r) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma16(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint4 ldg_pinned(const uint4* p) {     // stays where it is written: the compiler would sink the load to its first use
    uint4 v; asm volatile("ld.global.nc.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p)); return v;
}
__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }
__device__ __forceinline__ uint32_t bf_pack(float a, float b) { __nv_bfloat162 h = __floats2bfloat162_rn(a, b); return *reinterpret_cast<uint32_t*>(&h); }
__device__ __forceinline__ float bn_relu(float x, float mean, float istd, float g, float b) { const float z = (x - mean) * istd * g + b; return z > 0.f ? z : 0.f; }

constexpr int CHAIN_THREADS = 256, CHAIN_WARPS = CHAIN_THREADS / 32, CHAIN_R = 4;       // map rows of a task
inline int chain_set(int C) { return 4 * C + 16; }                // floats of a BN's constants: mean | 1/std | gamma | beta, then the scale of the convolution before it
}  // namespace

// Filters to bf16 in fragment order [16 output channels][16 input channels][tap][lane]: the lane's four registers of two MMAs' B operands (the
// columns permuted so that a thread's accumulators are four consecutive channels); constants of the BN.
__global__ void __launch_bounds__(256) eval_chain_pack_kernel(const ChainLayer* __restrict__ layers) {
    const ChainLayer& l = layers[blockIdx.y];
    const int C = l.C, steps = C / 16;
    if (l.w)
        for (int i = blockIdx.x * 256 + threadIdx.x; i < steps * steps * 9 * 32; i += gridDim.x * 256) {
            const int lane = i & 31, t = (i >> 5) % 9, kn = (i >> 5) / 9, k = kn % steps, n = kn / steps, g8 = lane >> 2, t4 = lane & 3;
            uint32_t r[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {                         // j: (column block, upper half of the 16 input channels)
                const int out = n * 16 + (g8 >> 1) * 4 + 2 * (j >> 1) + (g8 & 1), in = k * 16 + t4 * 2 + 8 * (j & 1);
                const float* w = l.w + ((long long)out * 9 + t) * C + in;
                r[j] = bf_pack(w[0], w[1]);
            }
            l.wdst[i] = make_uint4(r[0], r[1], r[2], r[3]);
        }
    if (blockIdx.x == 0) {
        for (int c = threadIdx.x; c < C; c += 256) {
            l.cdst[c] = l.gamma ? l.mean[c] : 0.f; l.cdst[C + c] = l.gamma ? (float)(1.0 / sqrt((double)l.var[c] + (double)l.eps)) : 1.f;
            l.cdst[2 * C + c] = l.gamma ? l.gamma[c] : 1.f; l.cdst[3 * C + c] = l.gamma ? l.beta[c] : 0.f;
        }
        if (threadIdx.x == 0) l.cdst[4 * C] = l.scale;
    }
}

template <int C, bool PAIR>
__global__ void __launch_bounds__(CHAIN_THREADS, 2) eval_chain_kernel(const ChainProb* __restrict__ probs) {
    constexpr int NG = C / 16, SET = 4 * C + 16;
    extern __shared__ __align__(128) uint8_t sm[];
    const ChainProb p = *probs;
    const int H = p.H, W = p.W, HW = H * W, Wp = W + 1, imgs = p.imgs, img0 = blockIdx.x * imgs;
    const uint32_t plane = (uint32_t)p.plane, img_bytes = (C / 8) * plane, buf_bytes = imgs * img_bytes;
    uint8_t* const s_a = sm;                                      // [2][imgs][C / 8][positions][8]
    uint8_t* const s_x = sm + 2 * buf_bytes;                      // [imgs][C / 16][H * W][16]
    float* const s_c = reinterpret_cast<float*>(s_x + (size_t)imgs * HW * C * 2);       // [2][SET]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g8 = lane >> 2, t4 = lane & 3;

    // ---- borders (and everything else) to zero, the first BN's constants, then x and a1 = relu(bn(x))
    for (uint32_t i = tid * 16; i < 2 * buf_bytes; i += CHAIN_THREADS * 16) *reinterpret_cast<uint4*>(s_a + i) = make_uint4(0u, 0u, 0u, 0u);
    for (int i = tid; i < 2 * SET; i += CHAIN_THREADS) s_c[i] = __ldg(p.cst + i);
    __syncthreads();
    {
        const int n_img = min(imgs, p.N - img0), chunks = n_img * HW * (C / 8);
        const uint4* src = reinterpret_cast<const uint4*>(p.x + (long long)img0 * HW * C);
        for (int i0 = tid; i0 < chunks; i0 += 4 * CHAIN_THREADS) {
            uint4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = __ldg(src + min(i0 + u * CHAIN_THREADS, chunks - 1));
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = i0 + u * CHAIN_THREADS;
                if (i >= chunks) break;
                const int g = i % (C / 8), q = i / (C / 8), im = q / HW, pix = q - im * HW, y = pix / W, x = pix - y * W;
                *reinterpret_cast<uint4*>(s_x + ((size_t)(im * NG + (g >> 1)) * HW + pix) * 32 + (g & 1) * 16) = v[u];
                const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w}; uint32_t o[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int c = g * 8 + 2 * k;
                    o[k] = bf_pack(bn_relu(bf_lo(w[k]), s_c[c], s_c[C + c], s_c[2 * C + c], s_c[3 * C + c]),
                                   bn_relu(bf_hi(w[k]), s_c[c + 1], s_c[C + c + 1], s_c[2 * C + c + 1], s_c[3 * C + c + 1]));
                }
                *reinterpret_cast<uint4*>(s_a + im * img_bytes + g * plane + ((y + 1) * Wp + x + 1) * 16) = make_uint4(o[0], o[1], o[2], o[3]);
            }
        }
    }

    // this lane's row of an ldmatrix: map column (and image of a pair) and 8-channel group
    const uint32_t a_lane = (uint32_t)(lane >> 4) * plane + (PAIR ? (uint32_t)((lane >> 3) & 1) * img_bytes + (uint32_t)(lane & 7) * 16u : (uint32_t)(lane & 15) * 16u);
    const uint32_t a_sm = sm_u32(s_a);
    const int strips = (H + CHAIN_R - 1) / CHAIN_R, xblocks = PAIR ? 1 : (W + 15) / 16, slots = PAIR ? imgs / 2 : imgs;
    const int tasks = NG * strips * xblocks * slots;
    // fragments of a task's filter rows: [filter row][filter column]
    uint4 b[3][3];
    auto frag = [&](int layer, int ng, int k, int r) {
        const uint4* w = p.wpk + ((long long)layer * NG * NG + ng * NG + k) * (9 * 32) + r * (3 * 32) + lane;
#pragma unroll
        for (int s = 0; s < 3; ++s) b[r][s] = ldg_pinned(w + s * 32);
    };
    if (warp < tasks) {
#pragma unroll
        for (int r = 0; r < 3; ++r) frag(0, warp % NG, 0, r);
    }
    const int layers = p.layers;
    for (int l = 0; l < layers; ++l) {
        __syncthreads();                                          // this layer's input and constants are in shared memory
        const bool second = l & 1, last = l + 1 == layers;
        const uint32_t src = a_sm + (second ? buf_bytes : 0u) + a_lane;
        uint8_t* const dst = s_a + (second ? 0u : buf_bytes);
        const float* const cs = s_c + ((l + 1) & 1) * SET;
        const float scale = cs[4 * C];
        for (int task = warp; task < tasks; task += CHAIN_WARPS) {
            const int ng = task % NG; int rest = task / NG;
            const int xb = rest % xblocks; rest /= xblocks;
            const int y0 = (rest % strips) * CHAIN_R, slot = rest / strips, x0 = xb * 16;
            float acc[CHAIN_R][2][4];
#pragma unroll
            for (int r = 0; r < CHAIN_R; ++r)
#pragma unroll
                for (int j = 0; j < 2; ++j) { acc[r][j][0] = acc[r][j][1] = acc[r][j][2] = acc[r][j][3] = 0.f; }
            uint32_t row[CHAIN_R + 2];                            // input rows y0 - 1 .. y0 + R; a strip that ends below the map reads the border row again
#pragma unroll
            for (int i = 0; i < CHAIN_R + 2; ++i) row[i] = src + (uint32_t)(slot * (PAIR ? 2 : 1)) * img_bytes + (uint32_t)(min(y0 + i, H + 1) * Wp + x0) * 16u;
            const int ntask = task + CHAIN_WARPS;
            const bool more = ntask < tasks;                      // whose fragments follow: the next task's, or those of the warp's first task in the next layer
            const int nl = more ? l : min(l + 1, layers - 1), nng = more ? ntask % NG : warp % NG;
#pragma unroll
            for (int k = 0; k < NG; ++k) {
                const bool end = k == NG - 1;
#pragma unroll
                for (int i = 0; i < CHAIN_R + 2; ++i) {
#pragma unroll
                    for (int s = 0; s < 3; ++s) {
                        uint32_t a[4];
                        ldsm4(row[i] + (uint32_t)(2 * k) * plane + (uint32_t)s * 16u, a);
#pragma unroll
                        for (int r = 0; r < 3; ++r) {
                            const int o = i - r;
                            if (o < 0 || o >= CHAIN_R) continue;
                            mma16(acc[o][0], a, b[r][s].x, b[r][s].y);
                            mma16(acc[o][1], a, b[r][s].z, b[r][s].w);
                        }
                    }
                    if (i >= CHAIN_R - 1 && (NG > 1 || !more)) frag(end ? nl : l, end ? nng : ng, end ? 0 : k + 1, i - (CHAIN_R - 1));
                }
            }
            // ---- epilogue: thread (g8, t4) holds columns g8 and g8 + 8 (or column g8 of two images) of each row, channels t4 * 4 .. + 3 of the sixteen
            const int c0 = ng * 16 + t4 * 4;
            const float4 mean = *reinterpret_cast<const float4*>(cs + c0), istd = *reinterpret_cast<const float4*>(cs + C + c0);
            const float4 ga = *reinterpret_cast<const float4*>(cs + 2 * C + c0), be = *reinterpret_cast<const float4*>(cs + 3 * C + c0);
#pragma unroll
            for (int o = 0; o < CHAIN_R; ++o)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int y = y0 + o, x = PAIR ? g8 : x0 + g8 + 8 * h, im = PAIR ? 2 * slot + h : slot;
                    if (y >= H || x >= W) continue;
                    float v[4] = {acc[o][0][2 * h] * scale, acc[o][0][2 * h + 1] * scale, acc[o][1][2 * h] * scale, acc[o][1][2 * h + 1] * scale};
                    const int pix = y * W + x;
                    uint2* const xs = reinterpret_cast<uint2*>(s_x + ((size_t)(im * NG + ng) * HW + pix) * 32 + t4 * 8);
                    if (second) { const uint2 xv = *xs; v[0] += bf_lo(xv.x); v[1] += bf_hi(xv.x); v[2] += bf_lo(xv.y); v[3] += bf_hi(xv.y); }
                    const uint2 w = make_uint2(bf_pack(v[0], v[1]), bf_pack(v[2], v[3]));
                    const uint2 a = make_uint2(bf_pack(bn_relu(bf_lo(w.x), mean.x, istd.x, ga.x, be.x), bn_relu(bf_hi(w.x), mean.y, istd.y, ga.y, be.y)),
                                               bf_pack(bn_relu(bf_lo(w.y), mean.z, istd.z, ga.z, be.z), bn_relu(bf_hi(w.y), mean.w, istd.w, ga.w, be.w)));
                    if (last) {
                        if (img0 + im < p.N) {
                            const long long at = ((long long)(img0 + im) * HW + pix) * C + c0;
                            if (p.x_out) *reinterpret_cast<uint2*>(p.x_out + at) = w;
                            if (p.a_out) *reinterpret_cast<uint2*>(p.a_out + at) = a;
                        }
                    } else {
                        if (second) *xs = w;
                        *reinterpret_cast<uint2*>(dst + im * img_bytes + (ng * 2 + (t4 >> 1)) * plane + ((y + 1) * Wp + x + 1) * 16 + (t4 & 1) * 8) = a;
                    }
                }
        }
        // the next layer's constants take the place of the last one's, which every warp is through with
        if (!last && tid < SET / 4)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n\tcp.async.commit_group;\n\tcp.async.wait_group 0;"
                         ::"r"(sm_u32(s_c + (l & 1) * SET + tid * 4)), "l"(p.cst + (long long)(l + 2) * SET + tid * 4) : "memory");
    }
}

// ------------------------------------------------------------------------------------------------ host side
// Images per CTA: as many as give every warp a task.  Shared memory decides what is taken: C = 64 maps only as far as two CTAs fit an SM (larger ones run
// faster on tcgen05, layer by layer); 16 and 32 channels as far as one does.
static size_t chain_smem(const ChainProb& p) { return (size_t)2 * p.imgs * (p.C / 8) * p.plane + (size_t)p.imgs * p.H * p.W * p.C * 2 + 2 * chain_set(p.C) * 4; }
bool eval_chain_geometry(ChainProb& p) {
    if (p.C != 16 && p.C != 32 && p.C != 64) return false;
    if (p.H < 2 || p.W < 2 || p.H > 64 || p.W > 64) return false;
    p.pair = p.W <= 8;
    const int Wp = p.W + 1, xb = p.pair ? 1 : (p.W + 15) / 16;
    // the last read: row H + 1, columns up to 16 per block, one more for the last filter column
    const int npos = std::max((p.H + 2) * Wp + 1, (p.H + 1) * Wp + (p.pair ? 8 : 16 * xb) + 2);
    p.plane = (npos * 16 + 127) / 128 * 128 + 64;                 // 64 beyond a multiple of 128: the two planes of sixteen channels fall on different banks
    const int per = p.C / 16 * ((p.H + CHAIN_R - 1) / CHAIN_R) * xb;
    p.imgs = p.pair ? 2 : 1;
    while (per * (p.pair ? p.imgs / 2 : p.imgs) < CHAIN_WARPS && p.imgs < 8) p.imgs *= 2;
    return chain_smem(p) <= (p.C == 64 ? 113u : 200u) * 1024;
}
size_t eval_chain_weight_bytes(int C, int layers) { return (size_t)layers * 9 * C * C * 2; }
size_t eval_chain_const_bytes(int C, int layers) { return (size_t)(layers + 1) * chain_set(C) * 4; }
int eval_chain_set_floats(int C) { return chain_set(C); }
void launch_eval_chain_pack(const ChainLayer* d, int n, int max_c, cudaStream_t s) {
    const int steps = max_c / 16;
    eval_chain_pack_kernel<<<dim3((steps * steps * 9 * 32 + 255) / 256, n), 256, 0, s>>>(d);
}
template <int C, bool PAIR> static bool launch_chain(const ChainProb* d, const ChainProb& h, cudaStream_t s) {
    if (cudaFuncSetAttribute(eval_chain_kernel<C, PAIR>, cudaFuncAttributeMaxDynamicSharedMemorySize, 202 * 1024) != cudaSuccess) { cudaGetLastError(); return false; }
    eval_chain_kernel<C, PAIR><<<dim3((h.N + h.imgs - 1) / h.imgs), CHAIN_THREADS, chain_smem(h), s>>>(d);
    return true;
}
bool launch_eval_chain(const ChainProb* d, const ChainProb& h, cudaStream_t s) {
    if (h.C == 16) return h.pair ? launch_chain<16, true>(d, h, s) : launch_chain<16, false>(d, h, s);
    if (h.C == 32) return h.pair ? launch_chain<32, true>(d, h, s) : launch_chain<32, false>(d, h, s);
    return h.pair ? launch_chain<64, true>(d, h, s) : launch_chain<64, false>(d, h, s);
}

}  // namespace resist
