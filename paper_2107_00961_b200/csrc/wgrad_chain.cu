// Weight gradients of the 3x3, stride-1 layers of a run of narrow blocks (train_chain.cu), all layers of all sub-ResNets in one launch:
//   dw[k][t][c] = sum over images and positions of dy[pos][k] * a[pos + shift_t][c].
//
// The images of all problems form one line of units that is cut evenly among the SMs; a CTA adds up its share of a problem and writes one fp32 partial per problem it
// touches, a second kernel adds those in order.  A unit's maps are brought to shared memory by cp.async while the last unit is computed, in the layout of
// chain_core.h ([8-channel group][position][8 channels]): ldmatrix.trans turns 16 positions x 16 channels into a fragment of either operand.
//
// A warp owns 16 x 16 channels of all nine taps and goes down the rows of a block of columns: a fragment of activation row i, shifted by filter column s, is a tap
// of the gradient rows i - 1 .. i + 1, so a step of 16 positions is 18 MMAs on one new gradient fragment and three new activation fragments (nine and
// as many ldmatrix clocks as MMA clocks without that).
//
// Precision: mma.sync rounds its running sums toward zero (measured: 1.1e-8 relative per step of a chain, all of one sign), so a chain ends after RS steps and is added to a
// second set of accumulators in fp32, rounded to nearest; the partials are added in double.  The kernels this replaces had chains of 14 steps and more.
//
// WGRAD_FIGURES
#include <algorithm>
#include "chain_core.h"

namespace resist {
using namespace chain;

constexpr int WGC_THREADS = 256, WGC_WARPS = 8;

namespace {
__device__ __forceinline__ void ldsm4t(uint32_t addr, uint32_t* r) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
// The CTA that takes unit u of `total`, cut into `ctas` shares: CTA j has units [j * total / ctas, (j + 1) * total / ctas)
__host__ __device__ inline int share_of(long long u, long long total, int ctas) {
    long long j = u * ctas / total;
    while (j + 1 < ctas && (j + 1) * total / ctas <= u) ++j;
    while (j > 0 && j * total / ctas > u) --j;
    return (int)j;
}
}  // namespace

// C channels; RS steps of a chain (rows of a strip)
template <int C, int RS>
__global__ void __launch_bounds__(WGC_THREADS, 1) wgrad_chain_kernel(const WgChainProb* __restrict__ probs, const WgChainLaunch g) {
    constexpr int KC = C == 64 ? 32 : C, GA = C / 8, GD = KC / 8, NC = C / 16, COMBOS = KC / 16 * NC, WPC = WGC_WARPS / COMBOS > 0 ? WGC_WARPS / COMBOS : 1;
    static_assert(COMBOS * WPC == WGC_WARPS, "a warp per 16 x 16 channels and part of the positions");
    extern __shared__ __align__(128) uint8_t sm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int H = g.H, W = g.W, HW = H * W, Wp = W + 1, imgs = g.imgs, Wd = g.dy_cols;
    const uint32_t a_plane = (uint32_t)g.a_plane, d_plane = (uint32_t)g.d_plane;
    const uint32_t a_img = GA * a_plane, d_img = GD * d_plane, a_bytes = imgs * a_img, stage = a_bytes + imgs * d_img;
    const long long total = (long long)g.nq * g.units;
    const long long u0 = blockIdx.x * total / gridDim.x, u1 = (blockIdx.x + 1) * total / gridDim.x;
    const int combo = warp / WPC, part = warp % WPC, kc = combo / NC, cc = combo % NC;       // 16 gradient channels, 16 activation channels
    const int dx = g.cols == 16 ? 8 : 0, dy = g.cols == 16 ? 0 : RS;                          // where a step's second eight positions lie

    for (uint32_t i = tid * 16; i < 2 * stage; i += WGC_THREADS * 16) *reinterpret_cast<uint4*>(sm + i) = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    // a unit's maps: a warp per row of either tensor
    auto fetch = [&](long long u, int buf) {
        if (u < u1) {
            const int q = (int)(u / g.units), img0 = (int)(u - (long long)q * g.units) * imgs;
            const WgChainProb& p = probs[C == 64 ? q >> 1 : q];
            const int k0 = C == 64 ? (q & 1) * 32 : 0, rows = imgs * H;
            uint8_t* const base = sm + buf * stage;
            for (int r = warp; r < rows; r += WGC_WARPS) {
                const int im = r / H, y = r - im * H;
                const uint32_t live = img0 + im < g.N ? 16u : 0u;      // images past the last one are zero
                const __nv_bfloat16* as = p.a + (live ? ((long long)(img0 + im) * HW + y * W) * C : 0);
                const __nv_bfloat16* ds = p.dy + (live ? ((long long)(img0 + im) * HW + y * W) * C + k0 : 0);
                const uint32_t ad = sm_u32(base + im * a_img) + (uint32_t)((y + 1) * Wp + 1) * 16u, dd = sm_u32(base + a_bytes + im * d_img) + (uint32_t)(y * Wd) * 16u;
                for (int i = lane; i < W * GA; i += 32)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(ad + (uint32_t)(i % GA) * a_plane + (uint32_t)(i / GA) * 16u), "l"(as + (live ? (long long)i * 8 : 0)), "r"(live) : "memory");
                for (int i = lane; i < W * GD; i += 32)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dd + (uint32_t)(i % GD) * d_plane + (uint32_t)(i / GD) * 16u), "l"(ds + (live ? (long long)(i / GD) * C + (i % GD) * 8 : 0)), "r"(live) : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // this lane's row of an ldmatrix: gradient: matrices (positions 0-7, 8-15) x (channels 0-7, 8-15), channel half first; activations: positions first
    const uint32_t second = (uint32_t)(dx * 16) + (uint32_t)dy * (uint32_t)Wp * 16u, second_d = (uint32_t)(dx * 16) + (uint32_t)dy * (uint32_t)Wd * 16u;
    const uint32_t d_lane = (uint32_t)(kc * 2 + ((lane >> 3) & 1)) * d_plane + (uint32_t)(lane >> 4) * second_d + (uint32_t)(lane & 7) * 16u;
    const uint32_t a_lane = (uint32_t)(cc * 2 + (lane >> 4)) * a_plane + (uint32_t)((lane >> 3) & 1) * second + (uint32_t)(lane & 7) * 16u;

    float sum[9][2][4];
    auto clear = [&](float (&v)[9][2][4]) {
#pragma unroll
        for (int t = 0; t < 9; ++t)
#pragma unroll
            for (int j = 0; j < 2; ++j) { v[t][j][0] = v[t][j][1] = v[t][j][2] = v[t][j][3] = 0.f; }
    };
    clear(sum);
    fetch(u0, 0);
    int buf = 0;
    for (long long u = u0; u < u1; ++u) {
        fetch(u + 1, buf ^ 1);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();                                          // this unit's maps are in shared memory
        const uint32_t a_base = sm_u32(sm + buf * stage) + a_lane, d_base = sm_u32(sm + buf * stage + a_bytes) + d_lane;
        const int strips = g.strips, blocks = strips * g.xblocks, tasks = blocks * imgs;
        for (int t = part; t < tasks; t += WPC) {
            const int im = t / blocks, bl = t - im * blocks, xb = bl / strips, y0 = (bl - xb * strips) * (dy ? 2 * RS : RS), x0 = xb * g.cols;
            const uint32_t ar = a_base + im * a_img + (uint32_t)(y0 * Wp + x0) * 16u, dr = d_base + im * d_img + (uint32_t)(y0 * Wd + x0) * 16u;
            const uint32_t a_row = (uint32_t)Wp * 16u, d_row = (uint32_t)Wd * 16u;
            float acc[9][2][4];
            clear(acc);
            uint32_t b[3][3][4], d[4];
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int s = 0; s < 3; ++s) ldsm4t(ar + (uint32_t)i * a_row + (uint32_t)s * 16u, b[i][s]);
#pragma unroll
            for (int i = 0; i < RS; ++i) {
                ldsm4t(dr + (uint32_t)i * d_row, d);
#pragma unroll
                for (int s = 0; s < 3; ++s) ldsm4t(ar + (uint32_t)(i + 2) * a_row + (uint32_t)s * 16u, b[(i + 2) % 3][s]);
#pragma unroll
                for (int r = 0; r < 3; ++r)
#pragma unroll
                    for (int s = 0; s < 3; ++s) {
                        mma16(acc[r * 3 + s][0], d, b[(i + r) % 3][s][0], b[(i + r) % 3][s][1]);
                        mma16(acc[r * 3 + s][1], d, b[(i + r) % 3][s][2], b[(i + r) % 3][s][3]);
                    }
            }
#pragma unroll
            for (int t9 = 0; t9 < 9; ++t9)
#pragma unroll
                for (int j = 0; j < 2; ++j)
#pragma unroll
                    for (int e = 0; e < 4; ++e) sum[t9][j][e] += acc[t9][j][e];
        }
        __syncthreads();                                          // every warp is through with the unit before it is overwritten
        buf ^= 1;
        const int q = (int)(u / g.units);
        if (u + 1 == u1 || (int)((u + 1) / g.units) != q) {       // the CTA's share of this problem ends here: the warps of the same channels added in order
            const int first = share_of((long long)q * g.units, total, gridDim.x);
            float* const dst = g.partial + ((long long)q * g.max_parts + (blockIdx.x - first)) * (9 * KC * C);
            const int g8 = lane >> 2, t4 = lane & 3;
            float* const red = reinterpret_cast<float*>(sm + 2 * stage);      // [COMBOS][9][16][16]
            for (int w = 0; w < WPC; ++w) {
                if (part == w)
#pragma unroll
                    for (int t9 = 0; t9 < 9; ++t9)
#pragma unroll
                        for (int j = 0; j < 2; ++j)
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                float2* v = reinterpret_cast<float2*>(red + ((combo * 9 + t9) * 16 + g8 + 8 * h) * 16 + j * 8 + t4 * 2);
                                float2 o = make_float2(sum[t9][j][2 * h], sum[t9][j][2 * h + 1]);
                                if (w > 0) { const float2 c = *v; o.x += c.x; o.y += c.y; }
                                *v = o;
                            }
                __syncthreads();
            }
            // partial [tap][k][c]
            for (int i = tid; i < 9 * KC * C; i += WGC_THREADS) {
                const int t9 = i / (KC * C), k = i / C % KC, c = i % C;
                dst[i] = red[((((k >> 4) * NC + (c >> 4)) * 9 + t9) * 16 + (k & 15)) * 16 + (c & 15)];
            }
            __syncthreads();
            clear(sum);
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// out[k][t][c] = the CTAs' partials in order
__global__ void __launch_bounds__(256) wgrad_chain_reduce_kernel(const WgChainProb* __restrict__ probs, const WgChainLaunch g, int ctas) {
    const int C = g.C, KC = C == 64 ? 32 : C, q = blockIdx.y, n = 9 * KC * C;
    const long long total = (long long)g.nq * g.units;
    const int first = share_of((long long)q * g.units, total, ctas), parts = share_of((long long)(q + 1) * g.units - 1, total, ctas) - first + 1;
    const float* __restrict__ src = g.partial + (long long)q * g.max_parts * n;
    float* const out = probs[C == 64 ? q >> 1 : q].out;
    const int k0 = C == 64 ? (q & 1) * 32 : 0;
    for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) {
        double s = 0.0;
#pragma unroll 8
        for (int p = 0; p < parts; ++p) s += (double)src[(long long)p * n + i];
        const int t = i / (KC * C), k = i / C % KC, c = i % C;
        out[((long long)(k0 + k) * 9 + t) * C + c] = (float)s;
    }
}

// ------------------------------------------------------------------------------------------------ host side
static size_t wgc_stage(const WgChainLaunch& g) { return (size_t)g.imgs * ((g.C / 8) * g.a_plane + (g.C == 64 ? 4 : g.C / 8) * g.d_plane); }
static size_t wgc_smem(const WgChainLaunch& g) { const int kc = g.C == 64 ? 32 : g.C; return 2 * wgc_stage(g) + (size_t)9 * kc * g.C * 4; }
// Blocks of 16 columns and chains of 8 rows, or 8 columns and twice 4 rows where that wastes less of the map; images per unit so that all warps have work and a unit
// is at least about 1024 positions of a warp's.
bool wgrad_chain_geometry(int C, int H, int W, int N, WgChainLaunch& g) {
    if ((C != 16 && C != 32 && C != 64) || H < 2 || W < 2 || H > 64 || W > 64) return false;
    double best = 0; WgChainLaunch r{};
    for (int mode = 0; mode < 3; ++mode) {
        WgChainLaunch t{}; t.C = C; t.H = H; t.W = W; t.N = N;
        t.cols = mode == 2 ? 8 : 16; t.rs = mode == 0 ? 8 : 4;
        const int rows = t.cols == 8 ? 2 * t.rs : t.rs;
        t.strips = (H + rows - 1) / rows; t.xblocks = (W + t.cols - 1) / t.cols;
        t.dy_cols = t.xblocks * t.cols;
        // activations: zero-bordered map, the last read one row below the last strip; gradient: rows of whole blocks.  64 bytes beyond a multiple of 128: neighbouring
        // channel groups fall on different banks
        t.a_plane = (((t.strips * rows + 2) * (W + 1) + t.dy_cols - W + 1) * 16 + 127) / 128 * 128 + 64;
        t.d_plane = (t.strips * rows * t.dy_cols * 16 + 127) / 128 * 128 + 64;
        const int wpc = C == 16 ? 8 : C == 32 ? 2 : 1, blocks = t.strips * t.xblocks;
        for (t.imgs = 1; t.imgs <= 8; t.imgs *= 2) {
            if (wgc_smem(t) > 225 * 1024) break;
            const int rounds = (blocks * t.imgs + wpc - 1) / wpc;
            // MMA clocks of a round, the flush and the unit's barriers, per image
            const double cost = (rounds * (t.rs * 18 * 16.0 + 200.0) + 500.0) / t.imgs;
            if (best == 0 || cost < best) { best = cost; r = t; }
        }
    }
    if (best == 0) return false;
    r.units = (N + r.imgs - 1) / r.imgs;
    g = r;
    return true;
}
// CTAs of a launch of nprob problems, and how many of them touch one problem at most; the bytes of their partial sums
int wgrad_chain_plan(WgChainLaunch& g, int nprob, int sms, size_t* partial_bytes) {
    g.nq = nprob * (g.C == 64 ? 2 : 1);
    const long long total = (long long)g.nq * g.units;
    const int ctas = (int)std::min<long long>(sms, total);
    g.max_parts = 0;
    for (int q = 0; q < g.nq; ++q)
        g.max_parts = std::max(g.max_parts, share_of((long long)(q + 1) * g.units - 1, total, ctas) - share_of((long long)q * g.units, total, ctas) + 1);
    *partial_bytes = (size_t)g.nq * g.max_parts * 9 * (g.C == 64 ? 32 : g.C) * g.C * 4;
    return ctas;
}
template <int C, int RS> static bool launch_wgc(const WgChainProb* d, const WgChainLaunch& g, int ctas, cudaStream_t s) {
    if (cudaFuncSetAttribute(wgrad_chain_kernel<C, RS>, cudaFuncAttributeMaxDynamicSharedMemorySize, 225 * 1024) != cudaSuccess) { cudaGetLastError(); return false; }
    wgrad_chain_kernel<C, RS><<<ctas, WGC_THREADS, wgc_smem(g), s>>>(d, g);
    return true;
}
bool launch_wgrad_chain(const WgChainProb* d, const WgChainLaunch& g, int ctas, cudaStream_t s) {
    bool ok;
    if (g.rs == 8) ok = g.C == 16 ? launch_wgc<16, 8>(d, g, ctas, s) : g.C == 32 ? launch_wgc<32, 8>(d, g, ctas, s) : launch_wgc<64, 8>(d, g, ctas, s);
    else ok = g.C == 16 ? launch_wgc<16, 4>(d, g, ctas, s) : g.C == 32 ? launch_wgc<32, 4>(d, g, ctas, s) : launch_wgc<64, 4>(d, g, ctas, s);
    const int n = 9 * (g.C == 64 ? 32 : g.C) * g.C;
    if (ok) wgrad_chain_reduce_kernel<<<dim3(std::min((n + 255) / 256, 36), g.nq), 256, 0, s>>>(d, g, ctas);
    return ok;
}

}  // namespace resist
