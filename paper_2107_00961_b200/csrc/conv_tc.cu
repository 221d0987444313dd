// Tensor-core convolutions for sm_100a: implicit GEMM on tcgen05.mma with the accumulators in TMEM and the
// operands staged in shared memory by TMA with the 128-byte swizzle.
//
// Positions.  A 1x1 layer is a plain GEMM over the pixels of the tensor ("flat").  A 3x3 layer walks the batch as
// one tall zero-padded map: every image contributes Hp = H + 1 rows of Wp = W + 1 positions, the first row and the
// last column being zero (they are the padding of both neighbours).  In that order the operand of filter tap (r,s)
// is the SAME run of positions shifted by (r-1)*Wp + (s-1), so a tile's input window (128 positions plus a halo of
// Wp + 1 on either side) is fetched ONCE per 64-channel slab and all nine taps read it through shared-memory
// descriptors whose start address is moved by whole 128-byte rows.  The window is fetched as boxes of R tall rows
// (R divides Hp, so a box never straddles two images); the zero row and column are the out-of-bounds fill of TMA.
//
// Shared memory.  One row = one position x 64 channels = 128 bytes, rows consecutive, 16-byte chunks of a row
// XOR-swizzled with the row index (CU_TENSOR_MAP_SWIZZLE_128B writes that pattern by absolute shared-memory address
// and the tensor core reads it back by absolute address, so a descriptor may start at any 128-byte row).  Activations are K-major operands; weights are K-major in forward
// ([out channel][64 in channels]) and MN-major in dgrad ([64 reduction channels][64 out columns] blocks).
//
// Kernel structure of forward / dgrad (352 threads, one CTA per SM, persistent over the work of all problems of the launch).  A
// unit of work is a PAIR of neighbouring 128-position tiles times one column tile of up to 256 output channels:
// warp 0 = TMA producer (a ring of activation windows, two per step, and a ring of weight tiles, one per (slab, tap), shared by
// the two tiles of the pair); warp 1 = MMA issuer, an accumulator in TMEM per tile; warps 2..9 = two epilogue groups of four warps,
// one per tile of the pair (TMEM -> registers -> scale, residual add, bf16 -> staging slabs of 64 columns -> TMA store or row copy-out,
// with per-tile column sums for the BN that follows); warp 10 = the residual, by TMA into the staging slabs.
// The weight-gradient kernel (224 threads) has a producer warp per operand (0: dy, 2: a), one issuer warp (1) and four epilogue warps.
// Every wait is bounded: on expiry the kernel records the place in the status word, drains its copies and MMAs, frees its
// TMEM and returns.
#include <cuda.h>
#include <cstdio>
#include <climits>
#include <cstring>
#include <algorithm>
#include <type_traits>
#include "internal.h"

namespace resist {

// ------------------------------------------------------------------------------------------------ device helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// One thread of a converged warp.  The compiler knows that elect.sync leaves a single thread, so the tcgen05 and TMA instructions
// behind it take their operands from uniform registers; behind "lane == 0" it has to assume that several threads may be there and
// wraps every one of them in a loop over the active threads (measured: 78 to 150 cycles per tcgen05.mma instead of the tensor
// core's own 48 / 64 / 128 at N = 64 / 128 / 256).
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// bounded wait: false when the barrier did not flip within the limit or another role of the CTA gave up
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    for (uint32_t i = 0; i < (1u << 22); ++i) {
        if (mbar_try(bar, parity)) return true;
        if (i > 64) { __nanosleep(64); if (*abort_flag) return false; }
    }
    return false;
}
// a plain store: the word lies in host memory (only ever written on the way out of a wait that gave up)
__device__ __forceinline__ void report_wait(int* status, int code) { *(volatile int*)status = code; __threadfence_system(); }
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const void* tmap, uint32_t bar, int c0, int c1) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
                 ::"r"(dst), "l"(tmap), "r"(bar), "r"(c0), "r"(c1) : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const void* tmap, uint32_t bar, int c0, int c1, int c2) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
                 ::"r"(dst), "l"(tmap), "r"(bar), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const void* tmap, uint32_t bar, int c0, int c1, int c2, int c3) {
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
                 ::"r"(dst), "l"(tmap), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
// Shared-memory matrix descriptor, 128-byte swizzle: start >> 4 | leading-dimension offset >> 4 at bit 16 | stride-dimension
// offset >> 4 at bit 32 | version 1 at bit 46 | swizzle mode 2 (128 bytes) at bit 61.  The base-offset field (bit 49) stays 0:
// the tensor core derives the XOR phase of a row from the row's absolute shared-memory address, exactly as TMA wrote it, so a
// start address moved by whole 128-byte rows needs nothing else (measured: with the row phase in the field the taps read the
// wrong 16-byte chunks).
__device__ __forceinline__ uint64_t desc_sw128(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* v) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
                 "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
                   "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]),
                   "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]),
                   "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                 : "r"(taddr));
}
__device__ __forceinline__ int floor_div(int a, int b) { int q = a / b; if ((a % b != 0) && ((a < 0) != (b < 0))) --q; return q; }
__device__ __forceinline__ void tma_store_2d(const void* tmap, uint32_t src, int c0, int c1) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(tmap), "r"(src), "r"(c0), "r"(c1) : "memory");
}
__device__ __forceinline__ void bar_sync_epi(int id) { asm volatile("bar.sync %0, 128;" ::"r"(id) : "memory"); }   // the four warps of one epilogue group
__device__ __forceinline__ bool bar_and_epi(int id, bool v) {     // barrier of the four warps of an epilogue group that also ANDs a flag
    uint32_t r;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %2, 0;\n\tbar.red.and.pred q, %1, 128, p;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(r) : "r"(id), "r"((uint32_t)v) : "memory");
    return r != 0;
}
__device__ __forceinline__ void bulk_wait_read(int pending) {     // at most `pending` of this thread's latest bulk stores may still be reading shared memory
    if (pending <= 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    else if (pending == 1) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
    else asm volatile("cp.async.bulk.wait_group.read 2;" ::: "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t a) { uint4 v; asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a)); return v; }
__device__ __forceinline__ void sts128(uint32_t a, uint4 v) { asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory"); }
__device__ __forceinline__ uint32_t lds32(uint32_t a) { uint32_t v; asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(a)); return v; }

// two fp32 operations per instruction
__device__ __forceinline__ uint64_t f2_pack(uint32_t lo, uint32_t hi) { uint64_t r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi)); return r; }
__device__ __forceinline__ void f2_unpack(uint64_t v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) { uint64_t r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) { uint64_t r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) { uint64_t r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ uint64_t f2_of_bf16x2(uint32_t w) { return f2_pack(w << 16, w & 0xFFFF0000u); }
__device__ __forceinline__ uint32_t bf16x2_of_f2(uint64_t v) { float lo, hi; f2_unpack(v, lo, hi); __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi); return *reinterpret_cast<uint32_t*>(&h); }

// A thread's 32 columns of a tile: accumulator * scale (+ residual: RES from the staging slab it goes back to, GADD from registers),
// rounded, into the staging slab; BN: relu(bn(.)) of the rounded value into a second slab.  st / st2: shared address of the row with the
// row's swizzle phase folded in (a 16-byte chunk is st ^ chunk * 16); scale2: the scale twice, 0 for a position outside the map (whose sum
// is of no pixel).  The kernel's epilogue is bound by instructions, not by the stores (skipping them changed nothing), hence the packed
// arithmetic and one instance per kind.
template <bool RES, bool GADD, bool BN>
__device__ __forceinline__ void epi_cols(const uint32_t* v, uint32_t st, uint32_t st2, int chunk0, uint64_t scale2, const uint4* ga, const float4* bnc) {
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        const uint32_t so = (uint32_t)(chunk0 + g) << 4;
        uint32_t w[4];
        if (RES || GADD) {
            const uint4 a = RES ? lds128(st ^ so) : ga[g];
            const uint32_t aw[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) w[k] = bf16x2_of_f2(f2_fma(f2_pack(v[g * 8 + 2 * k], v[g * 8 + 2 * k + 1]), scale2, f2_of_bf16x2(aw[k])));
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) w[k] = bf16x2_of_f2(f2_mul(f2_pack(v[g * 8 + 2 * k], v[g * 8 + 2 * k + 1]), scale2));
        }
        sts128(st ^ so, make_uint4(w[0], w[1], w[2], w[3]));
        if (BN) {                                                // evaluation: with running statistics
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float4 q0 = bnc[g * 8 + 2 * k], q1 = bnc[g * 8 + 2 * k + 1];
                const float z0 = (__uint_as_float(w[k] << 16) - q0.x) * q0.y * q0.z + q0.w, z1 = (__uint_as_float(w[k] & 0xFFFF0000u) - q1.x) * q1.y * q1.z + q1.w;
                __nv_bfloat162 hh = __floats2bfloat162_rn(z0 > 0.f ? z0 : 0.f, z1 > 0.f ? z1 : 0.f);
                w[k] = *reinterpret_cast<uint32_t*>(&hh);
            }
            sts128(st2 ^ so, make_uint4(w[0], w[1], w[2], w[3]));
        }
    }
}

constexpr int TC_THREADS = 224;              // wgrad kernel: producer warp of dy, MMA warp, producer warp of a, four epilogue warps
constexpr int TC_ISSUERS = 1;                // forward / dgrad kernel: MMA-issuing warps
constexpr int TC_RES_WARP = 1 + TC_ISSUERS + 8;              // forward / dgrad kernel: fetches the residual
constexpr int TC_CONV_THREADS = 32 * (TC_RES_WARP + 1);          // producer warp, MMA warps, two groups of four epilogue warps, residual warp
constexpr int TC_MAX_EB = 4;                                     // 16 KB staging slabs per epilogue group
constexpr int TC_MAX_STAGES = 12;
constexpr int TILE_M = 128;
constexpr int SLAB_BYTES = TILE_M * 128;      // 128 rows x 64 channels of bf16

struct TapRef { int wtap; int shift; };       // weight tap index (r*ksz + s); row shift of the operand inside the window
// One forward / dgrad problem.  The tensor maps come first so that each is 64-byte aligned.
//
// Positions and windows.  The positions of a problem are either the pixels of the output in order ("dense": 1x1 layers) or a
// tall map of Hp x Wp positions per image with `pad` zero rows before each image and `pad` zero columns after each row (3x3
// layers).  A tile is 128 consecutive positions [p0, p0 + 128).  Its operand for one tap group is a window of positions
// [p0 - hb, ...) fetched once per 64-channel slab; tap t of the group reads the window from row (p0 - hb - window start) +
// shift[t] on.  Window position (image, yy, xx) holds activation pixel ((yy - pad) * es + gys, xx * es + gxs) of that
// image, zero outside it: es = 2 with one group per input parity phase makes a stride-2 layer exact work (forward), and four
// problems, one per output phase, do the same for a stride-2 dgrad.
struct TcHot {                // everything the kernel's loops read: each role keeps a copy in shared memory
    const __nv_bfloat16* add; __nv_bfloat16* out;
    float* stat_tiles;        // [tiles_m][2][ncol]: column sums of the stored tile (of y and y^2, or with bwd_x of dz and dz * xhat), or nullptr
    const __nv_bfloat16* bwd_x;   // dgrad whose output feeds a BN+ReLU backward: input of that BN (constants in bn_stat, bn_gamma, bn_beta)
    int* status;
    const float* bn_stat; const float* bn_gamma; const float* bn_beta; __nv_bfloat16* bn_out;   // evaluation: bn_out = relu(bn(y)) with mean | 1/std in bn_stat; nullptr otherwise
    int store_y;              // 0: only bn_out is wanted
    int res_tma;              // 1: the residual comes through map_add
    int a_flat;               // 1: a window is one box of 128 pixels of the (channel, pixel) map
    int dense;                // 1: position index == output pixel index
    int add_mode;             // 0 none; 2 residual read at the output pixel; 3 residual read from a compact tensor that applies at even (y, x) only
    int ngroups; int gbeg[5]; int gxs[4], gys[4];
    int wtap[9], shift[9];    // per tap: weight tap index (r*ksz + s); row shift of the operand inside the window
    int es, pad;
    int Hp, Wp, n_img;
    int R, box_pos, nbox, hb, a_box_bytes;
    int tiles_m, tiles_n, n_tile, ncol;      // output tile grid; MMA N; channels of the output tensor
    int red, slabs;                          // reduction channels, 64-channel slabs
    int b_mn_major;                          // 0: forward (weights K-major); 1: dgrad (weights MN-major)
    int b_bytes;                             // bytes of one weight tile (one slab, one tap)
    int out_slabs;                           // 64-column slabs of the output tile
    int total_pos;
    float scale;
    int OH, OW, os, oy, ox;                  // position (image, yy, xx) -> output pixel ((yy - pad) * os + oy, xx * os + ox) of an OH x OW image
};
struct alignas(64) TcProb {
    CUtensorMap map_a;        // activations (forward: a; dgrad: dy): (channel, pixel) or (channel, x, y, image), possibly element-strided
    CUtensorMap map_b;        // weights [K][taps][C] viewed as (C, tap, K)
    CUtensorMap map_out;      // dense problems: the output as (channel, pixel), box 64 x 32 (one warp's rows of a slab)
    CUtensorMap map_bn;       // likewise bn_out
    CUtensorMap map_add;      // dense problems: the residual, box 64 x 128
    TcHot h;
};
static_assert(sizeof(TcHot) % 4 == 0, "copied word by word");

struct TcLaunch { int nprob, na, nb, a_stage, b_stage, tmem_cols, acc_stride, nbuf, groups, eb, res; };
// nbuf: accumulators per tile of a pair (2: the next pair's MMAs run under this pair's epilogues); groups: epilogue groups (one per tile
// of a pair); eb: 16 KB staging buffers (one 64-column slab each) per group; res: the staging buffers come through the residual warp
constexpr int TC_MAX_PROBS = 128;             // descriptors per launch (sub-ResNets x output phases)

__device__ __forceinline__ void copy_hot(TcHot* dst, const TcHot* src, int tid, int nthreads) {
    const uint32_t* s4 = reinterpret_cast<const uint32_t*>(src); uint32_t* d4 = reinterpret_cast<uint32_t*>(dst);
    for (int i = tid; i < (int)(sizeof(TcHot) / 4); i += nthreads) d4[i] = __ldg(s4 + i);
}

// BWD: the instance of dgrad launches (sums of the BN backward, no BN of the output); the other one is forward's and evaluation's.
template <bool BWD>
__global__ void __launch_bounds__(TC_CONV_THREADS, 1) conv_tc_kernel(const TcProb* __restrict__ probs, const TcLaunch L) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t bars[4 * TC_MAX_STAGES + 10 + 4 * TC_MAX_EB];
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s;
    __shared__ __align__(16) float stat_s2[2][4][2][256];
    __shared__ __align__(16) float bwd_s2[BWD ? 2 : 1][4][BWD ? 256 : 4];   // per group: -mean, 1/std, gamma, beta of the column tile (from L2 they cost a slab 1000 clocks)
    __shared__ int unit_end_s[TC_MAX_PROBS];                      // running sum of the problems' unit counts (a unit: two row tiles x one column tile)
    __shared__ int tilesm_s[TC_MAX_PROBS], tilesn_s[TC_MAX_PROBS];
    __shared__ TcHot hot_s[3 + TC_ISSUERS];                   // the current problem of the producer, the two epilogue groups, the MMA issuer
    const uint32_t a_full = smem_u32(&bars[0]), a_empty = smem_u32(&bars[TC_MAX_STAGES]);
    const uint32_t b_full = smem_u32(&bars[2 * TC_MAX_STAGES]), b_empty = smem_u32(&bars[3 * TC_MAX_STAGES]);
    const uint32_t acc_full = smem_u32(&bars[4 * TC_MAX_STAGES]), acc_empty = smem_u32(&bars[4 * TC_MAX_STAGES + 4]);
    const uint32_t drain = smem_u32(&bars[4 * TC_MAX_STAGES + 8]);
    const uint32_t res_full = smem_u32(&bars[4 * TC_MAX_STAGES + 10]), res_empty = smem_u32(&bars[4 * TC_MAX_STAGES + 10 + 2 * TC_MAX_EB]);   // [group][slab buffer]
    const uint32_t a_ring = smem_u32(smem), b_ring = a_ring + (uint32_t)(L.na * L.a_stage), stg_base = b_ring + (uint32_t)(L.nb * L.b_stage);
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // warp-uniform for the compiler too

    if (threadIdx.x == 0) {
        for (int s = 0; s < TC_MAX_STAGES; ++s) {
            mbar_init(a_full + 8 * s, 1); mbar_init(a_empty + 8 * s, 1); mbar_init(b_full + 8 * s, 1); mbar_init(b_empty + 8 * s, 1);
        }
        for (int s = 0; s < 4; ++s) { mbar_init(acc_full + 8 * s, 1); mbar_init(acc_empty + 8 * s, 4); }
        mbar_init(drain, 1);
        for (int s = 0; s < 2 * TC_MAX_EB; ++s) { mbar_init(res_full + 8 * s, 1); mbar_init(res_empty + 8 * s, 4); }
        abort_s = 0;
        int run = 0;
        for (int i = 0; i < L.nprob; ++i) {
            const TcHot* hp = &probs[i].h;
            run += ((hp->tiles_m + 1) >> 1) * hp->tiles_n; unit_end_s[i] = run;
            tilesm_s[i] = hp->tiles_m; tilesn_s[i] = hp->tiles_n;
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(L.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    chain_wait();                                                // from here on: tensors the previous kernel may have written or read
    const uint32_t tmem_base = tmem_base_s;
    // A unit of work is a pair of neighbouring row tiles (2 x 128 positions) times one column tile: the two tiles share every weight
    // tile, which is fetched once, and each has its own accumulator.  The units of all problems, column tile innermost, are dealt round-robin: the
    // CTAs that run side by side work on neighbouring tiles, share windows and weight tiles in L2 and read HBM as one moving front.
    // (Contiguous runs per CTA, with the column tile outermost, were measured too: no faster, and slower where the weights stream.)
    // The last, partial wave: when at most half of the CTAs would get a pair of it, its pairs are split into single tiles (a pair of 256
    // columns over 2304 reduction channels is 19 us of a launch of 60).
    const int u_total = unit_end_s[L.nprob - 1], u_step = (int)gridDim.x, u_begin = (int)blockIdx.x;
    const int u_full = u_total / u_step * u_step, u_rest = u_total - u_full;
    const int u_split = 2 * u_rest <= u_step ? u_full : u_total, u_stop = u_split + 2 * (u_total - u_split);
    struct Unit { int pi, tn, tm0, nt; };                        // problem, column tile, first row tile, row tiles (0: nothing to do)
    auto decode = [&](int u) {
        int half = -1;
        if (u >= u_split) { half = (u - u_split) & 1; u = u_split + ((u - u_split) >> 1); }
        Unit r; r.pi = 0; while (u >= unit_end_s[r.pi]) ++r.pi;
        const int loc = u - (r.pi ? unit_end_s[r.pi - 1] : 0), tiles_n = tilesn_s[r.pi];
        r.tm0 = 2 * (loc / tiles_n); r.tn = loc - (r.tm0 >> 1) * tiles_n;
        r.nt = r.tm0 + 1 < tilesm_s[r.pi] ? 2 : 1;
        if (half >= 0) { r.nt = half < r.nt ? 1 : 0; r.tm0 += half; }
        return r;
    };

    if (warp == 0) {
        // ---------------------------------------------------------------- TMA producer
        if (elect_one()) {
            uint32_t a_cnt = 0, b_cnt = 0; bool ok = true;
            int cur = -1; TcHot& h = hot_s[0];
            int sa = 0, sb_ = 0; uint32_t pha = 0, phb = 0;       // ring positions and phases
            for (int u = u_begin; u < u_stop && ok; u += u_step) {
                const Unit un = decode(u);
                if (!un.nt) continue;
                const int pi = un.pi, tn = un.tn, tm0 = un.tm0, nt = un.nt;
                if (pi != cur) { copy_hot(&h, &probs[pi].h, 0, 1); cur = pi; }
                const TcProb* pp = probs + pi;
                const int n_tile = h.n_tile, slabs = h.slabs, ngroups = h.ngroups, a_flat = h.a_flat, nbox = h.nbox,
                          a_box_bytes = h.a_box_bytes, R = h.R, Hp = h.Hp, pad = h.pad, es = h.es, b_bytes = h.b_bytes, mn = h.b_mn_major;
                // first box of each tile's window: its image and its first tall row in that image (a box is rows of one image, or whole images)
                int img0[2] = {0, 0}, row0[2] = {0, 0};
                const int box_img = R > Hp ? R / max(Hp, 1) : 1, box_row = R > Hp ? Hp : R;
                if (!a_flat)
                    for (int j = 0; j < nt; ++j) { const int trow = floor_div((tm0 + j) * TILE_M - h.hb, h.box_pos) * R; img0[j] = floor_div(trow, Hp); row0[j] = trow - img0[j] * Hp; }
                for (int sl = 0; sl < slabs && ok; ++sl) {
                    for (int g = 0; g < ngroups && ok; ++g) {
                        const int gx = h.gxs[g], gy = h.gys[g], t_end = h.gbeg[g + 1];
                        for (int j = 0; j < nt; ++j) {
                            const uint32_t dst = a_ring + (uint32_t)(sa * L.a_stage), full = a_full + 8 * sa;
                            if (!mbar_wait(a_empty + 8 * sa, pha ^ 1u, &abort_s)) { atomicExch(&abort_s, 1); report_wait(h.status, 1); ok = false; break; }
                            mbar_expect_tx(full, (uint32_t)(nbox * a_box_bytes));
                            if (a_flat) tma_load_2d(dst, &pp->map_a, full, sl * 64, (tm0 + j) * TILE_M);
                            else {
                                int img = img0[j], yy = row0[j];
                                for (int i = 0; i < nbox; ++i) {
                                    tma_load_4d(dst + (uint32_t)(i * a_box_bytes), &pp->map_a, full, sl * 64, gx, (yy - pad) * es + gy, img);
                                    yy += box_row; if (yy >= Hp) { yy = 0; img += box_img; }
                                }
                            }
                            ++a_cnt; if (++sa == L.na) { sa = 0; pha ^= 1u; }
                        }
                        if (!ok) break;
                        for (int tap = h.gbeg[g]; tap < t_end; ++tap) {
                            const uint32_t dst = b_ring + (uint32_t)(sb_ * L.b_stage), full = b_full + 8 * sb_;
                            const int wtap = h.wtap[tap];
                            if (!mbar_wait(b_empty + 8 * sb_, phb ^ 1u, &abort_s)) { atomicExch(&abort_s, 1); report_wait(h.status, 2); ok = false; break; }
                            mbar_expect_tx(full, (uint32_t)b_bytes);
                            if (!mn) tma_load_3d(dst, &pp->map_b, full, sl * 64, wtap, tn * n_tile);
                            else for (int c = 0; c * 64 < n_tile; ++c)
                                tma_load_3d(dst + (uint32_t)(c * 8192), &pp->map_b, full, tn * n_tile + c * 64, wtap, sl * 64);
                            ++b_cnt; if (++sb_ == L.nb) { sb_ = 0; phb ^= 1u; }
                        }
                    }
                }
            }
            if (!ok) {
                // another role gave up (or this one): wait, bounded, for the copies still in flight before the CTA leaves
                for (uint32_t c = a_cnt > (uint32_t)L.na ? a_cnt - L.na : 0; c < a_cnt; ++c)
                    for (int i = 0; i < 4096 && !mbar_try(a_full + 8 * (c % L.na), (c / L.na) & 1u); ++i) __nanosleep(64);
                for (uint32_t c = b_cnt > (uint32_t)L.nb ? b_cnt - L.nb : 0; c < b_cnt; ++c)
                    for (int i = 0; i < 4096 && !mbar_try(b_full + 8 * (c % L.nb), (c / L.nb) & 1u); ++i) __nanosleep(64);
            }
        }
    } else if (warp == 1) {
        // ---------------------------------------------------------------- MMA issuer: the reductions of both tiles of a pair, each into its own
        // accumulator.  (Everything the inner loops need sits in registers: between two asm statements the compiler would
        // fetch a field of the shared descriptor again every time.)
        if (elect_one()) {
            uint32_t cnt[2] = {0u, 0u}; bool ok = true;
            int cur = -1; TcHot& h = hot_s[3];
            int sa = 0, sb = 0; uint32_t pha = 0, phb = 0;
            const uint32_t nbuf1 = (uint32_t)L.nbuf - 1u;
            // upper half of a 128-byte-swizzle descriptor: stride between 8-row groups 1024 bytes, version, swizzle mode; the lower half is the
            // start address | leading-dimension offset << 16, both in 16-byte units
            const uint32_t desc_hi = (uint32_t)(desc_sw128(0, 0, 1024) >> 32), a_lbo = 1u << 16;
            for (int u = u_begin; u < u_stop && ok; u += u_step) {
                const Unit un = decode(u);
                if (!un.nt) continue;
                const int nt = un.nt;
                if (un.pi != cur) { copy_hot(&h, &probs[un.pi].h, 0, 1); cur = un.pi; }
                const int slabs = h.slabs, ngroups = h.ngroups, red = h.red, mn = h.b_mn_major, a_flat = h.a_flat, hb = h.hb, box_pos = h.box_pos;
                uint32_t a_off[2], d_tmem[2], full_bar[2];
                for (int j = 0; j < nt; ++j) {
                    const int p0 = (un.tm0 + j) * TILE_M - hb;
                    a_off[j] = a_flat ? 0u : (uint32_t)(p0 - floor_div(p0, box_pos) * box_pos) * 8u;
                    const uint32_t buf = (cnt[j] & nbuf1) * 2u + (uint32_t)j, aph = (cnt[j] >> nbuf1) & 1u;
                    ++cnt[j];
                    d_tmem[j] = tmem_base + buf * (uint32_t)L.acc_stride; full_bar[j] = acc_full + 8 * buf;
                    if (!mbar_wait(acc_empty + 8 * buf, aph ^ 1u, &abort_s)) { atomicExch(&abort_s, 1); report_wait(h.status, 3); ok = false; break; }
                }
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                // instruction descriptor: fp32 accumulate, bf16 x bf16, A K-major, B K-major or MN-major, N, M = 128
                const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)mn << 16) | ((uint32_t)(h.n_tile >> 3) << 17) | ((128u >> 4) << 24);
                const uint32_t b_lbo = mn ? (8192u >> 4) << 16 : 1u << 16;
                const uint32_t b_step = mn ? 128u : 2u;           // one K = 16 step: 16 rows of 128 bytes (MN-major) or 32 bytes along the row (K-major), in 16-byte units
                uint32_t acc = 0;
                for (int sl = 0; sl < slabs && ok; ++sl) {
                    const int ksteps = (min(64, red - sl * 64) + 15) >> 4;
                    for (int g = 0; g < ngroups && ok; ++g) {
                        uint32_t a_lo[2], a_rel[2];
                        const int t_end = h.gbeg[g + 1];
                        for (int j = 0; j < nt; ++j) {
                            if (!mbar_wait(a_full + 8 * sa, pha, &abort_s)) { atomicExch(&abort_s, 1); report_wait(h.status, 4); ok = false; break; }
                            a_lo[j] = (((a_ring + (uint32_t)(sa * L.a_stage)) >> 4) + a_off[j]) | a_lbo; a_rel[j] = a_empty + 8 * sa;
                            if (++sa == L.na) { sa = 0; pha ^= 1u; }
                        }
                        for (int tap = h.gbeg[g]; tap < t_end && ok; ++tap) {
                            const uint32_t shift = (uint32_t)h.shift[tap] * 8u, b_lo = ((b_ring + (uint32_t)(sb * L.b_stage)) >> 4) | b_lbo;
                            if (!mbar_wait(b_full + 8 * sb, phb, &abort_s)) { atomicExch(&abort_s, 1); report_wait(h.status, 5); ok = false; break; }
#pragma unroll
                            for (int j = 0; j < 2; ++j) {
                                if (j >= nt) break;
                                if (ksteps == 4) {
#pragma unroll
                                    for (int k16 = 0; k16 < 4; ++k16)
                                        umma_bf16(d_tmem[j], f2_pack(a_lo[j] + shift + 2u * (uint32_t)k16, desc_hi), f2_pack(b_lo + b_step * (uint32_t)k16, desc_hi), idesc, k16 ? 1u : acc);
                                } else
                                    for (int k16 = 0; k16 < ksteps; ++k16)
                                        umma_bf16(d_tmem[j], f2_pack(a_lo[j] + shift + 2u * (uint32_t)k16, desc_hi), f2_pack(b_lo + b_step * (uint32_t)k16, desc_hi), idesc, k16 ? 1u : acc);
                            }
                            acc = 1;
                            umma_commit(b_empty + 8 * sb);       // released once these MMAs have read the weight tile
                            if (++sb == L.nb) { sb = 0; phb ^= 1u; }
                        }
                        if (ok) for (int j = 0; j < nt; ++j) umma_commit(a_rel[j]);
                    }
                }
                if (ok) for (int j = 0; j < nt; ++j) umma_commit(full_bar[j]);   // accumulators complete
            }
            if (!ok) {
                // gave up: the MMAs already issued must have finished before the CTA frees its tensor memory
                umma_commit(drain);
                for (int i = 0; i < 65536 && !mbar_try(drain, 0u); ++i) __nanosleep(64);
            }
        }
    } else if (warp == TC_RES_WARP) {
        // ---------------------------------------------------------------- residual of dense problems: its 128 x 64 boxes go straight into
        // the staging slabs the epilogue will add to and store from, up to L.eb slabs ahead per group
        if (L.res && elect_one()) {
            bool ok = true; uint32_t q[2] = {0u, 0u};
            for (int u = u_begin; u < u_stop && ok; u += u_step) {
                const Unit un = decode(u);
                if (!un.nt) continue;
                const TcHot* hp = &probs[un.pi].h;
                const int load = __ldg(&hp->res_tma), out_slabs = __ldg(&hp->out_slabs), col0 = un.tn * __ldg(&hp->n_tile);
                for (int sl = 0; sl < out_slabs && ok; ++sl)
                    for (int j = 0; j < un.nt; ++j) {
                        const uint32_t sb = (uint32_t)j * TC_MAX_EB + q[j] % (uint32_t)L.eb;
                        if (!mbar_wait(res_empty + 8 * sb, ((q[j] / (uint32_t)L.eb) & 1u) ^ 1u, &abort_s)) { atomicExch(&abort_s, 1); report_wait(probs[un.pi].h.status, 7); ok = false; break; }
                        if (!load) mbar_arrive(res_full + 8 * sb);           // a problem without residual in the same launch only passes through the ring
                        else { mbar_expect_tx(res_full + 8 * sb, (uint32_t)SLAB_BYTES);
                        tma_load_2d(stg_base + ((uint32_t)(j * L.eb) + q[j] % (uint32_t)L.eb) * SLAB_BYTES, &probs[un.pi].map_add, res_full + 8 * sb, col0 + sl * 64, (un.tm0 + j) * TILE_M); }
                        ++q[j];
                    }
            }
            if (!ok)
                for (int j = 0; j < 2; ++j)
                    for (uint32_t c = q[j] > (uint32_t)L.eb ? q[j] - L.eb : 0; c < q[j]; ++c)
                        for (int i = 0; i < 4096 && !mbar_try(res_full + 8 * ((uint32_t)j * TC_MAX_EB + c % (uint32_t)L.eb), (c / (uint32_t)L.eb) & 1u); ++i) __nanosleep(64);
        }
    } else {
        // ---------------------------------------------------------------- epilogue: two groups of 4 warps (one TMEM lane quadrant each);
        // group g takes tile g of every pair.  Inside a tile the warps do not wait for one another: each stages and stores its own
        // 32 rows, slab by slab of 64 columns, through its quarter of the group's slab buffers.
        const int grp = (warp - 1 - TC_ISSUERS) >> 2, bid = 1 + grp;
        const int quad = warp & 3;
        const int m = quad * 32 + lane;                          // row of the tile = TMEM lane
        const int et = threadIdx.x - 32 * (1 + TC_ISSUERS) - grp * 128;   // 0..127 among the group's threads
        float (*const stat_s)[2][256] = stat_s2[grp];
        float4* const bnc_s = reinterpret_cast<float4*>(&stat_s2[grp][0][0][0]);   // evaluation keeps no statistics: mean, 1/std, gamma, beta per column
        bool ok = true;
        int cur = -1, cur_tn = -1; const TcHot& h = hot_s[1 + grp];
        uint32_t sc = 0, cnt = 0;                                // slabs staged; tiles taken
        const uint32_t eb = (uint32_t)L.eb, lag = eb >= 3u ? 2u : 1u;   // a slab is handed back to the residual warp when the store `lag` slabs later is due
        for (int u = u_begin; u < u_stop; u += u_step) {
            const Unit un = decode(u);
            if (grp >= un.nt) continue;
            const int pi = un.pi, tn = un.tn, tm = un.tm0 + grp;
            const TcProb* pp = probs + pi;
            const uint32_t buf = (cnt % (uint32_t)L.nbuf) * 2u + (uint32_t)grp, aph = (cnt / (uint32_t)L.nbuf) & 1u;
            ++cnt;
            if (pi != cur || ((h.bn_out || h.bwd_x) && tn != cur_tn)) {   // every warp of the group is through with the last problem's constants
                bar_sync_epi(bid);
                if (pi != cur) copy_hot(&hot_s[1 + grp], &probs[pi].h, et, 128);
                bar_sync_epi(bid);
                if (h.bn_out) {
                    for (int c = et; c < h.n_tile; c += 128) {
                        const int g = min(tn * h.n_tile + c, h.ncol - 1);
                        bnc_s[c] = make_float4(__ldg(h.bn_stat + g), __ldg(h.bn_stat + h.ncol + g), __ldg(h.bn_gamma + g), __ldg(h.bn_beta + g));
                    }
                    bar_sync_epi(bid);
                }
                if (BWD && h.bwd_x) {
                    float (*const w)[256] = reinterpret_cast<float (*)[256]>(&bwd_s2[BWD ? grp : 0][0][0]);
                    for (int c = et; c < h.n_tile; c += 128) {
                        const int g = min(tn * h.n_tile + c, h.ncol - 1);
                        w[0][c] = -__ldg(h.bn_stat + g); w[1][c] = __ldg(h.bn_stat + h.ncol + g); w[2][c] = __ldg(h.bn_gamma + g); w[3][c] = __ldg(h.bn_beta + g);
                    }
                    bar_sync_epi(bid);
                }
                cur = pi; cur_tn = tn;
            }
            const int n_tile = h.n_tile, ncol = h.ncol, add_mode = h.add_mode, dense = h.dense, res_tma = h.res_tma, store_y = h.store_y;
            const float scale = h.scale;
            const __nv_bfloat16* addp = h.add; __nv_bfloat16* outp = h.out; float* stat_tiles = h.stat_tiles; __nv_bfloat16* bn_out = BWD ? nullptr : h.bn_out;
            // position -> output pixel (and the residual's pixel)
            long long addpix = -1;
            auto pixel_of = [&](int pos) -> int {                // -1: a padding position; sets addpix of a compact residual
                addpix = -1;
                if (pos >= h.total_pos) return -1;
                if (dense && add_mode != 3) return pos;
                const int Wp = h.Wp, Hp = h.Hp, pad = h.pad, os = h.os, OH = h.OH, OW = h.OW;
                const int trow = pos / Wp, xx = pos - trow * Wp, img = trow / Hp, yy = trow - img * Hp;
                const int y = (yy - pad) * os + h.oy, x = xx * os + h.ox;
                if (!(yy >= pad && xx < Wp - pad && y < OH && x < OW)) return -1;
                if (add_mode == 3 && !((y | x) & 1)) addpix = ((long long)img * ((OH + 1) >> 1) + (y >> 1)) * ((OW + 1) >> 1) + (x >> 1);
                return (img * OH + y) * OW + x;
            };
            const int pix = pixel_of(tm * TILE_M + m);
            const bool valid = pix >= 0;
            if (add_mode == 2) addpix = pix;
            const int col0 = tn * n_tile;
            const bool gadd = !res_tma && add_mode >= 2 && valid && addpix >= 0;
            // a residual that TMA cannot bring: the first slab's is read ahead of the accumulator, a later one's once the last has been used
            const __nv_bfloat16* addrow = addp + (gadd ? addpix : 0) * ncol + col0;
            uint4 ga[8];
            auto load_add = [&](int c0) {                        // the 64 columns of a slab
#pragma unroll
                for (int g = 0; g < 8; ++g) { const int c = c0 + g * 8; ga[g] = (gadd && c < n_tile && col0 + c < ncol) ? __ldg(reinterpret_cast<const uint4*>(addrow + c)) : make_uint4(0u, 0u, 0u, 0u); }
            };
            const bool any_gadd = !res_tma && add_mode >= 2;
            if (any_gadd) load_add(0);
            // BN backward: lane (row group lane >> 3, chunk lane & 7) reads x the way the copy-out writes, a slab ahead of its use
            const __nv_bfloat16* bwd_x = BWD ? h.bwd_x : nullptr;
            uint4 xr[8];
            auto load_x = [&](int s0) {
                const int c = s0 + (lane & 7) * 8;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int px = __shfl_sync(0xffffffffu, pix, i * 4 + (lane >> 3));
                    xr[i] = (px >= 0 && c < n_tile && col0 + c < ncol) ? __ldg(reinterpret_cast<const uint4*>(bwd_x + (long long)px * ncol + col0 + c)) : make_uint4(0u, 0u, 0u, 0u);
                }
            };
            if (bwd_x) {
                load_x(0);
                // the rows of the group's next tile are asked into L2 now, a whole tile ahead of their use: the epilogue is the limit of the 1x1 layers,
                // and the little L1 beside 225 KB of shared memory (which layers: conv_tc_bwd_sums)
                const Unit nx = u + u_step < u_stop ? decode(u + u_step) : Unit{-1, 0, 0, 0};
                if (nx.pi == pi && grp < nx.nt) {
                    const int px2 = pixel_of((nx.tm0 + grp) * TILE_M + m);
                    if (px2 >= 0)
                        for (int c = nx.tn * n_tile; c < min((nx.tn + 1) * n_tile, ncol); c += 64) asm volatile("prefetch.global.L2 [%0];" ::"l"(bwd_x + (long long)px2 * ncol + c));
                }
            }
            const uint32_t scw = __float_as_uint(valid ? scale : 0.f);
            const uint64_t scale2 = f2_pack(scw, scw);
            ok = mbar_wait(acc_full + 8 * buf, aph, &abort_s);
            __syncwarp();
            ok = bar_and_epi(bid, ok);                           // one decision for the four warps: they share the group's barriers
            if (!ok) { atomicExch(&abort_s, 1); report_wait(h.status, 6); break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t t_row = tmem_base + buf * (uint32_t)L.acc_stride + ((uint32_t)(quad * 32) << 16);
            for (int s0 = 0; s0 < n_tile; s0 += 64) {
                const uint32_t sbuf = sc % eb;
                const uint32_t stg = stg_base + ((uint32_t)grp * eb + sbuf) * SLAB_BYTES, stg2 = stg_base + ((uint32_t)L.groups * eb + (uint32_t)grp) * SLAB_BYTES;
                if (elect_one()) {                               // the store last issued from this buffer has been read (with a BN: from the group's BN buffer too)
                    bulk_wait_read(bn_out ? 0 : L.res ? (int)lag - 1 : (int)eb - 1);
                    if (L.res && sc >= lag) mbar_arrive(res_empty + 8 * ((uint32_t)grp * TC_MAX_EB + (sc - lag) % eb));
                }
                __syncwarp();
                if (L.res && !mbar_wait(res_full + 8 * ((uint32_t)grp * TC_MAX_EB + sbuf), (sc / eb) & 1u, &abort_s)) { atomicExch(&abort_s, 1); report_wait(h.status, 8); }
                __syncwarp();
                ++sc;
                // 64 columns, or 32 if the tile ends there: columns past the tile's own are never stored (n_tile is a multiple of 64 or covers
                // all of the tensor's columns)
                const uint32_t st = (stg + (uint32_t)m * 128u) ^ ((uint32_t)(m & 7) << 4), st2 = (stg2 + (uint32_t)m * 128u) ^ ((uint32_t)(m & 7) << 4);
                const bool two = s0 + 32 < n_tile;
                uint32_t v[2][32];
                tmem_ld32(t_row + (uint32_t)s0, v[0]);
                if (two) tmem_ld32(t_row + (uint32_t)(s0 + 32), v[1]);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (s0 + 64 >= n_tile) {
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(acc_empty + 8 * buf); // this warp has read its quadrant of the accumulator
                }
                const float4* bq = bnc_s + s0;
                if (!bn_out && res_tma) { epi_cols<true, false, false>(v[0], st, st2, 0, scale2, ga, bq); if (two) epi_cols<true, false, false>(v[1], st, st2, 4, scale2, ga, bq); }
                else if (!bn_out && !any_gadd) { epi_cols<false, false, false>(v[0], st, st2, 0, scale2, ga, bq); if (two) epi_cols<false, false, false>(v[1], st, st2, 4, scale2, ga, bq); }
                else if (!bn_out) { epi_cols<false, true, false>(v[0], st, st2, 0, scale2, ga, bq); if (two) epi_cols<false, true, false>(v[1], st, st2, 4, scale2, ga + 4, bq); }
                else if (res_tma) { epi_cols<true, false, true>(v[0], st, st2, 0, scale2, ga, bq); if (two) epi_cols<true, false, true>(v[1], st, st2, 4, scale2, ga, bq + 32); }
                else if (!any_gadd) { epi_cols<false, false, true>(v[0], st, st2, 0, scale2, ga, bq); if (two) epi_cols<false, false, true>(v[1], st, st2, 4, scale2, ga, bq + 32); }
                else { epi_cols<false, true, true>(v[0], st, st2, 0, scale2, ga, bq); if (two) epi_cols<false, true, true>(v[1], st, st2, 4, scale2, ga + 4, bq + 32); }
                if (any_gadd && s0 + 64 < n_tile) load_add(s0 + 64);
                if (dense) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the bulk store reads what this thread wrote
                __syncwarp();                                    // the warp's 32 rows of the slab are complete
                if (dense) {
                    if (elect_one()) {
                        if (store_y) tma_store_2d(&pp->map_out, stg + (uint32_t)quad * 4096u, col0 + s0, tm * TILE_M + quad * 32);
                        if (bn_out) tma_store_2d(&pp->map_bn, stg2 + (uint32_t)quad * 4096u, col0 + s0, tm * TILE_M + quad * 32);
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    }
                } else {
                    // copy-out of a tall slab: 16-byte chunks, eight consecutive lanes per 128-byte run of one output pixel
                    const int ch = lane & 7, c = s0 + ch * 8;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int row = i * 4 + (lane >> 3), px = __shfl_sync(0xffffffffu, pix, row);
                        if (px >= 0 && c < n_tile && col0 + c < ncol) {
                            const uint32_t so = (uint32_t)(quad * 32 + row) * 128u + ((uint32_t)(ch ^ (row & 7)) << 4);
                            if (store_y) *reinterpret_cast<uint4*>(outp + (long long)px * ncol + col0 + c) = lds128(stg + so);
                            if (bn_out) *reinterpret_cast<uint4*>(bn_out + (long long)px * ncol + col0 + c) = lds128(stg2 + so);
                        }
                    }
                }
                if (bwd_x) {
                    // the sums the BN backward needs, of the stored (rounded) da: dz = da where relu's input was positive, and dz * xhat.  A lane
                    // has 8 columns of 8 rows in fp32; the four lanes of a column group are added in double, each lane ending with four of the
                    // sixteen sums (half as many shuffles as a butterfly of all of them), the warps as below.
                    const int ch = lane & 7;
                    uint64_t nm[4], is[4], ga2[4], be2[4], su[4] = {0, 0, 0, 0}, sq[4] = {0, 0, 0, 0};
                    const uint32_t w0 = smem_u32(&bwd_s2[BWD ? grp : 0][0][0]) + (uint32_t)(s0 + ch * 8) * 4u;
#pragma unroll
                    for (int k = 0; k < 4; k += 2) {
                        const uint4 a = lds128(w0 + 8u * k), b = lds128(w0 + 1024u + 8u * k), g = lds128(w0 + 2048u + 8u * k), e = lds128(w0 + 3072u + 8u * k);
                        nm[k] = f2_pack(a.x, a.y); nm[k + 1] = f2_pack(a.z, a.w); is[k] = f2_pack(b.x, b.y); is[k + 1] = f2_pack(b.z, b.w);
                        ga2[k] = f2_pack(g.x, g.y); ga2[k + 1] = f2_pack(g.z, g.w); be2[k] = f2_pack(e.x, e.y); be2[k + 1] = f2_pack(e.z, e.w);
                    }
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int row = i * 4 + (lane >> 3);
                        const uint4 d = lds128(stg + (uint32_t)(quad * 32 + row) * 128u + ((uint32_t)(ch ^ (row & 7)) << 4));
                        const uint32_t dw[4] = {d.x, d.y, d.z, d.w}, xw[4] = {xr[i].x, xr[i].y, xr[i].z, xr[i].w};
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const uint64_t xh = f2_mul(f2_add(f2_of_bf16x2(xw[k]), nm[k]), is[k]);
                            float z0, z1; f2_unpack(f2_fma(xh, ga2[k], be2[k]), z0, z1);
                            const uint64_t dz = f2_of_bf16x2(dw[k] & ((z0 > 0.f ? 0x0000FFFFu : 0u) | (z1 > 0.f ? 0xFFFF0000u : 0u)));
                            su[k] = f2_add(su[k], dz); sq[k] = f2_fma(dz, xh, sq[k]);
                        }
                    }
                    if (s0 + 64 < n_tile) load_x(s0 + 64);
                    const bool sqs = lane & 8, hi = lane & 16;   // which kind of sum, and which four columns, this lane ends with
                    auto pair = [&](int k, double* d) {          // columns 2k and 2k + 1 over the lane and its neighbour by bit 3
                        const uint64_t other = __shfl_xor_sync(0xffffffffu, sqs ? su[k] : sq[k], 8), own = sqs ? sq[k] : su[k];
                        float a0, a1, b0, b1; f2_unpack(own, a0, a1); f2_unpack(other, b0, b1);
                        d[0] = (double)a0 + (double)b0; d[1] = (double)a1 + (double)b1;
                    };
                    float w[4];
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        double lo2[2], hi2[2]; pair(k, lo2); pair(k + 2, hi2);
#pragma unroll
                        for (int j = 0; j < 2; ++j) w[2 * k + j] = (float)((hi ? hi2[j] : lo2[j]) + __shfl_xor_sync(0xffffffffu, hi ? lo2[j] : hi2[j], 16));
                    }
                    *reinterpret_cast<float4*>(&stat_s[quad][sqs ? 1 : 0][s0 + ch * 8 + (hi ? 4 : 0)]) = make_float4(w[0], w[1], w[2], w[3]);
                } else if (stat_tiles) {
                    // column sums of the stored (rounded) values: every warp over its own 32 rows, lane = two neighbouring columns;
                    // the four warps' sums are added in a fixed order once the tile's last slab is through
                    uint64_t su = 0, sq = 0;
#pragma unroll 8
                    for (int r = 0; r < 32; ++r) {
                        const uint64_t x = f2_of_bf16x2(lds32(stg + (uint32_t)(quad * 32 + r) * 128u + ((uint32_t)((lane >> 2) ^ (r & 7)) << 4) + ((uint32_t)(lane & 3) << 2)));
                        su = f2_add(su, x); sq = f2_fma(x, x, sq);
                    }
                    *reinterpret_cast<uint64_t*>(&stat_s[quad][0][s0 + 2 * lane]) = su;
                    *reinterpret_cast<uint64_t*>(&stat_s[quad][1][s0 + 2 * lane]) = sq;
                }
                __syncwarp();
            }
            if (stat_tiles) {
                bar_sync_epi(bid);                               // (the next tile's barrier behind its accumulator keeps these sums until they are read)
                for (int c = et; c < n_tile; c += 128) {
                    if (BWD && bwd_x) {
                        if (col0 + c < ncol)
#pragma unroll
                            for (int k = 0; k < 2; ++k)
                                stat_tiles[((long long)tm * 2 + k) * ncol + col0 + c] = (float)((((double)stat_s[0][k][c] + (double)stat_s[1][k][c]) + (double)stat_s[2][k][c]) + (double)stat_s[3][k][c]);
                    } else if (col0 + c < ncol) {
                        const float su = ((stat_s[0][0][c] + stat_s[1][0][c]) + stat_s[2][0][c]) + stat_s[3][0][c];
                        const float sq = ((stat_s[0][1][c] + stat_s[1][1][c]) + stat_s[2][1][c]) + stat_s[3][1][c];
                        stat_tiles[((long long)tm * 2 + 0) * ncol + col0 + c] = su;
                        stat_tiles[((long long)tm * 2 + 1) * ncol + col0 + c] = sq;
                    }
                }
            }
        }
        if (elect_one()) bulk_wait_read(0);                      // shared memory stays until the last bulk stores have read it
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(L.tmem_cols) : "memory");
    }
}

// ------------------------------------------------------------------------------------------------ zero stuffing
// Backward of a stride-2 layer runs as a stride-1 problem on dy spread out to the input resolution:
// up[n, 2p, 2q, :] = dy[n, p, q, :], zero elsewhere.  Then dgrad(up) and wgrad(a, up) at stride 1 are the
// stride-2 dgrad and wgrad, term for term.
__global__ void __launch_bounds__(256) zero_stuff_kernel(const UpProb* __restrict__ probs) {
    const UpProb& p = probs[blockIdx.y];
    const int G = p.K >> 3;
    const long long nv = (long long)p.N * p.H * p.W * G;
    const uint4* src = reinterpret_cast<const uint4*>(p.src);
    uint4* dst = reinterpret_cast<uint4*>(p.dst);
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < nv; v += (long long)gridDim.x * blockDim.x) {
        const int g = (int)(v % G); long long t = v / G; const int w = (int)(t % p.W); t /= p.W; const int h = (int)(t % p.H); const int n = (int)(t / p.H);
        uint4 val = make_uint4(0u, 0u, 0u, 0u);
        if (!(h & 1) && !(w & 1) && (h >> 1) < p.P && (w >> 1) < p.Q) val = src[(((long long)n * p.P + (h >> 1)) * p.Q + (w >> 1)) * G + g];
        dst[v] = val;
    }
}
void launch_zero_stuff(const UpProb* d, int nprob, long long max_vecs, cudaStream_t s) {
    long long gx = (max_vecs + 255) / 256; if (gx > 148 * 16) gx = 148 * 16; if (gx < 1) gx = 1;
    zero_stuff_kernel<<<dim3((unsigned)gx, nprob), 256, 0, s>>>(d);
}

// ------------------------------------------------------------------------------------------------ wgrad
// dw[k][r][s][c] = sum over output positions of dy[pos][k] * a[pos + shift(r,s)][c].  The reduction runs over the
// positions of the forward problem (pixels in order, or the tall zero-padded map, where dy reads as zero at the padding
// positions and adds nothing), 128 per pipeline stage: D[cout (128 lanes), cin] per tap, A = dy^T and B = shifted a,
// both MN-major straight from their 128-byte rows.  A CTA of the three-tap form accumulates a range of position chunks for one group of taps
// (taps that read the same window: up to three taps of a stride-1 layer, the taps of one input parity phase of a stride-2
// layer) and writes an fp32 partial, or, alone on its tile, the result; a second kernel adds the partials in a fixed order.
// The nine-tap form (stride 1): the two 64-row halves of A are the same 64 channels of dy, the second one map row further (the descriptor's
// leading offset is Wp rows instead of a slab), and the three 64-column parts of B the same channels of a, one position apart each.  One MMA
// of 128 x 192 then holds the taps (row 1; 0, 1, 2) in its lower and (row 0; 0, 1, 2) in its upper lanes, a second one row 2 (and row 1 again, unused).
// What bounds it: the tensor pipe, 74 % active at 64 channels and 1024 x 32 x 32 positions (a quarter of that is row 1 computed twice), then the
// boxes' way into shared memory.  Before, one thread produced both operands with two divisions per box and a chunk of 1536 clocks of MMAs took
// ~5500.  8 x 128 images, us: 64 channels 32 x 32 294 -> 94,
// 128 16 x 16 143 -> 103, 256 8 x 8 205 -> 146 (two splits; 101 with one, whose chains are too long), 512 4 x 4 171 -> 134.
struct alignas(64) TcWgradProb {
    CUtensorMap map_dy;       // (channel k, pixel) or (channel k, x, y, image)
    CUtensorMap map_a;        // likewise for a, possibly element-strided
    float* partial;           // [splits][taps][cout][cin]
    float* out;               // [cout][taps][cin]
    int* status;
    int dy_flat, a_flat, taps;
    int es, pad, Hp, Wp, n_img;
    int R, box_pos, nbox_dy, nbox_a, hb, hb_step, dy_box_bytes, a_box_bytes;
    int chunks;                                   // position chunks of 128 in total
    int cout, cin, m_tiles, n_tile, n_tiles, a_slabs;
    int tap_groups; int gbeg[10]; int gxs[9], gys[9];
    TapRef tap[9];                                // wtap = index of the tap in dw; shift = row shift inside the a window
    int splits, chunks_per_split;
    int dy_slab_bytes, a_slab_bytes;              // one 64-channel slab of a stage
    int nine, m_tile, dy_slabs, mma_n;            // nine: all taps of a 64 x 64 tile in one CTA (m_tile 64, one slab each)
    int dy_lead, a_lead;                          // byte step from 64 rows (columns) of an MMA's operand to the next 64
    int stage_bytes, stages, tmem_cols;
};

__global__ void __launch_bounds__(TC_THREADS, 1) conv_wgrad_tc_kernel(const TcWgradProb* __restrict__ probs) {
    const TcWgradProb& p = probs[blockIdx.y];
    const int ctas = p.m_tiles * p.n_tiles * p.tap_groups * p.splits;
    if ((int)blockIdx.x >= ctas) return;
    // everything the loops read, in registers (the descriptor lives in global memory)
    const int splits = p.splits, tap_groups = p.tap_groups, n_tiles = p.n_tiles, chunks = p.chunks, chunks_per_split = p.chunks_per_split;
    const int stages = p.stages, stage_bytes = p.stage_bytes, dy_slab_bytes = p.dy_slab_bytes, a_slab_bytes = p.a_slab_bytes, a_slabs = p.a_slabs;
    const int n_tile = p.n_tile, dy_flat = p.dy_flat, a_flat = p.a_flat, box_pos = p.box_pos, R = p.R, Hp = p.Hp, pad = p.pad, es = p.es;
    const int nine = p.nine, m_tile = p.m_tile, dy_slabs = p.dy_slabs;
    const int nbox_dy = p.nbox_dy, nbox_a = p.nbox_a, dy_box_bytes = p.dy_box_bytes, a_box_bytes = p.a_box_bytes, tmem_cols = p.tmem_cols;
    int id = blockIdx.x;
    const int split = id % splits; id /= splits;
    const int tg = id % tap_groups; id /= tap_groups;
    const int tn = id % n_tiles; const int tm = id / n_tiles;
    const int c_begin = split * chunks_per_split;
    const int c_end = min(c_begin + chunks_per_split, chunks);
    const int tap0 = p.gbeg[tg], ntap = nine ? 2 : p.gbeg[tg + 1] - tap0;      // nine: two accumulators of 192 columns
    const int gx = p.gxs[tg], gy = p.gys[tg];
    const int hb = p.hb - tg * p.hb_step;                        // the group's window of a starts hb positions before the chunk
    const int nc = c_end - c_begin;

    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t bars[2 * TC_MAX_STAGES + 2];
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s;
    __shared__ int shift8_s[4], wtap_s[4];                       // the group's taps: row shift in 16-byte units, index in dw
    const uint32_t bar_full = smem_u32(&bars[0]), bar_empty = smem_u32(&bars[TC_MAX_STAGES]), bar_acc = smem_u32(&bars[2 * TC_MAX_STAGES]);
    const uint32_t bar_drain = smem_u32(&bars[2 * TC_MAX_STAGES + 1]);
    const uint32_t ring = smem_u32(smem);
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // warp-uniform for the compiler too

    if (threadIdx.x == 0) {
        for (int s = 0; s < TC_MAX_STAGES; ++s) { mbar_init(bar_full + 8 * s, 2); mbar_init(bar_empty + 8 * s, 1); }   // each operand's producer announces its bytes
        mbar_init(bar_acc, 1); mbar_init(bar_drain, 1);
        abort_s = 0;
        for (int i = 0; i < ntap; ++i) { shift8_s[i] = p.tap[tap0 + (nine ? 3 * i : i)].shift * 8; wtap_s[i] = p.tap[tap0 + i].wtap; }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_d = tmem_base_s;

    if (warp == 0 || warp == 2) {
        // One producer per operand: warp 0 loads dy, warp 2 a.  A stage is up to two dozen boxes, and where each one lies is kept as (image, row)
        // counters: with both operands in one thread and a division or two per box, this thread was what the launch waited for.
        if (elect_one()) {
            const bool is_dy = warp == 0;
            const CUtensorMap* map = is_dy ? &p.map_dy : &p.map_a;
            const int flat = is_dy ? dy_flat : a_flat, slabs = is_dy ? dy_slabs : a_slabs, nbox = is_dy ? nbox_dy : nbox_a;
            const int c0 = is_dy ? tm * m_tile : tn * n_tile, box_bytes = is_dy ? dy_box_bytes : a_box_bytes, slab_bytes = is_dy ? dy_slab_bytes : a_slab_bytes;
            const int mul = is_dy ? 1 : es, x0 = is_dy ? 0 : gx, y0 = is_dy ? 0 : gy;
            const uint32_t first = ring + (is_dy ? 0u : (uint32_t)(dy_slabs * dy_slab_bytes)), tx = (uint32_t)(slabs * nbox * box_bytes);
            const int box_img = R > Hp ? R / max(Hp, 1) : 1, box_row = R > Hp ? Hp : R;      // a box is rows of one image, or whole images
            int pos = c_begin * TILE_M - (is_dy ? 0 : hb), img0 = 0, row0 = 0;
            if (!flat) { const int b = floor_div(pos, box_pos), trow = b * R; img0 = floor_div(trow, Hp); row0 = trow - img0 * Hp; pos -= b * box_pos; }   // pos: from the first box's start
            int i = 0; bool ok = true; int s = 0; uint32_t ph = 0;
            for (; i < nc; ++i) {
                if (!mbar_wait(bar_empty + 8 * s, ph ^ 1u, &abort_s)) { atomicExch(&abort_s, 1); report_wait(p.status, 11); ok = false; break; }
                const uint32_t dst = first + (uint32_t)(s * stage_bytes), full = bar_full + 8 * s;
                mbar_expect_tx(full, tx);
                if (flat) {
                    for (int j = 0; j < slabs; ++j) tma_load_2d(dst + (uint32_t)(j * slab_bytes), map, full, c0 + j * 64, pos);
                    pos += TILE_M;
                } else {
                    int img = img0, row = row0; uint32_t to = dst;
                    for (int b = 0; b < nbox; ++b) {
                        const int y = (row - pad) * mul + y0;
                        tma_load_4d(to, map, full, c0, x0, y, img);
                        for (int j = 1; j < slabs; ++j) tma_load_4d(to + (uint32_t)(j * slab_bytes), map, full, c0 + j * 64, x0, y, img);
                        to += (uint32_t)box_bytes; row += box_row; if (row >= Hp) { row = 0; img += box_img; }
                    }
                    for (pos += TILE_M; pos >= box_pos; pos -= box_pos) { row0 += box_row; if (row0 >= Hp) { row0 = 0; img0 += box_img; } }
                }
                if (++s == stages) { s = 0; ph ^= 1u; }
            }
            if (!ok)
                for (int c = max(0, i - stages); c < i; ++c)
                    for (int w = 0; w < 4096 && !mbar_try(bar_full + 8 * (c % stages), (uint32_t)(c / stages) & 1u); ++w) __nanosleep(64);
        }
    } else if (warp == 1) {
        // The issuer: every tap of the group into its own accumulator, so each is summed over the positions in order.  The last tap of an odd group
        // has two, for the first and the second 64 positions of every chunk, which the epilogue adds: the tensor core's sums lose a little
        // with every step of a chain (relative to 64 bits, 128 images of 32 x 32, 1x1 256 -> 64 channels: 5.8e-7 with one chain, 3.3e-7 with two).
        if (elect_one()) {
            // fp32 accumulate, bf16 x bf16, A and B MN-major, N = mma_n, M = 128
            const int mma_n = p.mma_n;
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(mma_n >> 3) << 17) | ((128u >> 4) << 24);
            const uint32_t desc_hi = (uint32_t)(desc_sw128(0, 0, 1024) >> 32), dy_lbo = (uint32_t)(p.dy_lead >> 4) << 16, a_lbo = (uint32_t)(p.a_lead >> 4) << 16;
            const uint32_t a_at = (uint32_t)(dy_slabs * dy_slab_bytes) >> 4, inc = (uint32_t)(TILE_M % box_pos);
            uint32_t sh[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) sh[q] = q < ntap ? (uint32_t)shift8_s[q] : 0u;
            // the chunk's first position inside the first box of either window
            const int pos = c_begin * TILE_M;
            uint32_t dy_off = dy_flat ? 0u : (uint32_t)(pos % box_pos), a_off = a_flat ? 0u : (uint32_t)(pos - hb - floor_div(pos - hb, box_pos) * box_pos);
            bool ok = true; int s = 0; uint32_t ph = 0, acc = 0;
            for (int i = 0; i < nc; ++i) {
                if (!mbar_wait(bar_full + 8 * s, ph, &abort_s)) { atomicExch(&abort_s, 1); report_wait(p.status, 12); ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t stage16 = (ring + (uint32_t)(s * stage_bytes)) >> 4;           // addresses in 16-byte units
                const uint32_t dy_lo = (stage16 + dy_off * 8u) | dy_lbo, a_lo = (stage16 + a_at + a_off * 8u) | a_lbo;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (q >= ntap) break;
                    const uint32_t d_t = tmem_d + (uint32_t)(q * mma_n), at = a_lo + sh[q];
                    const bool halves = q == ntap - 1 && (ntap & 1);
                    const uint32_t d_t2 = halves ? d_t + (uint32_t)mma_n : d_t, acc2 = halves ? acc : 1u;
#pragma unroll
                    for (int k16 = 0; k16 < 8; ++k16)          // 16 positions = 16 rows of 128 bytes per step
                        umma_bf16(k16 < 4 ? d_t : d_t2, f2_pack(dy_lo + 128u * (uint32_t)k16, desc_hi), f2_pack(at + 128u * (uint32_t)k16, desc_hi), idesc, k16 == 0 ? acc : k16 == 4 ? acc2 : 1u);
                }
                acc = 1;
                umma_commit(bar_empty + 8 * s);
                if (!dy_flat) { dy_off += inc; if (dy_off >= (uint32_t)box_pos) dy_off -= (uint32_t)box_pos; }
                if (!a_flat) { a_off += inc; if (a_off >= (uint32_t)box_pos) a_off -= (uint32_t)box_pos; }
                if (++s == stages) { s = 0; ph ^= 1u; }
            }
            if (ok) umma_commit(bar_acc);
            else {
                // gave up: the MMAs already issued must have finished before the CTA frees its tensor memory
                umma_commit(bar_drain);
                for (int w = 0; w < 65536 && !mbar_try(bar_drain, 0u); ++w) __nanosleep(64);
            }
        }
    } else {
        const int quad = warp & 3, m = quad * 32 + lane;
        const int cout = p.cout, cin = p.cin, taps = p.taps;
        float* const partial = p.partial; float* const outp = p.out;
        bool ok = nc > 0 ? mbar_wait(bar_acc, 0, &abort_s) : true;
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) { atomicExch(&abort_s, 1); report_wait(p.status, 13); }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // nine: lanes 0 - 63 hold the taps of rows 1 (first accumulator) and 2 (second) of the tile's channels, lanes 64 - 127 those of row 0
        // (first) and row 1 once more (second, not read)
        const bool upper = nine && quad >= 2;
        const int k = tm * m_tile + (upper ? m - 64 : m);
        if (ok && nine) {
            if ((quad & 1) * 32 < cout - tm * 64) {
                for (int q = 0; q < (upper ? 3 : 6); ++q) {
                    const int wt = upper ? q : 3 + q;
                    float* dst = splits > 1 ? partial + (((long long)split * taps + wt) * cout + k) * cin + tn * 64
                                            : outp + ((long long)k * taps + wt) * cin + tn * 64;
                    for (int c0 = 0; c0 < 64; c0 += 32) {
                        uint32_t v[32];
                        if (nc > 0) {
                            tmem_ld32(tmem_d + ((uint32_t)(quad * 32) << 16) + (uint32_t)(q * 64 + c0), v);
                            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                        } else { for (int j = 0; j < 32; ++j) v[j] = 0u; }
                        if (k < cout) {
#pragma unroll
                            for (int j = 0; j < 32; j += 4)
                                if (tn * 64 + c0 + j < cin) *reinterpret_cast<uint4*>(dst + c0 + j) = make_uint4(v[j], v[j + 1], v[j + 2], v[j + 3]);
                        }
                    }
                }
            }
        } else if (ok && quad * 32 < cout - tm * 128) {              // warp-uniform: this lane quadrant holds real output channels
            for (int tt = 0; tt < ntap; ++tt) {
                const int wt = wtap_s[tt];
                float* dst = splits > 1 ? partial + (((long long)split * taps + wt) * cout + k) * cin + tn * n_tile
                                        : outp + ((long long)k * taps + wt) * cin + tn * n_tile;
                for (int c0 = 0; c0 < n_tile; c0 += 32) {
                    uint32_t v[32];
                    if (nc > 0) {
                        tmem_ld32(tmem_d + ((uint32_t)(quad * 32) << 16) + (uint32_t)(tt * n_tile + c0), v);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                        if ((ntap & 1) && tt == ntap - 1) {      // first half + second half
                            uint32_t v2[32];
                            tmem_ld32(tmem_d + ((uint32_t)(quad * 32) << 16) + (uint32_t)(ntap * n_tile + c0), v2);
                            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                            for (int j = 0; j < 32; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) + __uint_as_float(v2[j]));
                        }
                    } else { for (int j = 0; j < 32; ++j) v[j] = 0u; }
                    if (k < cout) {
#pragma unroll
                        for (int j = 0; j < 32; j += 4)
                            if (c0 + j < n_tile && tn * n_tile + c0 + j < cin)
                                *reinterpret_cast<uint4*>(dst + c0 + j) = make_uint4(v[j], v[j + 1], v[j + 2], v[j + 3]);
                    }
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_d), "r"(tmem_cols) : "memory");
    }
}

// out[k][t][c] = sum over splits (ascending) of partial[split][t][k][c].  The partials mostly lie in L2; what counts is how many loads are in flight and what an index
// costs: a thread takes four input channels, eight splits' loads at a time.  (One value per thread with 64-bit divisions and a load per addition: the weight gradients with
// their sums took 4.73 ms of a wide step of 8 x 128 images instead of 4.32, 4.79 instead of 4.11 of one of 1024 images on the whole network, 1.85 instead of 1.60 at 8 x 16.)
// VEC 1 where an address or a count is not a multiple of four floats (a sub-ResNet's parameters begin where the layers before them end).
constexpr int WG_RED_THREADS = 128;
template <int VEC> __device__ __forceinline__ void wgrad_tc_reduce_rows(const TcWgradProb& p) {
    using V = typename std::conditional<VEC == 4, float4, float>::type;
    const unsigned cin = (unsigned)p.cin / VEC, cout = (unsigned)p.cout, taps = (unsigned)p.taps, n = taps * cout * cin, splits = (unsigned)p.splits;
    const V* __restrict__ partial = reinterpret_cast<const V*>(p.partial);
    V* __restrict__ out = reinterpret_cast<V*>(p.out);
    for (unsigned i = blockIdx.x * WG_RED_THREADS + threadIdx.x; i < n; i += gridDim.x * WG_RED_THREADS) {
        const unsigned r = i / cin, c = i - r * cin, k = r / taps, t = r - k * taps;
        const V* src = partial + ((size_t)t * cout + k) * cin + c;
        V s;
        if constexpr (VEC == 4) s = make_float4(0.f, 0.f, 0.f, 0.f); else s = 0.f;
        for (unsigned sp = 0; sp < splits; sp += 8) {
            V v[8];
#pragma unroll
            for (unsigned u = 0; u < 8; ++u) if (sp + u < splits) v[u] = __ldcg(src + (size_t)(sp + u) * n);
#pragma unroll
            for (unsigned u = 0; u < 8; ++u) if (sp + u < splits) {
                if constexpr (VEC == 4) { s.x += v[u].x; s.y += v[u].y; s.z += v[u].z; s.w += v[u].w; } else s += v[u];
            }
        }
        out[i] = s;
    }
}
__global__ void __launch_bounds__(WG_RED_THREADS) wgrad_tc_reduce_kernel(const TcWgradProb* __restrict__ probs) {
    const TcWgradProb& p = probs[blockIdx.y];
    if (p.splits <= 1) return;                                 // the convolution kernel wrote the result itself
    if (((p.cin & 3) | (int)(((uintptr_t)p.out | (uintptr_t)p.partial) & 15)) == 0) wgrad_tc_reduce_rows<4>(p); else wgrad_tc_reduce_rows<1>(p);
}

// ------------------------------------------------------------------------------------------------ BN statistics from the tiles' sums
// The convolution kernel leaves, per 128-position tile, the column sums of what it stored.  Here they are added in a fixed order in
// double: a CTA takes CH channels, 512 / CH rows of threads every (512 / CH)-th tile (eight tiles' loads in flight per thread; latency is
// all there is to this kernel), then the rows' sums.  MODE 0, forward: mean, 1/sqrt(var + eps) and the running statistics.
// MODE 1, backward: the two reduction sums and the gradients of beta and gamma.
template <int MODE, int CH>
__global__ void __launch_bounds__(512) bn_finalize_tiles_kernel(const BnProb* __restrict__ probs) {
    const BnProb& p = probs[blockIdx.y];
    constexpr int ROWS = 512 / CH;
    const int C = p.C, ch = threadIdx.x % CH, row = threadIdx.x / CH, c = blockIdx.x * CH + ch, n = p.chunks;
    if ((int)blockIdx.x * CH >= C) return;
    __shared__ double red[2][ROWS][CH + 1];
    const float* __restrict__ t = reinterpret_cast<const float*>(p.partial) + (c < C ? c : 0);
    double a0 = 0.0, a1 = 0.0;
    for (int k = row; k < n; k += 8 * ROWS) {                    // eight tiles of loads in flight per thread
        float v0[8], v1[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int kk = k + ROWS * u;
            v0[u] = kk < n ? __ldcg(t + (long long)kk * 2 * C) : 0.f; v1[u] = kk < n ? __ldcg(t + ((long long)kk * 2 + 1) * C) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) { a0 += (double)v0[u]; a1 += (double)v1[u]; }
    }
    red[0][row][ch] = a0; red[1][row][ch] = a1;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp >= CH) return;
    // warp = channel, lane = every 32nd row of sums; fixed butterfly
    a0 = red[0][lane][warp]; a1 = red[1][lane][warp];
    for (int r = lane + 32; r < ROWS; r += 32) { a0 += red[0][r][warp]; a1 += red[1][r][warp]; }
    for (int d = 16; d; d >>= 1) { a0 += __shfl_xor_sync(0xffffffffu, a0, d); a1 += __shfl_xor_sync(0xffffffffu, a1, d); }
    const int cc = blockIdx.x * CH + warp;
    if (lane != 0 || cc >= C) return;
    if (MODE == 1) {
        p.stat[2 * C + cc] = (float)a0; p.stat[3 * C + cc] = (float)a1;
        p.dbeta[cc] = (float)a0; p.dgamma[cc] = (float)a1;
        return;
    }
    const double m = (double)p.m, mean = a0 / m;
    double var = a1 / m - mean * mean; if (var < 0.0) var = 0.0;
    p.stat[cc] = (float)mean;
    p.stat[C + cc] = (float)(1.0 / sqrt(var + (double)p.eps));
    if (p.run_mean) {
        const double unb = p.m > 1 ? var * m / (m - 1.0) : var, mo = (double)p.momentum;
        p.run_mean[cc] = (float)((1.0 - mo) * (double)p.run_mean[cc] + mo * mean);
        p.run_var[cc] = (float)((1.0 - mo) * (double)p.run_var[cc] + mo * unb);
    }
}
// 16 channels per CTA while that gives every SM one, 4 below: the fewer channels, the fewer CTAs, and the tiles are then many
// (the ImageNet-stem step, whose 64-channel layers have 1568 tiles and filled 16 SMs: 21.40 -> 21.21 ms).
void launch_bn_finalize_tiles(const BnProb* d, int nprob, int max_c, int backward, cudaStream_t s) {
    const bool few = (max_c + 15) / 16 * nprob < 148;
    const int ch = few ? 4 : 16;
    const dim3 g((max_c + ch - 1) / ch, nprob);
    if (backward) { if (few) bn_finalize_tiles_kernel<1, 4><<<g, 512, 0, s>>>(d); else bn_finalize_tiles_kernel<1, 16><<<g, 512, 0, s>>>(d); }
    else { if (few) bn_finalize_tiles_kernel<0, 4><<<g, 512, 0, s>>>(d); else bn_finalize_tiles_kernel<0, 16><<<g, 512, 0, s>>>(d); }
}

// ------------------------------------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* f = nullptr; cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)f;
    }
    return fn;
}

// bf16 tensor map of `rank` dimensions (innermost first), 128-byte swizzle, zero fill out of bounds; estr = traversal strides
static bool encode_map(CUtensorMap* m, const void* base, int rank, const uint64_t* dims, const uint64_t* strides_bytes, const uint32_t* box,
                       const uint32_t* estr = nullptr) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t d[5]; cuuint64_t st[4]; cuuint32_t b[5]; cuuint32_t es[5];
    for (int i = 0; i < rank; ++i) { d[i] = dims[i]; b[i] = box[i]; es[i] = estr ? estr[i] : 1; if (i + 1 < rank) st[i] = strides_bytes[i]; }
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(base), d, st, b, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// [pixels][chan] as (channel, pixel), box 64 x rows
static bool encode_flat(CUtensorMap* m, const void* base, int chan, long long pixels, int rows = 128) {
    const uint64_t dims[2] = {(uint64_t)chan, (uint64_t)pixels}; const uint64_t st[1] = {(uint64_t)chan * 2}; const uint32_t box[2] = {64, (uint32_t)rows};
    return encode_map(m, base, 2, dims, st, box);
}
// [n_img][H][W][chan] as (channel, x, y, image): a box is box_h rows of Wp window positions of box_n images, every es-th pixel in x and y
static bool encode_tall(CUtensorMap* m, const void* base, int chan, int n_img, int H, int W, int Wp, int box_h, int box_n, int es) {
    const uint64_t dims[4] = {(uint64_t)chan, (uint64_t)W, (uint64_t)H, (uint64_t)n_img};
    const uint64_t st[3] = {(uint64_t)chan * 2, (uint64_t)chan * 2 * W, (uint64_t)chan * 2 * W * H};
    const uint32_t box[4] = {64, (uint32_t)(Wp * es), (uint32_t)(box_h * es), (uint32_t)box_n};
    const uint32_t estr[4] = {1, (uint32_t)es, (uint32_t)es, 1};
    return encode_map(m, base, 4, dims, st, box, estr);
}

// The tall map of a grid of Hg x Wg positions per image: Wp = Wg + pad positions per row, Hp rows per image (Hg + pad, rounded up
// to a multiple of the rows of a box: the extra rows read as zero like the padding).  A box is R consecutive tall rows: part of
// one image (R divides Hp), or box_n whole images.  Larger boxes mean fewer TMA issues per window but more rows fetched around it;
// the choice: at most 96 positions per box, at most 6.5 % of extra rows, then the largest box.
struct Tall { int Hp, Wp, R, box_pos, box_bytes, box_h, box_n; };
static bool tall_of(int Hg, int Wg, int pad, int es, Tall& t, int max_box = 96) {
    t.Wp = Wg + pad;
    const int H0 = Hg + pad;
    if (t.Wp * es > 256) return false;
    int best_r = 1, best_hp = H0;
    for (int r = 1; r <= H0; ++r) {
        const int hp = (H0 + r - 1) / r * r;
        if ((r > 1 && r * t.Wp > max_box) || r * t.Wp > 96 || r * es > 256 || (hp - H0) * 200 > 13 * H0 || (pad == 0 && hp != H0)) continue;   // pad = 0: positions are the pixels in order, no extra rows
        if (r * t.Wp > best_r * t.Wp) { best_r = r; best_hp = hp; }
    }
    t.Hp = best_hp; t.R = best_r; t.box_h = best_r; t.box_n = 1;
    if (best_r == best_hp) {                      // whole images: several per box when they are small
        int ni = max_box / (t.Hp * t.Wp); if (ni < 1) ni = 1; if (ni > 8) ni = 8;
        t.box_n = ni; t.R = t.Hp * ni;
    }
    t.box_pos = t.R * t.Wp; t.box_bytes = t.box_pos * 128;
    return true;
}
static int boxes_for(int span, int box_pos) { return (span + 2 * (box_pos - 1)) / box_pos; }   // boxes that cover `span` positions from any start

// The taps of output phase (u, v) of a stride-2 3x3 dgrad (u, v = parity of the input row and column), or of input phase (u, v)
// of a stride-2 3x3 forward / wgrad: tap (r, s) belongs to the phase with (r - 1) = u, (s - 1) = v modulo 2.
static int phase_taps(int u, int v, int rs[4][2]) {
    int n = 0;
    for (int r = 0; r < 3; ++r) for (int s = 0; s < 3; ++s)
        if ((((r - 1) % 2) + 2) % 2 == u && (((s - 1) % 2) + 2) % 2 == v) { rs[n][0] = r; rs[n][1] = s; ++n; }
    return n;
}

static int device_sms() {
    static const int n = [] { int dev = 0, v = 0; cudaGetDevice(&dev); cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev); return v > 0 ? v : 148; }();
    return n;
}
static bool tc_shape_ok(const ConvProb& p) {
    if ((p.ksz != 1 && p.ksz != 3) || p.stride < 1 || p.stride > 2) return false;
    if (p.C % 8 || p.K % 8) return false;
    if ((long long)p.N * (p.H + 1) * (p.W + 1) > (1ll << 30)) return false;
    return true;
}

// The window of a forward / dgrad tile: its tall map, the positions before the tile's first (hb) and the boxes that cover it.  "flat": one
// box of 128 pixels of a dense problem.
struct TcWindow { bool flat; Tall g; int hb, nbox; size_t bytes; };
static bool tc_window(const ConvProb& p, int mode, TcWindow& w) {
    w.flat = p.ksz == 1 && (p.stride == 1 || mode == CONV_DGRAD); w.hb = 0; w.nbox = 1; w.bytes = SLAB_BYTES;
    if (w.flat) return true;
    const bool s2 = p.stride == 2; const int pad = p.ksz == 3 ? 1 : 0;
    if (!tall_of(s2 ? p.P : p.H, s2 ? p.Q : p.W, pad, s2 && mode == CONV_FWD ? 2 : 1, w.g)) return false;
    int span = TILE_M;
    if (pad && !s2) { w.hb = w.g.Wp + 1; span += 2 * w.hb; }
    else if (pad && mode == CONV_FWD) { w.hb = w.g.Wp + 1; span += w.hb; }
    else if (pad) span += w.g.Wp + 1;                            // one output phase of a stride-2 dgrad
    w.nbox = boxes_for(span, w.g.box_pos); w.bytes = ((size_t)w.nbox * w.g.box_bytes + 1023) / 1024 * 1024;
    return true;
}

constexpr size_t TC_SMEM_BUDGET = 204 * 1024;
static size_t tc_budget(bool dgrad) { return dgrad ? TC_SMEM_BUDGET - 8 * 1024 : TC_SMEM_BUDGET; }      // dgrad keeps 8 KB of BN constants beside the rings
static int tc_weight_tile(int n, int mode) { return mode == CONV_FWD ? n * 128 : ((n + 63) / 64) * 8192; }
// The least a launch runs with: the two windows of a pair of tiles, one weight tile of n columns and a slab buffer per epilogue group, another
// one per group when a BN of the output (evaluation) leaves through it.
static bool tc_fits(size_t window, int n, int mode, bool bn) {
    return 2 * window + ((size_t)tc_weight_tile(n, mode) + 1023) / 1024 * 1024 + 2 * (bn ? 2 : 1) * (size_t)SLAB_BYTES <= tc_budget(mode == CONV_DGRAD);
}
static int tc_narrowest(int ncol) { return std::min(64, (ncol + 15) / 16 * 16); }
static int tc_columns(const ConvProb& p, int mode) { return mode == CONV_FWD ? p.K : p.C; }

// Number of TcProb descriptors a forward / dgrad problem needs (0: not supported): one, or one per output phase of a stride-2 3x3 dgrad.
// Maps so wide that two windows do not fit (3x3: about 120 positions and up) are left to the other kernel families.
int conv_tc_count(const ConvProb& p, int mode) {
    if (mode == CONV_WGRAD || !encode_fn() || !tc_shape_ok(p)) return 0;
    if (((uintptr_t)p.act | (uintptr_t)p.wgt | (uintptr_t)p.out | (uintptr_t)p.add) & 15) return 0;
    TcWindow w;
    if (!tc_window(p, mode, w) || !tc_fits(w.bytes, tc_narrowest(tc_columns(p, mode)), mode, p.bn_out != nullptr)) return 0;
    return (mode == CONV_DGRAD && p.ksz == 3 && p.stride == 2) ? 4 : 1;
}
// evaluation: is there room for the BN of the output in the epilogue?
bool conv_tc_bn_fits(const ConvProb& p) {
    TcWindow w; return tc_window(p, CONV_FWD, w) && tc_fits(w.bytes, tc_narrowest(p.K), CONV_FWD, true);
}
bool conv_tc_supported(const ConvProb& p, int mode) { return conv_tc_count(p, mode) > 0; }
// 128-position tiles of a forward problem (the rows of ConvProb::stat_tiles)
int conv_tc_stat_tiles(const ConvProb& p) {
    long long pos = (long long)p.N * p.P * p.Q;
    if (p.ksz == 1 && p.stride == 2) { Tall g; tall_of(p.P, p.Q, 0, 2, g); pos = (long long)p.N * g.Hp * g.Wp; }
    if (p.ksz != 1) { Tall g; tall_of(p.P, p.Q, 1, p.stride, g); pos = (long long)p.N * g.Hp * g.Wp; }
    return (int)((pos + TILE_M - 1) / TILE_M);
}

// likewise of a stride-1 dgrad problem
int conv_tc_dgrad_tiles(const ConvProb& p) {
    if (p.ksz == 1) return (int)(((long long)p.N * p.P * p.Q + TILE_M - 1) / TILE_M);
    Tall g; tall_of(p.H, p.W, 1, 1, g);
    return (int)(((long long)p.N * g.Hp * g.Wp + TILE_M - 1) / TILE_M);
}

// Are the BN backward's sums taken in this data gradient's epilogue?  `group`: problems of the launch.  The epilogue then reads x, and is what the
// launch waits for; a reduction of its own reads x and da once more, which from beyond L2 (126 MB) it does faster than an epilogue.  How far the
// epilogue keeps up depends on the MMAs beside it and on the columns.  Data gradient + sums, us fused | apart (x of the launch in MB):
//   1x1, 64 <- 256 channels 134 MB 175 | 200, 201 MB 243 | 273; 128 <- 512 101 MB 134 | 165; 1024 <- 256 134 MB 138 | 153, 201 MB 191 | 198: up to 250 MB;
//   1x1 of fewer reduction than output channels, 256 <- 64 103 MB 101 | 104, 206 MB 165 | 167, 537 MB 384 | 331; 256 <- 128 103 MB 124 | 120, 206 MB 210 | 200,
//   537 MB 514 | 427; 512 <- 256 103 MB 134 | 130, 201 MB 230 | 208; 3x3, 64 channels 103 MB 165 | 167, 134 MB 226 | 216, 201 MB 327 | 296; 128 channels
//   101 MB 173 | 189: up to L2.
// Not below 64 channels, where half of the lanes have nothing to read (32 <- 128, 34 MB 93 | 75, 134 MB 279 | 218).  Not at stride 2: the scattered rows
// of x cost the four phases 171 us where the pass took 130.
bool conv_tc_bwd_sums(const ConvProb& p, int group) {
    const double limit = p.ksz == 1 && (p.K >= p.C || p.C >= 1024) ? 250e6 : 126e6;
    return p.stride == 1 && p.C >= 64 && (double)group * p.N * p.H * p.W * p.C * 2 <= limit;
}

// One status word per process in pinned host memory that every device can write: a kernel stores into it only when a bounded wait
// gives up, and the host reads it after a synchronisation without a copy (a 4-byte copy and its wait took 10 us of every layer call).
int* conv_tc_status_word() {
    static int* word = [] { int* w = nullptr; if (cudaHostAlloc(&w, 256, cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) { cudaGetLastError(); return (int*)nullptr; } *w = 0; return w; }();
    return word;
}
int conv_tc_read_status() {
    volatile int* w = conv_tc_status_word();
    if (!w) return 0;
    const int v = *w;
    if (v) *w = 0;                                  // reported once
    return v;
}

// Columns per tile: up to 256, a multiple of 64 when there are several tiles.  A launch ends with its slowest CTA, so a launch of few units
// takes the width with the least (waves of pairs) x (clocks per pair) over `group` such problems, the last partial wave possibly in
// single tiles (see the kernel).  Clocks per tile: the tensor core needs 128 / 68 / 52 per MMA of 256 / 128 / 64 columns; the rings are fed
// from L2 at about 28 bytes per clock and SM (all SMs at once); an epilogue takes about 20 per column, and only runs under the next tile's
// MMAs when two accumulators per tile fit TMEM (up to 128 columns).  Narrower tiles read every window once more, so they have to promise
// 12 %, and from two full waves of the widest tiles on there is nothing to fill.  (Evaluation of 50 ImageNet-shaped images 2.19 -> 1.95 ms;
// with pairs really split where they are few, as this assumes, 1.87 -> 1.78, 4 images 0.98 -> 0.78.)
static void pick_n_tile(TcHot& t, int ntaps, int group, int phases, int mode, bool bn) {
    const int sms = device_sms();
    double best = 0; int best_n = 0; long long wide_pairs = 0;
    const int first = (t.ncol + 255) / 256;
    for (int tn = first; tn <= std::max(first, (t.ncol + 63) / 64); ++tn) {
        int n = (t.ncol + tn - 1) / tn;
        n = tn > 1 ? (n + 63) / 64 * 64 : (n + 15) / 16 * 16;
        if ((t.ncol + n - 1) / n != tn || !tc_fits(((size_t)t.nbox * t.a_box_bytes + 1023) / 1024 * 1024, n, mode, bn)) continue;
        const double mma = n > 128 ? n / 2.0 : n > 64 ? 68 : 52, steps = (double)ntaps * t.slabs * std::min(4, (t.red + 15) / 16);
        const double epi = 20.0 * n + 500, a_bytes = (double)t.slabs * t.ngroups * t.nbox * t.a_box_bytes, b_bytes = (double)t.slabs * ntaps * n * 128;
        auto unit = [&](int tiles) {
            const double run = std::max(tiles * steps * mma, (tiles * a_bytes + b_bytes) / 28) + 300;
            return n > 128 ? run + epi : std::max(run, epi);
        };
        const long long pairs = (long long)((t.tiles_m + 1) / 2) * tn * group * phases, rest = pairs % sms;
        const double time = (double)(pairs / sms) * unit(2) + (rest == 0 ? 0 : 2 * rest <= sms ? unit(1) : unit(2)) + (n > 128 ? 0 : epi);
        if (best_n && wide_pairs >= 2 * sms) break;
        if (!best_n) wide_pairs = pairs;
        if (!best_n || time < 0.88 * best) { best = time; best_n = n; }
    }
    t.n_tile = best_n; t.tiles_n = (t.ncol + best_n - 1) / best_n;
}

// Fills conv_tc_count() host-side TcProbs for this problem.  Returns the number written (0: not supported or encoding failed).
int conv_tc_fill(const ConvProb& p, int mode, void* host_tc) {
    const int count = conv_tc_count(p, mode);
    TcWindow win;
    if (!count || !tc_window(p, mode, win)) return 0;
    const Tall& g = win.g;
    const int taps = p.ksz * p.ksz;
    const int chan_a = mode == CONV_FWD ? p.C : p.K, ncol = tc_columns(p, mode);
    for (int ph = 0; ph < count; ++ph) {
        TcProb tp; memset(&tp, 0, sizeof(tp)); TcHot& t = tp.h;
        t.add = (const __nv_bfloat16*)p.add; t.out = (__nv_bfloat16*)p.out; t.status = conv_tc_status_word();
        t.stat_tiles = p.stat_tiles;
        if (mode == CONV_DGRAD && p.bn_x) { t.bwd_x = (const __nv_bfloat16*)p.bn_x; t.bn_stat = p.bn_stat; t.bn_gamma = p.bn_gamma; t.bn_beta = p.bn_beta; }
        t.n_img = p.N; t.ncol = ncol; t.red = chan_a; t.slabs = (chan_a + 63) / 64; t.scale = p.scale;
        t.b_mn_major = mode == CONV_DGRAD ? 1 : 0;
        t.es = 1; t.pad = 0; t.os = 1; t.oy = 0; t.ox = 0; t.ngroups = 1; t.gbeg[0] = 0;
        const void* act = p.act;
        long long out_pixels = 0;
        if (win.flat) {
            // plain GEMM over the pixels of the operand: forward at stride 1, dgrad at either stride (stride 2: over the P x Q pixels of dy)
            const int Hg = mode == CONV_DGRAD ? p.P : p.H, Wg = mode == CONV_DGRAD ? p.Q : p.W;
            t.a_flat = 1; t.Hp = Hg; t.Wp = Wg; t.R = 0; t.box_pos = TILE_M; t.nbox = 1; t.hb = 0; t.a_box_bytes = SLAB_BYTES;
            t.total_pos = p.N * Hg * Wg;
            { const int ti_ = 0; t.wtap[ti_] = 0; t.shift[ti_] = 0; } t.gbeg[1] = 1;
            if (!encode_flat(&tp.map_a, act, chan_a, t.total_pos)) return 0;
            if (p.stride == 2 && !p.out_compact) { t.dense = 0; t.OH = p.H; t.OW = p.W; t.os = 2; out_pixels = (long long)p.N * p.H * p.W; }   // scattered to the even positions
            else { t.dense = 1; t.OH = Hg; t.OW = Wg; out_pixels = t.total_pos; }
        } else if (p.ksz == 1) {
            // forward of a stride-2 1x1 layer: the positions are the output pixels, the window gathers every second input pixel
            t.a_flat = 0; t.dense = 1; t.es = 2; t.Hp = g.Hp; t.Wp = g.Wp; t.R = g.R; t.box_pos = g.box_pos; t.a_box_bytes = g.box_bytes; t.hb = win.hb; t.nbox = win.nbox;
            t.total_pos = p.N * g.Hp * g.Wp; t.OH = p.P; t.OW = p.Q; out_pixels = t.total_pos;
            { const int ti_ = 0; t.wtap[ti_] = 0; t.shift[ti_] = 0; } t.gbeg[1] = 1;
            if (!encode_tall(&tp.map_a, act, chan_a, p.N, p.H, p.W, g.Wp, g.box_h, g.box_n, 2)) return 0;
        } else if (p.stride == 1) {
            // 3x3 at stride 1: one window, nine taps; dgrad walks the taps mirrored
            t.a_flat = 0; t.dense = 0; t.pad = 1; t.Hp = g.Hp; t.Wp = g.Wp; t.R = g.R; t.box_pos = g.box_pos; t.a_box_bytes = g.box_bytes; t.hb = win.hb; t.nbox = win.nbox;
            t.total_pos = p.N * g.Hp * g.Wp; t.OH = p.H; t.OW = p.W; out_pixels = (long long)p.N * p.H * p.W;
            for (int w = 0; w < 9; ++w) { const int ti_ = w; t.wtap[ti_] = mode == CONV_DGRAD ? 8 - w : w; t.shift[ti_] = (w / 3) * g.Wp + (w % 3); }
            t.gbeg[1] = 9;
            if (!encode_tall(&tp.map_a, act, chan_a, p.N, p.H, p.W, g.Wp, g.box_h, g.box_n, 1)) return 0;
        } else if (mode == CONV_FWD) {
            // 3x3 at stride 2, forward: positions over the P x Q outputs, one window per input parity phase (element-strided fetch)
            t.a_flat = 0; t.dense = 0; t.pad = 1; t.es = 2; t.Hp = g.Hp; t.Wp = g.Wp; t.R = g.R; t.box_pos = g.box_pos; t.a_box_bytes = g.box_bytes; t.hb = win.hb; t.nbox = win.nbox;
            t.total_pos = p.N * g.Hp * g.Wp; t.OH = p.P; t.OW = p.Q; out_pixels = (long long)p.N * p.P * p.Q;
            int n = 0; t.ngroups = 0;
            for (int u = 0; u < 2; ++u) for (int v = 0; v < 2; ++v) {
                int rs[4][2]; const int k = phase_taps(u, v, rs);
                t.gxs[t.ngroups] = v; t.gys[t.ngroups] = u;
                for (int i = 0; i < k; ++i) {
                    const int di = rs[i][0] == 0 ? -1 : 0, dj = rs[i][1] == 0 ? -1 : 0;    // tap 0 reads the previous phase row / column
                    { const int ti_ = n++; t.wtap[ti_] = rs[i][0] * 3 + rs[i][1]; t.shift[ti_] = t.hb + di * g.Wp + dj; }
                }
                t.gbeg[++t.ngroups] = n;
            }
            if (!encode_tall(&tp.map_a, act, chan_a, p.N, p.H, p.W, g.Wp, g.box_h, g.box_n, 2)) return 0;
        } else {
            // 3x3 at stride 2, dgrad: one problem per output parity phase (u, v), positions over the P x Q grid of dy; input row 2i + u
            // takes dy row i + (u + 1 - r) / 2 through tap r
            const int u = ph >> 1, v = ph & 1;
            t.a_flat = 0; t.dense = 0; t.pad = 1; t.Hp = g.Hp; t.Wp = g.Wp; t.R = g.R; t.box_pos = g.box_pos; t.a_box_bytes = g.box_bytes; t.hb = win.hb; t.nbox = win.nbox;
            t.total_pos = p.N * g.Hp * g.Wp;
            t.OH = p.H; t.OW = p.W; t.os = 2; t.oy = u; t.ox = v; out_pixels = (long long)p.N * p.H * p.W;
            int rs[4][2]; const int k = phase_taps(u, v, rs);
            for (int i = 0; i < k; ++i) { const int ti_ = i; t.wtap[ti_] = rs[i][0] * 3 + rs[i][1]; t.shift[ti_] = ((u + 1 - rs[i][0]) / 2) * g.Wp + (v + 1 - rs[i][1]) / 2; }
            t.gbeg[1] = k;
            if (!encode_tall(&tp.map_a, act, chan_a, p.N, p.P, p.Q, g.Wp, g.box_h, g.box_n, 1)) return 0;
        }
        // residual
        t.add_mode = !p.add ? 0 : p.add_sub == 2 ? 3 : 2;
        const int ntaps = t.gbeg[t.ngroups];
        t.tiles_m = (t.total_pos + TILE_M - 1) / TILE_M;
        pick_n_tile(t, ntaps, p.group > 0 ? p.group : 1, count, mode, p.bn_out != nullptr);
        t.out_slabs = (t.n_tile + 63) / 64;
        t.b_bytes = tc_weight_tile(t.n_tile, mode);
        // weights [K][taps][C] viewed as (C, tap, K).  Forward: a tile is n_tile output channels (rows) x 64 input channels.
        // dgrad: a block is 64 reduction channels k (rows) x 64 output columns c.
        { const uint64_t dims[3] = {(uint64_t)p.C, (uint64_t)taps, (uint64_t)p.K};
          const uint64_t st[2] = {(uint64_t)p.C * 2, (uint64_t)taps * p.C * 2};
          const uint32_t box[3] = {64, 1, mode == CONV_FWD ? (uint32_t)t.n_tile : 64u};
          if (!encode_map(&tp.map_b, p.wgt, 3, dims, st, box)) return 0; }
        t.store_y = 1;
        if (p.bn_out) { t.bn_out = (__nv_bfloat16*)p.bn_out; t.bn_stat = p.bn_stat; t.bn_gamma = p.bn_gamma; t.bn_beta = p.bn_beta; t.store_y = p.bn_only ? 0 : 1; }
        if (t.dense) {
            if (!encode_flat(&tp.map_out, p.out, ncol, out_pixels, 32)) return 0;
            if (p.bn_out && !encode_flat(&tp.map_bn, p.bn_out, ncol, out_pixels, 32)) return 0;
            if (t.add_mode == 2) { t.res_tma = 1; if (!encode_flat(&tp.map_add, p.add, ncol, out_pixels)) return 0; }
        }
        memcpy((char*)host_tc + (size_t)ph * sizeof(TcProb), &tp, sizeof(tp));
    }
    return count;
}
size_t conv_tc_prob_bytes() { return sizeof(TcProb); }
// units of work of a problem: pairs of row tiles x column tiles
int conv_tc_tiles(const void* host_tc) { const TcHot* t = &((const TcProb*)host_tc)->h; return ((t->tiles_m + 1) / 2) * t->tiles_n; }
// packs what a launch has to know about its largest problem into one number: window KB (12 bits), weight-tile KB (12), flags
// (4; 1: residual through TMA, 2: BN of the output, 4: dgrad), MMA N (36)
size_t conv_tc_smem(const void* host_tc) {
    const TcHot* t = &((const TcProb*)host_tc)->h;
    const size_t a_stage = ((size_t)t->nbox * t->a_box_bytes + 1023) / 1024, b_stage = ((size_t)t->b_bytes + 1023) / 1024;
    return (a_stage << 52) | (b_stage << 40) | ((size_t)((t->res_tma ? 1 : 0) | (t->bn_out ? 2 : 0) | (t->b_mn_major ? 4 : 0)) << 36) | (size_t)t->n_tile;
}
// field-wise maximum of two packed values
size_t conv_tc_merge(size_t a, size_t b) {
    return (std::max(a >> 52, b >> 52) << 52) | (std::max((a >> 40) & 0xFFF, (b >> 40) & 0xFFF) << 40) | ((((a >> 36) | (b >> 36)) & 0xF) << 36) |
           std::max(a & 0xFFFFFFFFF, b & 0xFFFFFFFFF);
}

// Shared memory and tensor memory of a launch; returns the dynamic shared memory (tc_fits says which problems get here).
static size_t tc_layout(size_t packed, TcLaunch& L) {
    L.a_stage = (int)(packed >> 52) * 1024; L.b_stage = (int)((packed >> 40) & 0xFFF) * 1024;
    const int n_tile = (int)(packed & 0xFFFFFFFFF);
    // Shared memory.  Two epilogue groups of L.eb 16 KB slab buffers: a residual is fetched into them ahead of its use and wants three
    // (one being added to, one being stored, one in flight), else two; a BN of the output takes one more per group.  A layer runs at the
    // bytes it keeps in flight.  1x1 layers: four windows (two pairs of tiles), then weight tiles.  3x3 layers read a window nine times,
    // so it is the weight tiles that stream: one slab buffer per group, two windows, four weight tiles, then more windows (measured
    // at 128 channels on 16 x 16 maps, 1024 images: 148 us with two weight tiles and four windows, 125 us with four and three).
    const size_t a = (size_t)L.a_stage, b = (size_t)L.b_stage;
    const size_t budget = tc_budget((packed >> 36) & 4);
    const int flags = (int)((packed >> 36) & 0xF), extra = flags & 2 ? 1 : 0;
    L.groups = 2; L.res = flags & 1;
    auto staging = [&] { return (size_t)L.groups * (L.eb + extra) * SLAB_BYTES; };
    if (a <= 16 * 1024) {                                        // 1x1 layers: windows of one box
        L.eb = L.res ? 3 : 2;
        while (L.eb > 1 && staging() + 4 * a + (L.res ? 1 : 3) * b > budget) --L.eb;
        const size_t rings = budget - staging();
        L.na = 4; while (L.na > 2 && (size_t)L.na * a + 2 * b > rings) --L.na;
        L.nb = 1; while (L.nb < 8 && (size_t)L.na * a + (size_t)(L.nb + 1) * b <= rings) ++L.nb;
        while (L.na < TC_MAX_STAGES && (size_t)(L.na + 1) * a + (size_t)L.nb * b <= rings) ++L.na;
    } else {                                                     // several taps per window: weight tiles are what streams
        L.eb = 1;
        const size_t rings = budget - staging();
        L.na = 2; L.nb = 1; while (L.nb < 4 && 2 * a + (size_t)(L.nb + 1) * b <= rings) ++L.nb;
        while (L.na < 4 && (size_t)(L.na + 1) * a + (size_t)L.nb * b <= rings) ++L.na;
        while (L.nb < 8 && (size_t)L.na * a + (size_t)(L.nb + 1) * b <= rings) ++L.nb;
    }
    L.acc_stride = (n_tile + 31) / 32 * 32;
    L.nbuf = L.acc_stride <= 128 ? 2 : 1;
    L.tmem_cols = 32; while (L.tmem_cols < 2 * L.nbuf * L.acc_stride) L.tmem_cols *= 2;
    // at least 120 KB of shared memory so that two CTAs that allocate tensor memory never share an SM
    return std::max((size_t)L.na * a + (size_t)L.nb * b + staging(), (size_t)120 * 1024) + 1024;
}

// max_tiles: the most units (pairs of row tiles x column tiles) of a problem; packed: conv_tc_merge over its problems
// pdl: programmatic launch.  For evaluation, a chain of convolutions; in training the linked launches made the steps slower (ImageNet-shaped
// 22.6 -> 24.4 ms with the forward half linked): between the convolutions run streaming kernels that want the whole SM.
void launch_conv_tc_probs(const void* d_tc, int nprob, int max_tiles, size_t packed, cudaStream_t s, bool pdl) {
    static bool configured = false; static int sms = 0;
    if (!configured) {
        cudaFuncSetAttribute(conv_tc_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(tc_budget(false) + 1024));
        cudaFuncSetAttribute(conv_tc_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(tc_budget(true) + 1024));
        int dev = 0; cudaGetDevice(&dev); cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        configured = true;
    }
    TcLaunch L{};
    L.nprob = nprob;
    const size_t smem = tc_layout(packed, L);
    const bool dgrad = (packed >> 36) & 4;
    // a CTA per row tile while there are SMs for them: the kernel then splits the pairs (of few units there is no full wave, only the last one)
    const int grid = (int)std::max(1ll, std::min(2ll * max_tiles * nprob, (long long)sms));
    cudaLaunchConfig_t cfg = {}; cfg.gridDim = dim3(grid); cfg.blockDim = dim3(TC_CONV_THREADS); cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cudaLaunchAttribute at[1]; at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization; at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at; cfg.numAttrs = pdl ? 1 : 0;
    cudaLaunchKernelEx(&cfg, dgrad ? conv_tc_kernel<true> : conv_tc_kernel<false>, (const TcProb*)d_tc, (const TcLaunch)L);
}

// ---- wgrad host side
struct WgGeom { TcWgradProb t; size_t partial_bytes; long long cost; int box_h, box_n; };

static bool wg_geometry_box(const ConvProb& p, int target_ctas, WgGeom& w, int max_box, bool nine, int max_chain = INT_MAX);
// Both operands of a 3x3 weight gradient are windows of boxes, so a stage is large and the boxes' rounding decides how many stages
// fit: the largest boxes that still leave two stages are taken (fewer TMA issues), else the size with the most stages.
// A stride-1 3x3 layer has two forms: 128 x 128 tiles with one filter row's three taps per CTA, or 64 x 64 tiles with all nine taps, which load
// both operands once and, at 64 channels, leave no half of the MMA's lanes idle.  The cheaper one by the split's cost is taken.  us at
// 8 x 128 images, three taps | nine: 64 channels 32 x 32 294 | 94, 128 16 x 16 102 | 119, 256 8 x 8 146 | 101 with one split, 146 with two, 512 4 x 4 134 | 150.
static bool wg_geometry(const ConvProb& p, int target_ctas, WgGeom& w) {
    if (p.ksz == 1) return wg_geometry_box(p, target_ctas, w, 96, false);
    const int caps[5] = {96, 64, 48, 32, 24};
    bool found = false; size_t partial = 0;
    for (int nine = 0; nine < (p.stride == 1 ? 2 : 1); ++nine) {
        WgGeom best; int best_stages = 0;
        // its sums must not run longer than the other form's, one of whose three taps has chains of half the length: sqrt((1 + 1 + 1 / 4) / 3)
        const int max_chain = found && nine ? (int)(0.866 * w.t.chunks_per_split) : INT_MAX;
        for (int i = 0; i < 5 && best_stages < 2; ++i) {
            WgGeom g;
            if (!wg_geometry_box(p, target_ctas, g, caps[i], nine != 0, max_chain)) continue;
            if (g.t.stages > best_stages) { best = g; best_stages = g.t.stages; }
        }
        if (!best_stages) continue;
        partial = std::max(partial, best.partial_bytes);         // a launch of more problems may take the other form
        if (best.cost < 0 || (found && best.cost >= w.cost)) continue;
        w = best; found = true;
    }
    w.partial_bytes = partial;
    return found;
}
static bool wg_geometry_box(const ConvProb& p, int target_ctas, WgGeom& w, int max_box, bool nine, int max_chain) {
    if (!tc_shape_ok(p)) return false;
    if (((uintptr_t)p.act | (uintptr_t)p.wgt) & 15) return false;
    TcWgradProb& t = w.t; memset(&t, 0, sizeof(t));
    const int taps = p.ksz * p.ksz;
    t.taps = taps; t.n_img = p.N; t.cout = p.K; t.cin = p.C; t.es = 1; t.pad = 0;
    long long total_pos;
    if (p.ksz == 1 && p.stride == 1) {
        t.dy_flat = 1; t.a_flat = 1; t.Hp = p.H; t.Wp = p.W; t.box_pos = TILE_M; t.nbox_dy = 1; t.nbox_a = 1; t.hb = 0;
        t.dy_box_bytes = SLAB_BYTES; t.a_box_bytes = SLAB_BYTES; total_pos = (long long)p.N * p.H * p.W;
        t.tap_groups = 1; t.gbeg[1] = 1; t.tap[0] = TapRef{0, 0};
    } else if (p.ksz == 1) {
        // stride-2 1x1: the positions are the P x Q pixels of dy in order; a is gathered at every second pixel
        Tall g; if (!tall_of(p.P, p.Q, 0, 2, g)) return false;
        w.box_h = g.box_h; w.box_n = g.box_n;
        t.dy_flat = 1; t.a_flat = 0; t.es = 2; t.Hp = g.Hp; t.Wp = g.Wp; t.R = g.R; t.box_pos = g.box_pos; t.hb = 0;
        t.nbox_dy = 1; t.dy_box_bytes = SLAB_BYTES; t.nbox_a = boxes_for(TILE_M, g.box_pos); t.a_box_bytes = g.box_bytes;
        total_pos = (long long)p.N * g.Hp * g.Wp;
        t.tap_groups = 1; t.gbeg[1] = 1; t.tap[0] = TapRef{0, 0};
    } else if (p.stride == 1) {
        Tall g; if (!tall_of(p.H, p.W, 1, 1, g, max_box)) return false;
        w.box_h = g.box_h; w.box_n = g.box_n;
        t.dy_flat = 0; t.a_flat = 0; t.pad = 1; t.Hp = g.Hp; t.Wp = g.Wp; t.R = g.R; t.box_pos = g.box_pos; t.hb = g.Wp + 1;
        t.dy_box_bytes = g.box_bytes; t.a_box_bytes = g.box_bytes;
        if (nine) {
            t.nine = 1; t.hb = 1;                        // dy from the chunk on, a from one position before it, both for one more row of the map
            t.nbox_dy = boxes_for(TILE_M + g.Wp, g.box_pos); t.nbox_a = boxes_for(TILE_M + g.Wp + 2, g.box_pos);
            t.tap[0] = TapRef{0, 0}; t.tap[3] = TapRef{3, g.Wp};       // where the two accumulators' windows start
        } else {
            t.nbox_dy = boxes_for(TILE_M, g.box_pos); t.nbox_a = boxes_for(TILE_M + 2, g.box_pos); t.hb_step = g.Wp;      // a group is the three taps of a filter row
            for (int i = 0; i < 9; ++i) t.tap[i] = TapRef{i, i % 3};
        }
        total_pos = (long long)p.N * g.Hp * g.Wp;
        t.tap_groups = 0;                                // groups of up to three taps: set below, once the column tile is known
    } else {
        Tall g; if (!tall_of(p.P, p.Q, 1, 2, g, max_box)) return false;
        Tall gd; if (!tall_of(p.P, p.Q, 1, 1, gd, max_box)) return false;
        if (gd.R != g.R || gd.Hp != g.Hp) return false;          // both operands walk the same boxes of rows
        w.box_h = g.box_h; w.box_n = g.box_n;
        t.dy_flat = 0; t.a_flat = 0; t.pad = 1; t.es = 2; t.Hp = g.Hp; t.Wp = g.Wp; t.R = g.R; t.box_pos = g.box_pos; t.hb = g.Wp + 1;
        t.nbox_dy = boxes_for(TILE_M, g.box_pos); t.nbox_a = boxes_for(TILE_M + t.hb, g.box_pos); t.dy_box_bytes = g.box_bytes; t.a_box_bytes = g.box_bytes;
        total_pos = (long long)p.N * g.Hp * g.Wp;
        int n = 0; t.tap_groups = 0;
        for (int u = 0; u < 2; ++u) for (int v = 0; v < 2; ++v) {
            int rs[4][2]; const int k = phase_taps(u, v, rs);
            t.gxs[t.tap_groups] = v; t.gys[t.tap_groups] = u;
            for (int i = 0; i < k; ++i) t.tap[n++] = TapRef{rs[i][0] * 3 + rs[i][1], t.hb + (rs[i][0] == 0 ? -1 : 0) * g.Wp + (rs[i][1] == 0 ? -1 : 0)};
            t.gbeg[++t.tap_groups] = n;
        }
    }
    t.chunks = (int)((total_pos + TILE_M - 1) / TILE_M);
    t.m_tile = t.nine ? 64 : 128; t.dy_slabs = t.m_tile / 64;
    t.m_tiles = (p.K + t.m_tile - 1) / t.m_tile;
    // columns of one CTA: the input channels in tiles of at most 256 (1x1) or 128 (3x3: up to four taps in 512 columns of tensor memory)
    const int n_cap = taps == 1 ? 256 : t.nine ? 64 : 128;
    t.n_tiles = (p.C + n_cap - 1) / n_cap;
    t.n_tile = (p.C + t.n_tiles - 1) / t.n_tiles;
    t.n_tile = t.n_tiles > 1 ? (t.n_tile + 63) / 64 * 64 : (t.n_tile + 15) / 16 * 16;
    t.n_tiles = (p.C + t.n_tile - 1) / t.n_tile;
    if (t.nine) t.n_tile = 64;
    t.a_slabs = (t.n_tile + 63) / 64;
    if (t.nine) { t.tap_groups = 1; t.gbeg[1] = 9; }
    else if (taps == 9 && p.stride == 1) { for (int g = 0; g < 3; ++g) { t.gbeg[g + 1] = 3 * (g + 1); t.gxs[g] = 0; t.gys[g] = 0; } t.tap_groups = 3; }
    int max_acc = 0; for (int g = 0; g < t.tap_groups; ++g) { const int n = t.gbeg[g + 1] - t.gbeg[g]; max_acc = std::max(max_acc, n + (n & 1)); }   // an odd group's last tap has two
    t.mma_n = t.nine ? 192 : t.n_tile;
    if (t.nine) max_acc = 2;
    t.tmem_cols = 32; while (t.tmem_cols < max_acc * t.mma_n) t.tmem_cols *= 2;
    if (t.tmem_cols > 512) return false;
    t.dy_slab_bytes = (t.nbox_dy * t.dy_box_bytes + 1023) / 1024 * 1024;
    t.a_slab_bytes = (t.nbox_a * t.a_box_bytes + 1023) / 1024 * 1024;
    t.dy_lead = t.nine ? t.Wp * 128 : t.dy_slab_bytes; t.a_lead = t.nine ? 128 : t.a_slab_bytes;
    t.stage_bytes = t.dy_slabs * t.dy_slab_bytes + t.a_slabs * t.a_slab_bytes;
    t.stages = TC_MAX_STAGES; while (t.stages > 1 && (size_t)t.stages * t.stage_bytes > TC_SMEM_BUDGET) --t.stages;
    if ((size_t)t.stages * t.stage_bytes > TC_SMEM_BUDGET) return false;
    // Split of the positions.  target_ctas is twice this problem's share of the SMs.  Every CTA pays a fixed cost (set-up, the
    // accumulators' way out) worth about six chunks, and a launch takes whole waves, so the split is the one that minimises
    // waves x (chunks per CTA + 6): mostly one full wave.  (A chunk of the nine-tap form takes 3/4 of the others' time.)  The partial buffer is sized for the most splits any share could pick.
    const int fixed = t.m_tiles * t.n_tiles * t.tap_groups;
    const int want_max = std::max(1, std::min(std::min(t.chunks, 256), target_ctas / fixed));
    const int share = std::max(1, target_ctas / 2);
    long long best_cost = -1; int best_cps = t.chunks;
    for (int sp = 1; sp <= want_max; ++sp) {
        const int cps = (t.chunks + sp - 1) / sp, eff = (t.chunks + cps - 1) / cps;
        if (cps > max_chain) continue;
        const long long waves = ((long long)fixed * eff + share - 1) / share, cost = waves * ((t.nine ? 3 : 4) * (long long)cps + 24);
        if (best_cost < 0 || cost < best_cost) { best_cost = cost; best_cps = cps; }
    }
    w.cost = best_cost; t.chunks_per_split = best_cps; t.splits = (t.chunks + best_cps - 1) / best_cps;
    w.partial_bytes = want_max > 1 ? (size_t)want_max * taps * p.K * p.C * 4 : 0;
    return true;
}

bool conv_wgrad_tc_supported(const ConvProb& p, int target_ctas, size_t* partial_bytes) {
    WgGeom g; if (!encode_fn() || !wg_geometry(p, target_ctas, g)) return false;
    if (partial_bytes) *partial_bytes = g.partial_bytes;
    return true;
}

// p.act = a, p.wgt = dy, p.out = dw (fp32), p.partial = workspace of at least partial_bytes
bool conv_wgrad_tc_fill(const ConvProb& p, int target_ctas, void* host_tc) {
    WgGeom g; if (!wg_geometry(p, target_ctas, g)) return false;
    TcWgradProb& t = g.t;
    if (t.dy_flat) { if (!encode_flat(&t.map_dy, p.wgt, p.K, (long long)p.N * p.P * p.Q)) return false; }
    else if (!encode_tall(&t.map_dy, p.wgt, p.K, p.N, p.P, p.Q, t.Wp, g.box_h, g.box_n, 1)) return false;
    if (t.a_flat) { if (!encode_flat(&t.map_a, p.act, p.C, (long long)p.N * p.H * p.W)) return false; }
    else if (!encode_tall(&t.map_a, p.act, p.C, p.N, p.H, p.W, t.Wp, g.box_h, g.box_n, t.es)) return false;
    t.partial = p.partial; t.out = (float*)p.out; t.status = conv_tc_status_word();
    memcpy(host_tc, &t, sizeof(t));
    return true;
}
size_t conv_wgrad_tc_prob_bytes() { return sizeof(TcWgradProb); }
int conv_wgrad_tc_ctas(const void* h) { const TcWgradProb* t = (const TcWgradProb*)h; return t->m_tiles * t->n_tiles * t->tap_groups * t->splits; }
size_t conv_wgrad_tc_smem(const void* h) { const TcWgradProb* t = (const TcWgradProb*)h; return std::max((size_t)t->stages * t->stage_bytes, (size_t)120 * 1024) + 1024; }
long long conv_wgrad_tc_out_elems(const void* h) { const TcWgradProb* t = (const TcWgradProb*)h; return (long long)t->taps * t->cout * t->cin; }

void launch_conv_wgrad_tc_probs(const void* d_tc, int nprob, int max_ctas, size_t max_smem, long long max_out, cudaStream_t s) {
    static bool configured = false;
    if (!configured) { cudaFuncSetAttribute(conv_wgrad_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(TC_SMEM_BUDGET + 1024)); configured = true; }
    conv_wgrad_tc_kernel<<<dim3(max_ctas, nprob), TC_THREADS, max_smem, s>>>((const TcWgradProb*)d_tc);
    long long gx = (max_out + 4 * WG_RED_THREADS - 1) / (4 * WG_RED_THREADS); if (gx > 1184) gx = 1184; if (gx < 1) gx = 1;
    wgrad_tc_reduce_kernel<<<dim3((unsigned)gx, nprob), WG_RED_THREADS, 0, s>>>((const TcWgradProb*)d_tc);
}

}  // namespace resist
