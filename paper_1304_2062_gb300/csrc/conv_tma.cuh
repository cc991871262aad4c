// 3x3 convolution (padding 1, NHWC bf16) as a persistent, warp-specialised
// implicit GEMM on the tcgen05 tensor cores with TMA operand loads:
//
//   D[m][n] = sum_k A(m, k) B(n, k),  m = output pixel, n = output channel,
//   k = tap * C + c,  A(m, tap * C + c) = In[pixel m shifted by tap][c],
//   B = a K-major [N][9 C] weight matrix.
//
// Tiles of D are 128 pixels (8 x 16 of one image; pairs of pixels with 32 output
// channels) by BN channels. TMA boxes bring the pixels around a tile, CK channels at a
// time, and BN x CK weights a tap, in the swizzled K-major layout the tensor core reads
// (CK = 64: 128-byte swizzle; CK = 32: 64-byte swizzle); the tensor map's out-of-bounds
// zero fill is the convolution's padding.
//
// Roles (one CTA per SM, tiles strided over CTAs):
//   warp 0, one thread   TMA producer: fills a ring of stages, each guarded by a "full"
//                        (transaction bytes) and an "empty" (tensor core done) mbarrier;
//   warp 1               allocates tensor memory and issues tcgen05.mma (M = 128, K = 16)
//                        into one of several accumulators, committing to "empty" per stage
//                        and to "acc full" per tile;
//   warps 2-9            epilogue, two groups of four: tcgen05.ld of the accumulator rows
//                        their lane quarter may access, the functor EPI, "acc empty" (so the
//                        next tiles' MMAs overlap it), and a TMA store.
//
// Every wait is bounded (about 2 s at the full clock). One that runs out sets *err and the
// shared abort flag; the CTA then stops, lets what it issued complete
// (bounded), releases its tensor memory and returns. CTAs that find *err
// set do nothing.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "conv_tc.cuh"
#include "wgrad_plan.h"

namespace se2n {
namespace nn {
namespace tma {

// The order in which an output's products of 16 channels are added. It is part of the
// result: another one moves a few stored BF16 values across a rounding boundary, and
// that spreads (a different order in one layer changes the network's output by 2e-3). With
// up to 64 (32 for 96 of them) channels a block and 32 or 64 outputs, images of whole 16 x 8
// tiles have always been summed blocks first, then horizontal and vertical offsets of the
// source; everything else taps first, then channels (taps of the weights: the source
// offsets run backwards where they are mirrored).
enum SumOrder {
    ORDER_BLOCKS = 0,  // (32- or 64-channel block of the kernel, sx, sy)
    ORDER_OFFSETS = 1, // (sx, sy, block): a 64-channel block in blocks of 32
    ORDER_TAPS = 2     // (tap, block)
};

// Geometry of one convolution launch (passed by value).
struct ConvGeo {
    int B, H, W, C;      // A tensor: B images of H x W pixels, C channels
    int bw, bh;          // tile shape in pixels (bw * bh == 128)
    int tiles_x, tiles_y, mtiles, ntiles, tiles;
    int nchunk;          // C / CK
    int flip;            // 1: taps mirrored (data gradient)
    int order;           // of the sums: SumOrder
};

// K-major matrix descriptor of dense rows of CK channels (8-row atoms).
template <int CK>
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)(16u >> 4) << 16;
    d |= (uint64_t)((uint32_t)(8 * CK * 2) >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)(CK == 64 ? 2 : 4) << 61;
    return d;
}

__device__ __forceinline__ void arrive_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, int c3,
                                            uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];\n" ::"r"(dst),
        "l"((uint64_t)map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int c0, int c1, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n" ::"r"(
            dst),
        "l"((uint64_t)map), "r"(c0), "r"(c1), "r"(bar)
        : "memory");
}

// Issued by one lane of a converged warp that runs the whole loop together: its
// control flow and descriptors are then warp-uniform, which an issuing loop inside
// "if (lane == 0)" is not (every instruction then moves its descriptors to
// uniform registers first: 32-channel layer 195 us against 130, batch 64).
__device__ __forceinline__ void mma_f16_elect(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                              uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n elect.sync _|q, 0xffffffff;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}
// NK products of 16 channels each, both operands 32 bytes further on every time. One
// election and one block of instructions: what the issuing warp spends on a product
// (some ten instructions with an election each, 50 cycles) is as much as the product takes
// with 32 or 64 columns.
template <int NK>
__device__ __forceinline__ void mma_chain_elect(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                                uint32_t accumulate) {
    static_assert(NK == 2 || NK == 4, "32 or 64 channels");
    if constexpr (NK == 2)
        asm volatile(
            "{\n .reg .pred p, q, t;\n .reg .b64 a, b;\n setp.ne.b32 p, %4, 0;\n setp.eq.b32 t, 0, 0;\n"
            " elect.sync _|q, 0xffffffff;\n add.s64 a, %1, 2;\n add.s64 b, %2, 2;\n"
            " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
            " @q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, t;\n}\n" ::"r"(tmem_d),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
    else
        asm volatile(
            "{\n .reg .pred p, q, t;\n .reg .b64 a, b, c, d, e, f;\n setp.ne.b32 p, %4, 0;\n setp.eq.b32 t, 0, 0;\n"
            " elect.sync _|q, 0xffffffff;\n add.s64 a, %1, 2;\n add.s64 b, %2, 2;\n add.s64 c, %1, 4;\n"
            " add.s64 d, %2, 4;\n add.s64 e, %1, 6;\n add.s64 f, %2, 6;\n"
            " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
            " @q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, t;\n"
            " @q tcgen05.mma.cta_group::1.kind::f16 [%0], c, d, %3, t;\n"
            " @q tcgen05.mma.cta_group::1.kind::f16 [%0], e, f, %3, t;\n}\n" ::"r"(tmem_d),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}
__device__ __forceinline__ void mma_commit_elect(uint32_t bar) {
    asm volatile(
        "{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n"
        " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(bar)
        : "memory");
}
// Bounded wait of a whole warp.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int *abort) {
    return __all_sync(0xffffffffu, tc::mbar_wait(bar, parity, abort));
}

__device__ __forceinline__ void tile_origin(const ConvGeo &g, int t, int &b, int &x0, int &y0, int &nt) {
    const int mt = t % g.mtiles;
    nt = t / g.mtiles;
    const int per_img = g.tiles_x * g.tiles_y;
    b = mt / per_img;
    const int r = mt - b * per_img;
    y0 = (r / g.tiles_x) * g.bh;
    x0 = (r % g.tiles_x) * g.bw;
}

// EPI provides
//   SMEM_FLOATS, prepare(sm, i, n)    constants copied to shared memory by the
//                                      epilogue threads i = 0..n-1 once per CTA
//   Pre, prefetch(m, n)               what compute(m, n) reads from device memory (may be loaded
//                                      before the accumulator is complete)
//   PrePix, prefetch_pixel(m)         the same for finish(m)
//   compute(m, n, v[16], float &state, sm, pre, valid, p[8])  the 16 outputs of pixel m, columns
//                                      n..n+15, as BF16 pairs; called by whole warps, of pixel 0
//                                      for lanes without one
//   compute_pair(m, n, v[2][16], float (&state)[2], sm, pre, pre1, valid, p[2][8])  the same of
//                                      pixels m and m + 1 (k_conv_pair)
//   writes(), second(n), column(n)    whether they are wanted, in which tensor column n goes and where
//   finish(m, float state, sm, pre)   after the last column group of pixel m
// ---------------------------------------------------------------------------
// Narrow layers (64 or 96 output channels): halo boxes and resident weights.
//
// Tiles are 8 x 16 pixels. For each channel block one TMA box brings the
// 10 x 18 pixels around a tile, and each of the nine taps is the same box read from
// pixel (sy + 1) * 10 + sx + 1 on: the operand's groups of eight rows are image rows,
// one box row (10 pixels) apart, and the swizzle is a function of the shared-memory
// address alone, so a group may start anywhere in a swizzle atom. 180 box rows feed
// the nine taps; the TMA unit writes box rows at 2.7 cycles each, and a box a horizontal
// offset makes 480 of them, one a tap 1152. (64 -> 64 channels, batch 64, 128 x 128: 76 us against
// 86 with a box a horizontal offset.) All weights of the layer (9 C x BN) are loaded into shared memory
// once per CTA, so the K loop moves no weight rows at all. Pixels of a tile outside the
// image are computed and not stored.
// ---------------------------------------------------------------------------

constexpr int HBW = 8, HBH = 16;              // tile 8 x 16 pixels
constexpr int HPITCH = HBW + 2;               // pixels a box row
constexpr int HROWS = HPITCH * (HBH + 2);     // 180 pixels a box
constexpr int kHaloThreads = 320;             // producer, MMA issuer and eight epilogue warps

template <int BN, int CK>
struct HaloCfg {
    static_assert(BN % 16 == 0 && BN >= 16 && BN <= 128, "narrow layers");
    static constexpr int A_BYTES = HROWS * CK * 2;
    static constexpr int STAGE = (A_BYTES + 1023) / 1024 * 1024;
    static constexpr int BBLK = BN * CK * 2;   // one (tap, channel block) of weights
    static constexpr int OB = BN % 64 == 0 ? 64 : 32;  // channels of an output box
    static constexpr int ACC_COLS = BN <= 32 ? 32 : BN <= 64 ? 64 : 128;
    static constexpr int NACC = 4;             // accumulators
    static constexpr int TMEM_COLS = NACC * ACC_COLS;
    static constexpr int SMEM_BUDGET = 196608;
};

// Outputs of these kernels leave through shared memory: every epilogue warp packs OB
// channels of its image rows into a buffer of its own (in the swizzled layout of a
// TMA box, so that the lanes' 16-byte stores do not meet) and stores it as one box.
// From registers a lane's 32 bytes a pixel are two stores of 16 bytes, each a partial
// sector among 32 lines (32 -> 32 channels with the pooling, batch 64, 256 x 256: 133 us
// against 153; 64 -> 64 at 128 x 128 67 against 76; 96 columns of data gradient, batch 32,
// 85 against 133).
// Pixels outside the image are clipped by the box.
constexpr int kOutBytes = 4096;  // a warp's buffer

template <int OB>
__device__ __forceinline__ void out_put(uint32_t buf, int row, int c, const uint32_t (&p)[8]) {
    const int key = OB == 64 ? row & 7 : (row >> 1) & 3, j = c >> 3;
    const uint32_t a = buf + (uint32_t)(row * OB * 2);
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(a + (uint32_t)((j ^ key) << 4)), "r"(p[0]), "r"(p[1]),
                 "r"(p[2]), "r"(p[3])
                 : "memory");
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(a + (uint32_t)(((j + 1) ^ key) << 4)), "r"(p[4]),
                 "r"(p[5]), "r"(p[6]), "r"(p[7])
                 : "memory");
}
// the warp's buffer may be written again
__device__ __forceinline__ void out_reuse(int lane) {
    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");
    __syncwarp();
}
__device__ __forceinline__ void out_store(uint32_t buf, const CUtensorMap *map, int c, int x, int y, int b, int lane) {
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    __syncwarp();
    if (lane == 0) {
        asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3, %4}], [%5];\n" ::"l"(
                         (uint64_t)map),
                     "r"(c), "r"(x), "r"(y), "r"(b), "r"(buf)
                     : "memory");
        asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
    }
}
__device__ __forceinline__ void out_drain(int lane) {
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory");
    __syncwarp();
}

// Descriptor of a tile's pixels in a box: image rows HPITCH pixels apart.
template <int CK>
__device__ __forceinline__ uint64_t sdesc_box(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)(16u >> 4) << 16;
    d |= (uint64_t)((uint32_t)(HPITCH * CK * 2) >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)(CK == 64 ? 2 : 4) << 61;
    return d;
}

template <int BN, int CK, class EPI>
__global__ void __launch_bounds__(kHaloThreads, 1)
    k_conv_halo(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                const __grid_constant__ CUtensorMap mapO, const __grid_constant__ CUtensorMap mapO2, const ConvGeo g,
                const EPI epi, int S, int *err) {
    using Cf = HaloCfg<BN, CK>;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    const int nblk = 9 * g.nchunk;                       // resident weight blocks
    const uint32_t wres = base;                          // nblk x BBLK
    const uint32_t stages = wres + nblk * Cf::BBLK;      // S x STAGE
    const uint32_t obuf = stages + S * Cf::STAGE;        // the epilogue warps' output buffers
    const uint32_t bar_w = obuf + 8 * kOutBytes;
    const uint32_t bar_full = bar_w + 8;
    const uint32_t bar_empty = bar_full + 8 * S;
    const uint32_t bar_afull = bar_empty + 8 * S;
    const uint32_t bar_aempty = bar_afull + 8 * Cf::NACC;
    const uint32_t tmem_slot = bar_aempty + 8 * Cf::NACC;
    volatile int *abort = (volatile int *)(smem_raw + (tmem_slot + 4 - raw));
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    // tiles t = nt * mtiles + mt; CTA c takes n tile c % ntiles and every
    // (gridDim.x / ntiles)-th m tile from c / ntiles (gridDim.x % ntiles == 0)
    const int first_tile = (blockIdx.x % g.ntiles) * g.mtiles + blockIdx.x / g.ntiles;
    const int end_tile = (blockIdx.x % g.ntiles + 1) * g.mtiles;
    const int tile_step = gridDim.x / g.ntiles;

    if (threadIdx.x == 0) {
        *abort = *(volatile int *)err;
        tc::mbar_init(bar_w, 1);
        for (int s = 0; s < S; ++s) {
            tc::mbar_init(bar_full + 8 * s, 1);
            tc::mbar_init(bar_empty + 8 * s, 1);
        }
        for (int a = 0; a < Cf::NACC; ++a) {
            tc::mbar_init(bar_afull + 8 * a, 1);
            tc::mbar_init(bar_aempty + 8 * a, 4);
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"((uint64_t)&mapA) : "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"((uint64_t)&mapB) : "memory");
    }
    __syncthreads();
    if (*abort) return;
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(tmem_slot),
                     "r"((uint32_t)Cf::TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    uint32_t tmem_base;
    asm volatile("ld.shared.u32 %0, [%1];\n" : "=r"(tmem_base) : "r"(tmem_slot));
    tmem_base = __shfl_sync(0xffffffffu, tmem_base, 0);

    if (warp == 0) {
        if (lane == 0) {
            // ---------------- TMA producer ----------------
            // this CTA's tiles all have the n tile blockIdx.x % ntiles: its weights stay resident
            const int nt0 = blockIdx.x % g.ntiles;
            arrive_expect_tx(bar_w, (uint32_t)(nblk * Cf::BBLK));
            for (int tap = 0; tap < 9; ++tap)
                for (int ch = 0; ch < g.nchunk; ++ch)
                    tma_load_2d(wres + (tap * g.nchunk + ch) * Cf::BBLK, &mapB, tap * g.C + ch * CK, nt0 * BN, bar_w);
            int s = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int t = first_tile; t < end_tile && ok; t += tile_step) {
                int b, x0, y0, nt;
                tile_origin(g, t, b, x0, y0, nt);
                for (int ch = 0; ch < g.nchunk; ++ch) {
                    if (!tc::mbar_wait(bar_empty + 8 * s, ph ^ 1u, abort)) {
                        ok = false;
                        break;
                    }
                    arrive_expect_tx(bar_full + 8 * s, Cf::A_BYTES);
                    tma_load_4d(stages + s * Cf::STAGE, &mapA, ch * CK, x0 - 1, y0 - 1, b, bar_full + 8 * s);
                    if (++s == S) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
            }
            if (!ok) {
                const long long t0 = clock64();
                while (clock64() - t0 < 200000LL) {
                }
            }
        }
    } else if (warp == 1) {
        {  // the whole warp
            // ---------------- MMA issuer ----------------
            constexpr uint32_t IDESC = tc::idesc_bf16_f32<BN>();
            const uint64_t a_desc0 = sdesc_box<CK>(stages), w_desc0 = sdesc<CK>(wres);
            const int wstep = (g.nchunk * Cf::BBLK) >> 4;  // weights of the next tap, in 16-byte units
            int s = 0, acc = 0;
            uint32_t ph = 0, aph = 0;
            bool ok = mbar_wait_warp(bar_w, 0, abort);
            uint32_t last_bar = 0, last_par = 0;
            for (int t = first_tile; t < end_tile && ok; t += tile_step) {
                if (!mbar_wait_warp(bar_aempty + 8 * acc, aph ^ 1u, abort)) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                const uint32_t d = tmem_base + (uint32_t)(acc * Cf::ACC_COLS);
                // weights of source offset t = 3 syi + sxi: tap t, or 8 - t when mirrored
                const uint64_t dw0 = w_desc0 + (g.flip ? (uint64_t)(8 * wstep) : 0);
                const uint64_t step = (uint64_t)(int64_t)(g.flip ? -wstep : wstep);
                for (int ch = 0; ch < g.nchunk; ++ch) {
                    const int sl = s + ch < S ? s + ch : s + ch - S;
                    if (!mbar_wait_warp(bar_full + 8 * sl, s + ch < S ? ph : ph ^ 1u, abort)) {
                        ok = false;
                        break;
                    }
                    if (g.order != ORDER_BLOCKS) continue;  // all blocks first
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    const uint64_t da = a_desc0 + (uint64_t)((uint32_t)(sl * Cf::STAGE) >> 4);
                    const uint64_t dw = dw0 + (uint64_t)((uint32_t)(ch * Cf::BBLK) >> 4);
#pragma unroll
                    for (int sxi = 0; sxi < 3; ++sxi)
#pragma unroll
                        for (int syi = 0; syi < 3; ++syi)
                            mma_chain_elect<CK / 16>(d, da + (uint64_t)((syi * HPITCH + sxi) * CK * 2 / 16),
                                                     dw + (uint64_t)(syi * 3 + sxi) * step, IDESC,
                                                     syi + sxi > 0 || ch > 0 ? 1u : 0u);
                    mma_commit_elect(bar_empty + 8 * sl);
                    last_bar = bar_empty + 8 * sl;
                    last_par = s + ch < S ? ph : ph ^ 1u;
                }
                if (!ok) break;
                if (g.order != ORDER_BLOCKS) {
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    for (int tap = 0; tap < 9; ++tap) {
                        const int t = g.flip ? 8 - tap : tap;
                        for (int ch = 0; ch < g.nchunk; ++ch) {
                            const int sl = s + ch < S ? s + ch : s + ch - S;
                            const uint64_t da = a_desc0 + (uint64_t)((uint32_t)(sl * Cf::STAGE + (t / 3 * HPITCH + t % 3) * CK * 2) >> 4);
                            const uint64_t dw = w_desc0 + (uint64_t)((uint32_t)((tap * g.nchunk + ch) * Cf::BBLK) >> 4);
                            mma_chain_elect<CK / 16>(d, da, dw, IDESC, tap + ch > 0 ? 1u : 0u);
                            if (tap == 8) {
                                mma_commit_elect(bar_empty + 8 * sl);
                                last_bar = bar_empty + 8 * sl;
                                last_par = s + ch < S ? ph : ph ^ 1u;
                            }
                        }
                    }
                }
                s += g.nchunk;
                if (s >= S) {
                    s -= S;
                    ph ^= 1u;
                }
                mma_commit_elect(bar_afull + 8 * acc);
                if (++acc == Cf::NACC) {
                    acc = 0;
                    aph ^= 1u;
                }
            }
            if (!ok && last_bar) tc::mbar_wait(last_bar, last_par, nullptr);
        }
    } else {
        // ---------------- epilogue (two groups of four warps) ----------------
        // The groups take the CTA's tiles in turn, so each has two tiles' time
        // for one; what a tile's outputs need from device memory is loaded
        // before its accumulator is waited for.
        __shared__ float epi_const[EPI::SMEM_FLOATS];
        epi.prepare(epi_const, threadIdx.x - 64, 256);
        asm volatile("bar.sync 1, 256;\n" ::: "memory");  // the epilogue warps only
        const int q = warp & 3, group = (warp - 2) >> 2;
        const uint32_t buf = obuf + (uint32_t)(warp - 2) * kOutBytes;
        int acc = group;
        uint32_t aph = 0;
        for (int t = first_tile + group * tile_step; t < end_tile; t += 2 * tile_step) {
            int b, x0, y0, nt;
            tile_origin(g, t, b, x0, y0, nt);
            const int r = q * 32 + lane;
            const int y = y0 + r / HBW, x = x0 + r % HBW;
            const bool valid = x < g.W && y < g.H;
            const int m = valid ? (b * g.H + y) * g.W + x : 0;
            typename EPI::Pre pre[BN / 16];
#pragma unroll
            for (int j = 0; j < BN / 16; ++j) pre[j] = epi.prefetch(m, nt * BN + 16 * j);
            const typename EPI::PrePix pp = epi.prefetch_pixel(m);
            if (!mbar_wait_warp(bar_afull + 8 * acc, aph, abort)) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * Cf::ACC_COLS);
            float state = 0.0f;
#pragma unroll
            for (int j = 0; j < BN / 16; ++j) {
                uint32_t v[16];
                tc::tmem_ld16(taddr + (uint32_t)(16 * j), v);
                float f[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) f[i] = __uint_as_float(v[i]);
                const int n = nt * BN + 16 * j;
                uint32_t p[8];
                epi.compute(m, n, f, state, epi_const, pre[j], valid, p);
                if (epi.writes()) {
                    constexpr int OB = Cf::OB;
                    if (16 * j % OB == 0) out_reuse(lane);
                    out_put<OB>(buf, lane, 16 * j % OB, p);
                    if (16 * (j + 1) % OB == 0)
                        out_store(buf, epi.second(n) ? &mapO2 : &mapO, epi.column(n + 16 - OB), x0, y0 + 4 * q, b, lane);
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
            __syncwarp();
            if (lane == 0) arrive(bar_aempty + 8 * acc);
            if (valid) epi.finish(m, state, epi_const, pp);
            acc += 2;
            if (acc >= Cf::NACC) {
                acc = group;
                aph ^= 1u;
            }
        }
        out_drain(lane);
    }
    __syncthreads();
    if (threadIdx.x == 0 && *abort) atomicExch(err, 1);
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base),
                     "r"((uint32_t)Cf::TMEM_COLS));
    }
}


// ---------------------------------------------------------------------------
// Layers with 32 output channels: columns of two pixels.
//
// A matrix product of 128 rows, 16 channels and 32 columns takes as long as one of 64
// columns (about 48 cycles: reading the pixels from shared memory), and that is what
// bounds k_conv_halo there. So a row of the operand is a pair of pixels, the output
// 2 x 32 columns. Of the pair itself, the even pixels' channels go into both outputs
// (horizontal source offsets 0 and -1), so do the odd ones' (1 and 0): 64 columns
// each, whose weights are neighbours when a row of taps is kept in the order 1, 0, -1.
// The odd pixel of the pair before belongs to the even output alone, the even pixel of the
// next to the odd one: 32 columns. 24 products a 32 channels and 256 pixels
// instead of 36. The pixels of either parity are a box of their own (of the tensor as
// W / 2 columns of 2 C channels).
// Measured (forward, batch 64, 256 x 256): 32 -> 32 channels 130 us with the pooling (169),
// 96 -> 32 236 (317), 32 -> 32 with the head 98 (137).
// ---------------------------------------------------------------------------

struct PairCfg {
    static constexpr int A_BYTES = HROWS * 64;  // 32 channels of the pixels of one parity
    static constexpr int A_SLOT = (A_BYTES + 1023) / 1024 * 1024;
    static constexpr int STAGE = 2 * A_SLOT;
    static constexpr int BBLK = 32 * 64;        // one (tap, channel block) of weights
    static constexpr int ACC_COLS = 64, NACC = 4, TMEM_COLS = NACC * ACC_COLS;
    static constexpr int SMEM_BUDGET = 196608;
};

template <class EPI>
__global__ void __launch_bounds__(kHaloThreads, 1)
    k_conv_pair(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                const __grid_constant__ CUtensorMap mapO, const __grid_constant__ CUtensorMap mapO2, const ConvGeo g,
                const EPI epi, int S, int *err) {
    using Cf = PairCfg;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    const int nblk = 9 * g.nchunk;                       // resident weight blocks
    const uint32_t wres = base;                          // nblk x BBLK
    const uint32_t stages = wres + nblk * Cf::BBLK;      // S x STAGE
    const uint32_t obuf = stages + S * Cf::STAGE;        // the epilogue warps' output buffers
    const uint32_t bar_w = obuf + 8 * kOutBytes;
    const uint32_t bar_full = bar_w + 8;
    const uint32_t bar_empty = bar_full + 8 * S;
    const uint32_t bar_afull = bar_empty + 8 * S;
    const uint32_t bar_aempty = bar_afull + 8 * Cf::NACC;
    const uint32_t tmem_slot = bar_aempty + 8 * Cf::NACC;
    volatile int *abort = (volatile int *)(smem_raw + (tmem_slot + 4 - raw));
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int first_tile = blockIdx.x, end_tile = g.mtiles, tile_step = gridDim.x;

    if (threadIdx.x == 0) {
        *abort = *(volatile int *)err;
        tc::mbar_init(bar_w, 1);
        for (int s = 0; s < S; ++s) {
            tc::mbar_init(bar_full + 8 * s, 1);
            tc::mbar_init(bar_empty + 8 * s, 1);
        }
        for (int a = 0; a < Cf::NACC; ++a) {
            tc::mbar_init(bar_afull + 8 * a, 1);
            tc::mbar_init(bar_aempty + 8 * a, 4);
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"((uint64_t)&mapA) : "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"((uint64_t)&mapB) : "memory");
    }
    __syncthreads();
    if (*abort) return;
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(tmem_slot),
                     "r"((uint32_t)Cf::TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    uint32_t tmem_base;
    asm volatile("ld.shared.u32 %0, [%1];\n" : "=r"(tmem_base) : "r"(tmem_slot));
    tmem_base = __shfl_sync(0xffffffffu, tmem_base, 0);

    if (warp == 0) {
        if (lane == 0) {
            // ---------------- TMA producer ----------------
            arrive_expect_tx(bar_w, (uint32_t)(nblk * Cf::BBLK));
            for (int i = 0; i < nblk; ++i) {
                // block (syi, ch, j): the tap of source offset (syi - 1, 1 - j), mirrored when flip
                const int j = i % 3, ch = i / 3 % g.nchunk, syi = i / (3 * g.nchunk);
                const int tap = g.flip ? 8 - (syi * 3 + 2 - j) : syi * 3 + 2 - j;
                tma_load_2d(wres + i * Cf::BBLK, &mapB, tap * g.C + ch * 32, 0, bar_w);
            }
            int s = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int t = first_tile; t < end_tile && ok; t += tile_step) {
                int b, x0, y0, nt;
                tile_origin(g, t, b, x0, y0, nt);
                for (int ch = 0; ch < g.nchunk; ++ch) {
                    if (!tc::mbar_wait(bar_empty + 8 * s, ph ^ 1u, abort)) {
                        ok = false;
                        break;
                    }
                    arrive_expect_tx(bar_full + 8 * s, 2 * Cf::A_BYTES);
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        tma_load_4d(stages + s * Cf::STAGE + h * Cf::A_SLOT, &mapA, h * g.C + ch * 32, x0 - 1, y0 - 1, b,
                                    bar_full + 8 * s);
                    if (++s == S) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
            }
            if (!ok) {
                const long long t0 = clock64();
                while (clock64() - t0 < 200000LL) {
                }
            }
        }
    } else if (warp == 1) {
        {  // the whole warp
            // ---------------- MMA issuer ----------------
            constexpr uint32_t IDESC2 = tc::idesc_bf16_f32<64>(), IDESC1 = tc::idesc_bf16_f32<32>();
            const uint64_t a_desc0 = sdesc_box<32>(stages), w_desc0 = sdesc<32>(wres);
            const uint64_t wrow = (uint64_t)(uint32_t)((3 * g.nchunk * Cf::BBLK) >> 4);  // the next vertical offset
            int s = 0, acc = 0;
            uint32_t ph = 0, aph = 0;
            bool ok = mbar_wait_warp(bar_w, 0, abort);
            uint32_t last_bar = 0, last_par = 0;
            for (int t = first_tile; t < end_tile && ok; t += tile_step) {
                if (!mbar_wait_warp(bar_aempty + 8 * acc, aph ^ 1u, abort)) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                const uint32_t d = tmem_base + (uint32_t)(acc * Cf::ACC_COLS);
                // The products of 32 channels with one row of taps, X = 0 .. 3: the odd pixel of the
                // pair before (source offset -1 of the even output), the even pixel (0 of the even, -1
                // of the odd output), the odd one (1 and 0), the even pixel of the next (1 of the odd
                // output). Either output meets its offsets in ascending order as X ascends, in
                // descending order as it descends. first: the first of this X, whose outputs met
                // there for the first time are set, not added to.
                const bool desc = g.order == ORDER_TAPS && g.flip;
                auto products = [&](int X, int syi, uint64_t da, uint64_t dw, bool first) {
                    constexpr uint32_t W1 = Cf::BBLK / 16, ODD = Cf::A_SLOT / 16, PX = 64 / 16;
                    const uint64_t a = da + (uint64_t)(syi * HPITCH * PX), w = dw + (uint64_t)(uint32_t)syi * wrow;
                    if (X == 0) {
                        mma_chain_elect<2>(d, a + ODD, w + 2 * W1, IDESC1, first && !desc ? 0u : 1u);
                    } else if (X == 3) {
                        mma_chain_elect<2>(d + 32u, a + 2 * PX, w, IDESC1, first && desc ? 0u : 1u);
                    } else {
                        const uint64_t ax = a + PX + (X == 2 ? ODD : 0u), wx = w + (X == 1 ? W1 : 0u);
                        if (first && (X == 1) != desc) {
                            mma_chain_elect<2>(d, ax, wx, IDESC1, desc ? 0u : 1u);
                            mma_chain_elect<2>(d + 32u, ax, wx + W1, IDESC1, desc ? 1u : 0u);
                        } else {
                            mma_chain_elect<2>(d, ax, wx, IDESC2, 1u);
                        }
                    }
                };
                for (int ch = 0; ch < g.nchunk; ++ch) {
                    const int sl = s + ch < S ? s + ch : s + ch - S;
                    if (!mbar_wait_warp(bar_full + 8 * sl, s + ch < S ? ph : ph ^ 1u, abort)) {
                        ok = false;
                        break;
                    }
                    if (g.order != ORDER_BLOCKS) continue;  // all blocks first
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    const uint64_t da = a_desc0 + (uint64_t)((uint32_t)(sl * Cf::STAGE) >> 4);
                    const uint64_t dw = w_desc0 + (uint64_t)((uint32_t)(3 * ch * Cf::BBLK) >> 4);
#pragma unroll
                    for (int X = 0; X < 4; ++X)
#pragma unroll
                        for (int syi = 0; syi < 3; ++syi) products(X, syi, da, dw, ch == 0 && syi == 0);
                    mma_commit_elect(bar_empty + 8 * sl);
                    last_bar = bar_empty + 8 * sl;
                    last_par = s + ch < S ? ph : ph ^ 1u;
                }
                if (!ok) break;
                if (g.order != ORDER_BLOCKS) {
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
#pragma unroll 1
                    for (int i = 0; i < 12; ++i) {
                        const int X = g.order == ORDER_OFFSETS ? i / 3 : desc ? 3 - (i & 3) : i & 3;
                        const int syi = g.order == ORDER_OFFSETS ? i % 3 : desc ? 2 - (i >> 2) : i >> 2;
                        const bool first = g.order == ORDER_OFFSETS ? syi == 0 : i < 4;
                        for (int ch = 0; ch < g.nchunk; ++ch) {
                            const int sl = s + ch < S ? s + ch : s + ch - S;
                            products(X, syi, a_desc0 + (uint64_t)((uint32_t)(sl * Cf::STAGE) >> 4),
                                     w_desc0 + (uint64_t)((uint32_t)(3 * ch * Cf::BBLK) >> 4), first && ch == 0);
                        }
                    }
                    for (int ch = 0; ch < g.nchunk; ++ch) {
                        const int sl = s + ch < S ? s + ch : s + ch - S;
                        mma_commit_elect(bar_empty + 8 * sl);
                        last_bar = bar_empty + 8 * sl;
                        last_par = s + ch < S ? ph : ph ^ 1u;
                    }
                }
                s += g.nchunk;
                if (s >= S) {
                    s -= S;
                    ph ^= 1u;
                }
                mma_commit_elect(bar_afull + 8 * acc);
                if (++acc == Cf::NACC) {
                    acc = 0;
                    aph ^= 1u;
                }
            }
            if (!ok && last_bar) tc::mbar_wait(last_bar, last_par, nullptr);
        }
    } else {
        // ---------------- epilogue (two groups of four warps) ----------------
        // The groups take the CTA's tiles in turn, so each has two tiles' time
        // for one; what a tile's outputs need from device memory is loaded
        // before its accumulator is waited for.
        __shared__ float epi_const[EPI::SMEM_FLOATS];
        epi.prepare(epi_const, threadIdx.x - 64, 256);
        asm volatile("bar.sync 1, 256;\n" ::: "memory");  // the epilogue warps only
        const int q = warp & 3, group = (warp - 2) >> 2;
        const uint32_t buf = obuf + (uint32_t)(warp - 2) * kOutBytes;
        int acc = group;
        uint32_t aph = 0;
        for (int t = first_tile + group * tile_step; t < end_tile; t += 2 * tile_step) {
            int b, x0, y0, nt;
            tile_origin(g, t, b, x0, y0, nt);
            const int r = q * 32 + lane;
            const int y = y0 + r / HBW, x = x0 + r % HBW;
            const bool valid = x < g.W && y < g.H;
            const int m = valid ? ((b * g.H + y) * g.W + x) * 2 : 0;  // the even pixel
            typename EPI::Pre pre[2][2];
            typename EPI::PrePix pp[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
#pragma unroll
                for (int j = 0; j < 2; ++j) pre[h][j] = epi.prefetch(m + h, 16 * j);
                pp[h] = epi.prefetch_pixel(m + h);
            }
            if (!mbar_wait_warp(bar_afull + 8 * acc, aph, abort)) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * Cf::ACC_COLS);
            float state[2] = {0.0f, 0.0f};
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                float f[2][16];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t v[16];
                    tc::tmem_ld16(taddr + (uint32_t)(32 * h + 16 * j), v);
#pragma unroll
                    for (int i = 0; i < 16; ++i) f[h][i] = __uint_as_float(v[i]);
                }
                uint32_t p[2][8];
                epi.compute_pair(m, 16 * j, f, state, epi_const, pre[0][j], pre[1][j], valid, p);
                if (epi.writes()) {
                    if (j == 0) out_reuse(lane);
                    out_put<32>(buf, 2 * lane, 16 * j, p[0]);
                    out_put<32>(buf, 2 * lane + 1, 16 * j, p[1]);
                    if (j == 1) out_store(buf, &mapO, 0, 2 * x0, y0 + 4 * q, b, lane);
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
            __syncwarp();
            if (lane == 0) arrive(bar_aempty + 8 * acc);
            if (valid) {
                epi.finish(m, state[0], epi_const, pp[0]);
                epi.finish(m + 1, state[1], epi_const, pp[1]);
            }
            acc += 2;
            if (acc >= Cf::NACC) {
                acc = group;
                aph ^= 1u;
            }
        }
        out_drain(lane);
    }
    __syncthreads();
    if (threadIdx.x == 0 && *abort) atomicExch(err, 1);
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base),
                     "r"((uint32_t)Cf::TMEM_COLS));
    }
}


// ---------------------------------------------------------------------------
// Wide layers (64 channels a chunk, weights too large to stay in shared
// memory): halo boxes and groups of tiles that share each weight.
//
// With 128 pixels and BN weight rows loaded for every tap and 64 channels (four MMAs) the
// layers are bound by what L2 delivers (14 TB/s, tensor pipe 23 .. 38 % active). Here the boxes
// of 10 x 18 pixels of a tile, one a chunk, stay for all nine taps (180 rows a chunk instead
// of 1152), and each tap's weights serve the G tiles of a group, each with an
// accumulator of its own: per tile and chunk 23 KB + 9 BN / G * 128 bytes instead of
// 9 (16 KB + BN * 128). G is as large as the accumulators, four boxes a group and
// enough groups for every SM allow. Roles as in k_conv_halo, with rings of boxes (in the
// order of the first tap, released in that order with the last) and of weights. The rings
// share what there is of shared memory. (Two or three chunks of weights a slot, or one
// tile a group and twice the boxes, are no faster: 192 -> 64 281 and 403 us.)
// Measured (forward, batch 64, 256 x 256): 192 -> 64 channels 292 us (381 with a box a
// tap), all layers of 128 and 256 outputs 487 (495).
// ---------------------------------------------------------------------------

template <int BN>
struct GroupCfg {
    static_assert(BN == 64 || BN == 128, "accumulators of 64 or 128 columns");
    static constexpr int A_BYTES = HROWS * 128;     // one box
    static constexpr int A_SLOT = (A_BYTES + 1023) / 1024 * 1024;
    static constexpr int W_BYTES = BN * 128;        // the weights of a tap and chunk
    static constexpr int NACC = 512 / BN, GMAX = NACC / 2;  // accumulators; tiles a group at most
    static constexpr int AMAX = 6, WMAX = 8;        // ring slots at most
    static constexpr int OB = 32, OUT_BYTES = 2048; // channels of an output box, a warp's buffer
    static constexpr int SMEM_BUDGET = 212992;      // both rings
    static constexpr int SMEM_REST = 1024 + 8 * OUT_BYTES + 512;
};

template <int BN, class EPI>
__global__ void __launch_bounds__(kHaloThreads, 1)
    k_conv_group(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                const __grid_constant__ CUtensorMap mapO, const __grid_constant__ CUtensorMap mapO2, const ConvGeo g,
                 const EPI epi, int G, int AS, int WS, int *err) {
    using Cf = GroupCfg<BN>;
    constexpr int NACC = Cf::NACC;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    const uint32_t wbase = base + AS * Cf::A_SLOT;
    const uint32_t obuf = wbase + WS * Cf::W_BYTES;  // the epilogue warps' output buffers
    const uint32_t bar_full = obuf + 8 * Cf::OUT_BYTES;
    const uint32_t bar_empty = bar_full + 8 * AS;
    const uint32_t bar_wfull = bar_empty + 8 * AS;
    const uint32_t bar_wempty = bar_wfull + 8 * WS;
    const uint32_t bar_afull = bar_wempty + 8 * WS;
    const uint32_t bar_aempty = bar_afull + 8 * NACC;
    const uint32_t tmem_slot = bar_aempty + 8 * NACC;
    volatile int *abort = (volatile int *)(smem_raw + (tmem_slot + 4 - raw));
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    // groups u = nt * mgroups + mg: tiles mg * G .. of n tile nt
    const int mgroups = (g.mtiles + G - 1) / G, groups = mgroups * g.ntiles;

    if (threadIdx.x == 0) {
        *abort = *(volatile int *)err;
        for (int s = 0; s < AS; ++s) {
            tc::mbar_init(bar_full + 8 * s, 1);
            tc::mbar_init(bar_empty + 8 * s, 1);
        }
        for (int s = 0; s < WS; ++s) {
            tc::mbar_init(bar_wfull + 8 * s, 1);
            tc::mbar_init(bar_wempty + 8 * s, 1);
        }
        for (int a = 0; a < NACC; ++a) {
            tc::mbar_init(bar_afull + 8 * a, 1);
            tc::mbar_init(bar_aempty + 8 * a, 4);
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"((uint64_t)&mapA) : "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"((uint64_t)&mapB) : "memory");
    }
    __syncthreads();
    if (*abort) return;
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(tmem_slot), "r"(512u));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    uint32_t tmem_base;
    asm volatile("ld.shared.u32 %0, [%1];\n" : "=r"(tmem_base) : "r"(tmem_slot));
    tmem_base = __shfl_sync(0xffffffffu, tmem_base, 0);

    // tiles t0 .. t0 + n - 1 (in tile_origin's numbering) of group u
    auto group_tiles = [&](int u, int &t0, int &n) {
        const int nt = u / mgroups, m0 = (u - nt * mgroups) * G;
        t0 = nt * g.mtiles + m0;
        n = min(G, g.mtiles - m0);
    };

    if (warp == 0) {
        if (lane == 0) {
            // ---------------- TMA producer ----------------
            int s = 0, ws = 0;
            uint32_t ph = 0, wph = 0;
            bool ok = true;
            for (int u = blockIdx.x; u < groups && ok; u += gridDim.x) {
                int t0, n;
                group_tiles(u, t0, n);
                for (int tap = 0; tap < 9 && ok; ++tap)
                    for (int ch = 0; ch < g.nchunk && ok; ++ch) {
                        if (!tc::mbar_wait(bar_wempty + 8 * ws, wph ^ 1u, abort)) {
                            ok = false;
                            break;
                        }
                        arrive_expect_tx(bar_wfull + 8 * ws, Cf::W_BYTES);
                        tma_load_2d(wbase + ws * Cf::W_BYTES, &mapB, tap * g.C + ch * 64, (t0 / g.mtiles) * BN,
                                    bar_wfull + 8 * ws);
                        if (++ws == WS) {
                            ws = 0;
                            wph ^= 1u;
                        }
                        for (int i = 0; i < n && tap == 0; ++i) {
                            int b, x0, y0, nt;
                            tile_origin(g, t0 + i, b, x0, y0, nt);
                            if (!tc::mbar_wait(bar_empty + 8 * s, ph ^ 1u, abort)) {
                                ok = false;
                                break;
                            }
                            arrive_expect_tx(bar_full + 8 * s, Cf::A_BYTES);
                            tma_load_4d(base + s * Cf::A_SLOT, &mapA, ch * 64, x0 - 1, y0 - 1, b, bar_full + 8 * s);
                            if (++s == AS) {
                                s = 0;
                                ph ^= 1u;
                            }
                        }
                    }
            }
            if (!ok) {
                // loads already issued finish on their own within microseconds
                const long long t0 = clock64();
                while (clock64() - t0 < 200000LL) {
                }
            }
        }
    } else if (warp == 1) {
        {  // the whole warp
            // ---------------- MMA issuer ----------------
            constexpr uint32_t IDESC = tc::idesc_bf16_f32<BN>();
            const uint64_t a_desc0 = sdesc_box<64>(base), w_desc0 = sdesc<64>(wbase);
            int s = 0, ws = 0, acc0 = 0;  // acc0: the group's first accumulator
            uint32_t ph = 0, wph = 0, aph = 0;
            bool ok = true;
            for (int u = blockIdx.x; u < groups && ok; u += gridDim.x) {
                int t0, n;
                group_tiles(u, t0, n);
                uint32_t p = aph;
                for (int i = 0; i < n; ++i) {
                    const int acc = acc0 + i < NACC ? acc0 + i : acc0 + i - NACC;
                    if (acc0 + i == NACC) p ^= 1u;
                    if (!mbar_wait_warp(bar_aempty + 8 * acc, p ^ 1u, abort)) {
                        ok = false;
                        break;
                    }
                }
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                for (int tap = 0; tap < 9 && ok; ++tap) {
                    const int t = g.flip ? 8 - tap : tap;  // source offset 3 (sy + 1) + sx + 1
                    const uint64_t off = a_desc0 + (uint64_t)(uint32_t)((t / 3 * HPITCH + t % 3) * 8);
                    // the boxes of (chunk, tile) are slots s + ch n + i (mod AS), waited for with
                    // the first tap and released with the last
                    int sl = s;
                    uint32_t slp = ph;
                    for (int ch = 0; ch < g.nchunk; ++ch) {
                        if (!mbar_wait_warp(bar_wfull + 8 * ws, wph, abort)) {
                            ok = false;
                            break;
                        }
                        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                        const uint64_t dw = w_desc0 + (uint64_t)((uint32_t)ws * (Cf::W_BYTES / 16));
                        int acc = acc0;
                        for (int i = 0; i < n; ++i) {
                            if (tap == 0) {
                                if (!mbar_wait_warp(bar_full + 8 * sl, slp, abort)) {
                                    ok = false;
                                    break;
                                }
                                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                            }
                            mma_chain_elect<4>(tmem_base + (uint32_t)(acc * BN),
                                               off + (uint64_t)((uint32_t)sl * (Cf::A_SLOT / 16)), dw, IDESC,
                                               tap + ch > 0 ? 1u : 0u);
                            if (tap == 8) mma_commit_elect(bar_empty + 8 * sl);
                            if (++acc == NACC) acc = 0;
                            if (++sl == AS) {
                                sl = 0;
                                slp ^= 1u;
                            }
                        }
                        if (!ok) break;
                        mma_commit_elect(bar_wempty + 8 * ws);
                        if (++ws == WS) {
                            ws = 0;
                            wph ^= 1u;
                        }
                    }
                }
                if (!ok) break;
                s += n * g.nchunk;
                if (s >= AS) {
                    s -= AS;
                    ph ^= 1u;
                }
                for (int i = 0; i < n; ++i) {
                    mma_commit_elect(bar_afull + 8 * acc0);
                    if (++acc0 == NACC) {
                        acc0 = 0;
                        aph ^= 1u;
                    }
                }
            }
            if (!ok) {
                // tensor core idle before release
                mma_commit_elect(bar_wempty + 8 * ws);
                tc::mbar_wait(bar_wempty + 8 * ws, wph, nullptr);
            }
        }
    } else {
        // ---------------- epilogue (two groups of four warps, as in k_conv_halo) ----------------
        __shared__ float epi_const[EPI::SMEM_FLOATS];
        epi.prepare(epi_const, threadIdx.x - 64, 256);
        asm volatile("bar.sync 1, 256;\n" ::: "memory");  // the epilogue warps only
        const int q = warp & 3, half = (warp - 2) >> 2;
        const uint32_t buf = obuf + (uint32_t)(warp - 2) * Cf::OUT_BYTES;
        int acc = 0;
        uint32_t aph = 0;
        int turn = 0;
        bool ok = true;
        for (int u = blockIdx.x; u < groups && ok; u += gridDim.x) {
            int t0, n;
            group_tiles(u, t0, n);
            for (int i = 0; i < n; ++i, turn ^= 1) {
                if (turn == half) {
                    int b, x0, y0, nt;
                    tile_origin(g, t0 + i, b, x0, y0, nt);
                    const int r = q * 32 + lane;
                    const int y = y0 + r / HBW, x = x0 + r % HBW;
                    const bool valid = x < g.W && y < g.H;
                    const int m = valid ? (b * g.H + y) * g.W + x : 0;
                    if (!mbar_wait_warp(bar_afull + 8 * acc, aph, abort)) {
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * BN);
                    float state = 0.0f;
#pragma unroll 2
                    for (int j = 0; j < BN / 16; ++j) {
                        const typename EPI::Pre pre = epi.prefetch(m, nt * BN + 16 * j);
                        uint32_t v[16];
                        tc::tmem_ld16(taddr + (uint32_t)(16 * j), v);
                        float f[16];
#pragma unroll
                        for (int c = 0; c < 16; ++c) f[c] = __uint_as_float(v[c]);
                        const int n = nt * BN + 16 * j;
                        uint32_t p[8];
                        epi.compute(m, n, f, state, epi_const, pre, valid, p);
                        if (16 * j % Cf::OB == 0) out_reuse(lane);
                        out_put<Cf::OB>(buf, lane, 16 * j % Cf::OB, p);
                        if (16 * (j + 1) % Cf::OB == 0)
                            out_store(buf, epi.second(n) ? &mapO2 : &mapO, epi.column(n + 16 - Cf::OB), x0, y0 + 4 * q, b,
                                      lane);
                    }
                    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                    __syncwarp();
                    if (lane == 0) arrive(bar_aempty + 8 * acc);
                    if (valid) epi.finish(m, state, epi_const, epi.prefetch_pixel(m));
                }
                if (++acc == NACC) {
                    acc = 0;
                    aph ^= 1u;
                }
            }
        }
        out_drain(lane);
    }
    __syncthreads();
    if (threadIdx.x == 0 && *abort) atomicExch(err, 1);
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base), "r"(512u));
    }
}

// ---------------------------------------------------------------------------
// Weight gradient: dW[co][tap * C + ci] += sum over pixels p of
// In[p shifted by tap][ci] * gz[p][co], as D[m][n] = sum over k of A(m, k) B(n, k)
// with k the pixels. Both operands come from NHWC tensors, so they are MN-major
// in shared memory: a TMA box of 64 channels x BKX pixels x some image rows lands
// as one 128-byte swizzled row a pixel.
//
// What bounds it is reading the operands out of shared memory (about 80 cycles a
// product of 128 x 64 x 16), and with few channels the rate at which the TMA unit writes
// box rows (2.7 cycles a row, whether of 64 or of 128 bytes), so the kernel loads few and
// full ones and wastes few products:
//  * A box of In holds the R + 2 image rows and BKX + 2 columns around a block of
//    R x BKX pixels of gz. Every tap reads it from another pixel on (the swizzle is a
//    function of the shared-memory address alone), and two taps are the two 64-row
//    groups of one M = 128 operand, the leading byte offset their distance:
//    (dy -1, 0) of each column offset, one image row apart, and dy 1 of two
//    neighbouring column offsets, one pixel apart. 5 products for 9 taps, and 2.3 box
//    rows a pixel of gz (6 products and 5.1 rows with a box a column offset, 15 rows
//    with one a tap and operand).
//  * Layers whose channels are not whole groups of 64 (C = 32, 96, and 8, the
//    first layer's) are read with F = 2 or 8 neighbouring pixels as one column,
//    tensors of F C channels and W / F columns: D of a column offset s then
//    holds, for pixel px of In's column and pg of gz's, the tap
//    dx = F s + px - pg; s = -1, 0, 1 give every combination that is a tap, the
//    others are left out by the epilogue (or not loaded, where a group of 64
//    channels holds no such pixels). 1 / F of the box rows.
// A unit of work is (64 channels of In, 64 of gz, a range of pixel blocks),
// accumulated in tensor memory (up to 5 tiles of 64 columns) and added to dW with FP32
// atomics. The tensor core's sums truncate, so a sum loses bits in proportion to its
// length, and the length is part of the result (4e-5 of a gradient of 32 images when it
// is a third): wgrad_plan.h ends every sum where it ended when a unit was a tile of
// 128 (tap, channel) rows, or earlier, however long the range of a CTA is. Up to three
// CTAs share a unit's tiles.
// Measured (batch 32, 256 x 256): all 14 layers 1540 us (4832 with a box a tap and
// operand; 888 with as many ranges as SMs).
// ---------------------------------------------------------------------------

constexpr int kWgXSlots = 3, kWgGSlots = 2;  // ring slots of In and of gz
// a box of In, and its slot: the last operand's second group may end one pixel behind it
template <int BKX>
constexpr int kWgXBytes = (kWgR + 2) * (BKX + 2) * 128;
template <int BKX>
constexpr int kWgXSlot = (kWgXBytes<BKX> + 128 + 1023) / 1024 * 1024;

// MN-major matrix descriptor, 128-byte swizzle: leading byte offset = stride
// between 64-row groups, stride byte offset = stride between 8-pixel groups.
__device__ __forceinline__ uint64_t sdesc_mn(uint32_t saddr, uint32_t lbo) {
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)(1024u >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// kind::f16, D FP32, A and B BF16, both MN-major.
template <int N>
__device__ __forceinline__ constexpr uint32_t idesc_bf16_mn() {
    return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(128 >> 4) << 24);
}

template <int BKX>
__global__ void __launch_bounds__(192, 1)
    k_wgrad_tma(const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapG, const WgradGeo g,
                float *dw, int *err) {
    constexpr int R = kWgR, XS = kWgXSlots, GS = kWgGSlots, TMEM_COLS = 512;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    constexpr uint32_t ROW = (BKX + 2) * 128u, GROW = BKX * 128u;  // one image row of a box of In, of gz
    constexpr uint32_t X_BYTES = kWgXBytes<BKX>, X_SLOT = kWgXSlot<BKX>, G_BYTES = R * GROW;
    const uint32_t gbase = base + XS * X_SLOT;
    const uint32_t bar_xfull = gbase + GS * G_BYTES;
    const uint32_t bar_xempty = bar_xfull + 8 * XS;
    const uint32_t bar_gfull = bar_xempty + 8 * XS;
    const uint32_t bar_gempty = bar_gfull + 8 * GS;
    const uint32_t bar_done = bar_gempty + 8 * GS;
    const uint32_t bar_drained = bar_done + 8;
    const uint32_t tmem_slot = bar_drained + 8;
    volatile int *abort = (volatile int *)(smem_raw + (tmem_slot + 4 - raw));
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;

    // the unit: channel groups cg (of In) and ng (of gz), pixel blocks [kb0, kb1)
    const int part = blockIdx.x % g.parts, unit = blockIdx.x / g.parts;
    const int ks = unit % g.ksplit, gr = unit / g.ksplit;
    const int c0 = (gr % g.cgroups) * 64, n0 = (gr / g.cgroups) * 64;
    const int kb0 = ks * g.per, kb1 = min(g.kblocks, kb0 + g.per);
    int s0, s1;
    wgrad_offsets(g, c0, n0, s0, s1);

    if (threadIdx.x == 0) {
        *abort = *(volatile int *)err;
        for (int s = 0; s < XS; ++s) {
            tc::mbar_init(bar_xfull + 8 * s, 1);
            tc::mbar_init(bar_xempty + 8 * s, 1);
        }
        for (int s = 0; s < GS; ++s) {
            tc::mbar_init(bar_gfull + 8 * s, 1);
            tc::mbar_init(bar_gempty + 8 * s, 1);
        }
        tc::mbar_init(bar_done, 1);
        tc::mbar_init(bar_drained, 4);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"((uint64_t)&mapX) : "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"((uint64_t)&mapG) : "memory");
    }
    __syncthreads();
    // the unit's tiles; this CTA's: part, part + parts, ..
    const int ns = s1 - s0 + 1, nt = wgrad_tiles(s0, s1), parts = (nt + g.tiles - 1) / g.tiles;
    if (*abort || kb0 >= kb1 || part >= parts) return;
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(tmem_slot),
                     "r"((uint32_t)TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    uint32_t tmem_base;
    asm volatile("ld.shared.u32 %0, [%1];\n" : "=r"(tmem_base) : "r"(tmem_slot));
    tmem_base = __shfl_sync(0xffffffffu, tmem_base, 0);

    // origin of pixel block kb
    auto block = [&](int kb, int &b, int &y0, int &x0) {
        const int xb = kb % g.xblocks, r = kb / g.xblocks;
        b = r / g.yblocks;
        y0 = (r - b * g.yblocks) * R;
        x0 = xb * BKX;
    };

    if (warp == 0) {
        if (lane == 0) {
            // ---------------- TMA producer ----------------
            int xs = 0, gs = 0;
            uint32_t xph = 0, gph = 0;
            bool ok = true;
            for (int kb = kb0; kb < kb1 && ok; ++kb) {
                int b, y0, x0;
                block(kb, b, y0, x0);
                if (!tc::mbar_wait(bar_gempty + 8 * gs, gph ^ 1u, abort)) {
                    ok = false;
                    break;
                }
                arrive_expect_tx(bar_gfull + 8 * gs, G_BYTES);
                tma_load_4d(gbase + gs * G_BYTES, &mapG, n0, x0, y0, b, bar_gfull + 8 * gs);
                if (++gs == GS) {
                    gs = 0;
                    gph ^= 1u;
                }
                if (!tc::mbar_wait(bar_xempty + 8 * xs, xph ^ 1u, abort)) {
                    ok = false;
                    break;
                }
                arrive_expect_tx(bar_xfull + 8 * xs, X_BYTES);
                tma_load_4d(base + xs * X_SLOT, &mapX, c0, x0 - 1, y0 - 1, b, bar_xfull + 8 * xs);
                if (++xs == XS) {
                    xs = 0;
                    xph ^= 1u;
                }
            }
            if (!ok) {
                // loads already issued finish on their own within microseconds
                const long long t0 = clock64();
                while (clock64() - t0 < 200000LL) {
                }
            }
        }
    } else if (warp == 1) {
        {  // the whole warp
            // ---------------- MMA issuer ----------------
            constexpr uint32_t IDESC = idesc_bf16_mn<64>();
            const uint64_t x_desc0 = sdesc_mn(base, ROW), x_desc1 = sdesc_mn(base, 128u);
            const uint64_t g_desc0 = sdesc_mn(gbase, GROW);
            int xs = 0, gs = 0;
            uint32_t xph = 0, gph = 0;
            bool ok = true;
            uint32_t last_bar = 0, last_par = 0, dph = 0;
            int in = 0;  // blocks of the sum so far
            for (int kb = kb0; kb < kb1 && ok; ++kb) {
                if (in == g.len) {  // the accumulators have been read
                    if (!mbar_wait_warp(bar_drained, dph, abort)) {
                        ok = false;
                        break;
                    }
                    dph ^= 1u;
                    in = 0;
                }
                int b, y0, x0;
                block(kb, b, y0, x0);
                const int rows = min(R, g.H - y0);
                if (!mbar_wait_warp(bar_gfull + 8 * gs, gph, abort)) {
                    ok = false;
                    break;
                }
                if (!mbar_wait_warp(bar_xfull + 8 * xs, xph, abort)) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                // 16 pixels = 2048 bytes; descriptors = the first ones plus constants (in 16-byte
                // units); image row j of gz against row j (dy = -1) of the box and the next two
                const uint64_t dx = (uint64_t)((uint32_t)xs * (X_SLOT / 16) + (uint32_t)(s0 + 1) * 8u);
                const uint64_t dg = g_desc0 + (uint64_t)((uint32_t)gs * (G_BYTES / 16));
                const uint64_t d0 = x_desc0 + dx, d1 = x_desc1 + dx + 2 * ROW / 16;
#pragma unroll
                for (int j = 0; j < R; ++j) {
                    if (j >= rows) break;
#pragma unroll
                    for (int kk = 0; kk < BKX / 16; ++kk) {
                        const uint64_t off = (j * ROW + kk * 2048u) / 16, goff = (j * GROW + kk * 2048u) / 16;
                        const uint32_t add = j + kk > 0 || in > 0 ? 1u : 0u;
                        for (int t = part; t < nt; t += parts)
                            mma_f16_elect(tmem_base + (uint32_t)(t * 64),
                                          (t < ns ? d0 + (uint64_t)(t * 8) : d1 + (uint64_t)((t - ns) * 16)) + off, dg + goff,
                                          IDESC, add);
                    }
                }
                mma_commit_elect(bar_xempty + 8 * xs);
                last_bar = bar_xempty + 8 * xs;
                last_par = xph;
                if (++xs == XS) {
                    xs = 0;
                    xph ^= 1u;
                }
                mma_commit_elect(bar_gempty + 8 * gs);
                if (++gs == GS) {
                    gs = 0;
                    gph ^= 1u;
                }
                if (++in == g.len || kb + 1 == kb1) mma_commit_elect(bar_done);
            }
            if (!ok && last_bar)
                tc::mbar_wait(last_bar, last_par, nullptr);  // tensor core idle before release
        }
    } else {
        // ---------------- epilogue (warps 2..5): atomic adds into dW, sum after sum ----------------
        const int q = warp & 3;
        uint32_t ph = 0;
        for (int kb = kb0; kb < kb1; kb += g.len, ph ^= 1u) {
            if (!mbar_wait_warp(bar_done, ph, abort)) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const int i = (q & 1) * 32 + lane;   // channel of In in the group
            const int e = c0 + i;
            const int px = g.F > 1 ? e / g.C : 0, ci = e - px * g.C;
            for (int t = part; t < nt; t += parts) {
                // tiles (dy -1 | 0) of each s, then (s | s + 1) of dy 1
                const int s = t < ns ? s0 + t : s0 + 2 * (t - ns) + (q >> 1);
                const int dy = t < ns ? (q >> 1) - 1 : 1;
                if (s > s1) continue;  // no tap (warp-uniform)
                const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(t * 64);
#pragma unroll 1
                for (int j0 = 0; j0 < 64; j0 += 16) {
                    uint32_t v[16];
                    tc::tmem_ld16(taddr + (uint32_t)j0, v);
                    const int f = n0 + j0;  // 16 channels of one pixel: Cout is a multiple of 32
                    const int pg = g.F > 1 ? f / g.Cout : 0, co = f - pg * g.Cout;
                    const int dx = g.F * s + px - pg;
                    if (dx >= -1 && dx <= 1) {
                        float *p = dw + ((long long)co * 9 + (dy + 1) * 3 + (dx + 1)) * g.C + ci;
#pragma unroll
                        for (int c = 0; c < 16; ++c) atomicAdd(p + (long long)c * 9 * g.C, __uint_as_float(v[c]));
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
            __syncwarp();
            if (lane == 0) arrive(bar_drained);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && *abort) atomicExch(err, 1);
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base),
                     "r"((uint32_t)TMEM_COLS));
    }
}

}  // namespace tma
}  // namespace nn
}  // namespace se2n
