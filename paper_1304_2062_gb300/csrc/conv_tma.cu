// Host side of the TMA tensor-core convolutions (conv_tma.cuh): tensor-map
// encoding, shape checks, the epilogue functors and the launches for the
// forward convolution (optionally with the network's 1x1 head and input
// skip fused into the last layer) and the data gradient.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <mutex>

#include "conv_tma.cuh"
#include "nn.h"

using namespace se2n::nn;

// Set by a TMA convolution whose bounded wait ran out (never expected).
__device__ int g_tma_fault;

namespace {

__device__ __forceinline__ uint32_t pack2(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *(const uint32_t *)&h;
}

__device__ __forceinline__ void pack16(const float (&w)[16], uint32_t (&p)[8]) {
#pragma unroll
    for (int q = 0; q < 8; ++q) p[q] = pack2(w[2 * q], w[2 * q + 1]);
}
// relu?(v + bias) as bf16; nb bias values (the output channels).
// pool: also the 2x2 averages of the bf16 outputs (a + b + c + d of the rows in turn, FP32); a
// warp has to hold 8 x 4 pixels then (k_conv_halo, k_conv_group). It saves the
// kernel that read the output again: 120 us for the three poolings at 64 images of
// 256 x 256, for about 40 of a longer epilogue. The upsampling in the same way (four
// stores for one) took as long here as in its own kernel, which is bound by
// writing.
struct FwdEpi {
    const float *bias;
    int relu, nb;
    __nv_bfloat16 *pool;
    int W;
    static constexpr int SMEM_FLOATS = 256;
    __device__ __forceinline__ void prepare(float *sm, int i, int n) const {
        for (int k = i; k < nb; k += n) sm[k] = bias[k];
    }
    struct Pre {};
    struct PrePix {};
    __device__ __forceinline__ Pre prefetch(int, int) const { return {}; }
    __device__ __forceinline__ PrePix prefetch_pixel(int) const { return {}; }
    __device__ __forceinline__ bool writes() const { return true; }
    __device__ __forceinline__ bool second(int) const { return false; }
    __device__ __forceinline__ int column(int n) const { return n; }
    __device__ __forceinline__ void pack(int n, const float (&v)[16], const float *sm, uint32_t (&p)[8]) const {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            float a = v[2 * q] + sm[n + 2 * q], b = v[2 * q + 1] + sm[n + 2 * q + 1];
            if (relu) {
                a = fmaxf(a, 0.0f);
                b = fmaxf(b, 0.0f);
            }
            p[q] = pack2(a, b);
        }
    }
    // average of two channels of four pixels
    static __device__ __forceinline__ uint32_t mean(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
        const float s0 = __uint_as_float(a << 16) + __uint_as_float(b << 16) + __uint_as_float(c << 16) +
                         __uint_as_float(d << 16);
        const float s1 = __uint_as_float(a & 0xffff0000u) + __uint_as_float(b & 0xffff0000u) +
                         __uint_as_float(c & 0xffff0000u) + __uint_as_float(d & 0xffff0000u);
        return pack2(0.25f * s0, 0.25f * s1);
    }
    __device__ __forceinline__ __nv_bfloat16 *pool_at(int m) const {
        const int row = m / W;
        return pool + ((long long)(row >> 1) * (W >> 1) + ((m - row * W) >> 1)) * nb;
    }
    __device__ __forceinline__ void compute(int m, int n, const float (&v)[16], float &, const float *sm, Pre,
                                            bool valid, uint32_t (&p)[8]) const {
        pack(n, v, sm, p);
        if (!pool) return;
        // the 2 x 2 pixels are lanes l, l ^ 1, l ^ 8, l ^ 9: each gets four of the 16
        // channels of all of them, in two exchanges
        const int lane = threadIdx.x & 31;
        const bool odd = lane & 1, hi = lane & 8;
        uint32_t pa[4], pb[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t mine = odd ? p[4 + k] : p[k];
            const uint32_t oth = __shfl_xor_sync(0xffffffffu, odd ? p[k] : p[4 + k], 1);
            pa[k] = odd ? oth : mine;
            pb[k] = odd ? mine : oth;
        }
        uint32_t o[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const uint32_t ma = hi ? pa[2 + k] : pa[k], mb = hi ? pb[2 + k] : pb[k];
            const uint32_t oa = __shfl_xor_sync(0xffffffffu, hi ? pa[k] : pa[2 + k], 8);
            const uint32_t ob = __shfl_xor_sync(0xffffffffu, hi ? pb[k] : pb[2 + k], 8);
            o[k] = mean(hi ? oa : ma, hi ? ob : mb, hi ? ma : oa, hi ? mb : ob);
        }
        if (valid) *(uint2 *)(pool_at(m) + n + (odd ? 8 : 0) + (hi ? 4 : 0)) = make_uint2(o[0], o[1]);
    }
    __device__ __forceinline__ void compute_pair(int m, int n, const float (&v)[2][16], float (&)[2], const float *sm,
                                                 Pre, Pre, bool valid, uint32_t (&pr)[2][8]) const {
        uint32_t(&p)[8] = pr[0], (&r)[8] = pr[1];
        pack(n, v[0], sm, p);
        pack(n, v[1], sm, r);
        if (!pool) return;
        // the other two pixels are lane l ^ 8's: each lane gets half of the channels
        const bool hi = threadIdx.x & 8;
        uint32_t o[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t ma = hi ? p[4 + k] : p[k], mb = hi ? r[4 + k] : r[k];
            const uint32_t oa = __shfl_xor_sync(0xffffffffu, hi ? p[k] : p[4 + k], 8);
            const uint32_t ob = __shfl_xor_sync(0xffffffffu, hi ? r[k] : r[4 + k], 8);
            o[k] = mean(hi ? oa : ma, hi ? ob : mb, hi ? ma : oa, hi ? mb : ob);
        }
        if (valid) *(uint4 *)(pool_at(m) + n + (hi ? 8 : 0)) = make_uint4(o[0], o[1], o[2], o[3]);
    }
    __device__ __forceinline__ void finish(int, float, const float *, PrePix) const {}
};

// The last convolution (32 channels, ReLU) with the 1x1 head and the input
// skip: d[m][:] = bf16(relu(v + bias)) as FwdEpi (stored for the
// backward pass only: inference needs y alone), and
// y[m] = f[m] (mask[m] != 0) + hb + sum_c hw[c] d[m][c] (FP32, c in order).
struct HeadEpi {
    const float *bias;
    const float *hw, *hb, *f;
    const uint8_t *mask;
    float *y;
    bool keep;  // d is wanted
    static constexpr int SMEM_FLOATS = 65;  // bias[32], hw[32], hb
    __device__ __forceinline__ void prepare(float *sm, int i, int n) const {
        for (int k = i; k < 65; k += n) sm[k] = k < 32 ? bias[k] : k < 64 ? hw[k - 32] : hb[0];
    }
    struct Pre {};
    struct PrePix {
        float f;
        uint8_t mask;
    };
    __device__ __forceinline__ Pre prefetch(int, int) const { return {}; }
    __device__ __forceinline__ PrePix prefetch_pixel(int m) const { return {f[m], mask[m]}; }
    __device__ __forceinline__ bool writes() const { return keep; }
    __device__ __forceinline__ bool second(int) const { return false; }
    __device__ __forceinline__ int column(int n) const { return n; }
    __device__ __forceinline__ void compute(int, int n, const float (&v)[16], float &st, const float *sm, Pre, bool,
                                            uint32_t (&p)[8]) const {
        float w[16];
        if (n == 0) st = sm[64];
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            w[q] = fmaxf(v[q] + sm[n + q], 0.0f);
            w[q] = __bfloat162float(__float2bfloat16_rn(w[q]));
            st = fmaf(sm[32 + n + q], w[q], st);
        }
        pack16(w, p);
    }
    __device__ __forceinline__ void compute_pair(int m, int n, const float (&v)[2][16], float (&st)[2],
                                                 const float *sm, const Pre &a, const Pre &a1, bool valid,
                                                 uint32_t (&p)[2][8]) const {
        compute(m, n, v[0], st[0], sm, a, valid, p[0]);
        compute(m + 1, n, v[1], st[1], sm, a1, valid, p[1]);
    }
    __device__ __forceinline__ void finish(int m, float st, const float *, PrePix p) const {
        y[m] = (p.mask ? p.f : 0.0f) + st;
    }
};

// Data gradient: columns < split go to the first tensor (times (act > 0) when act
// is given), the others to the second.
struct DgradEpi {
    const __nv_bfloat16 *act;
    int split;
    static constexpr int SMEM_FLOATS = 1;
    __device__ __forceinline__ void prepare(float *, int, int) const {}
    struct Pre {
        uint4 a0, a1;  // the 16 activations (bf16)
    };
    struct PrePix {};
    __device__ __forceinline__ Pre prefetch(int m, int n) const {
        Pre p{};
        if (act && n < split) {
            const uint4 *a4 = (const uint4 *)(act + (long long)m * split + n);
            p.a0 = a4[0];
            p.a1 = a4[1];
        }
        return p;
    }
    __device__ __forceinline__ PrePix prefetch_pixel(int) const { return {}; }
    __device__ __forceinline__ bool writes() const { return true; }
    __device__ __forceinline__ bool second(int n) const { return n >= split; }
    __device__ __forceinline__ int column(int n) const { return n < split ? n : n - split; }
    __device__ __forceinline__ void compute(int, int n, const float (&v)[16], float &, const float *, const Pre &a, bool,
                                            uint32_t (&p)[8]) const {
        float w[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) w[q] = v[q];
        if (act && n < split) {
            const uint32_t aw[8] = {a.a0.x, a.a0.y, a.a0.z, a.a0.w, a.a1.x, a.a1.y, a.a1.z, a.a1.w};
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const __nv_bfloat162 h = *(const __nv_bfloat162 *)&aw[q];
                if (!(__bfloat162float(h.x) > 0.0f)) w[2 * q] = 0.0f;
                if (!(__bfloat162float(h.y) > 0.0f)) w[2 * q + 1] = 0.0f;
            }
        }
        pack16(w, p);
    }
    __device__ __forceinline__ void compute_pair(int m, int n, const float (&v)[2][16], float (&st)[2],
                                                 const float *sm, const Pre &a, const Pre &a1, bool valid,
                                                 uint32_t (&p)[2][8]) const {
        compute(m, n, v[0], st[0], sm, a, valid, p[0]);
        compute(m + 1, n, v[1], st[1], sm, a1, valid, p[1]);
    }
    __device__ __forceinline__ void finish(int, float, const float *, PrePix) const {}
};

PFN_cuTensorMapEncodeTiled_v12000 encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        return (PFN_cuTensorMapEncodeTiled_v12000)p;
    }();
    return fn;
}

int sm_count() {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    return n;
}

int *fault_ptr() {
    void *p = nullptr;
    if (cudaGetSymbolAddress(&p, g_tma_fault) != cudaSuccess) return nullptr;
    return (int *)p;
}

// The tensors a kernel's output boxes go to (second: the columns from the first's
// last on; no tensor: p null), and their maps: 8 or 16 pixels of 4 image rows, ob channels.
struct OutTensor {
    __nv_bfloat16 *p;
    int channels, ld;
};
struct OutTensors {
    OutTensor t[2];
};
bool out_maps(PFN_cuTensorMapEncodeTiled_v12000 enc, const OutTensors &o, int B, int H, int W, int ob, int px,
              CUtensorMap (&m)[2]) {
    for (int k = 0; k < 2; ++k) {
        const OutTensor &t = o.t[k].p ? o.t[k] : o.t[0];
        if (!t.p) continue;  // no output is wanted: the maps are not used
        if (t.channels % ob) return false;
        const cuuint64_t dims[4] = {(cuuint64_t)t.channels, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)B};
        const cuuint64_t ld = (cuuint64_t)t.ld * 2;
        const cuuint64_t strides[3] = {ld, ld * W, ld * W * H};
        const cuuint32_t box[4] = {(cuuint32_t)ob, (cuuint32_t)px, 4, 1};
        const cuuint32_t es[4] = {1, 1, 1, 1};
        if (enc(&m[k], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, (void *)t.p, dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, ob == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return false;
    }
    return true;
}

// Images whose narrow layers are summed blocks first (conv_tma.cuh, SumOrder).
bool whole_tiles(int H, int W) { return W % 16 == 0 && H % 8 == 0; }

// Narrow layers: 8 x 16 tiles, halo boxes, weights resident in shared memory.
template <int BN, int CK, class EPI>
cudaError_t launch_halo(const __nv_bfloat16 *A, int B, int H, int W, int C, const __nv_bfloat16 *wmat, int N, int flip,
                        const EPI &epi, const OutTensors &o, cudaStream_t s) {
    using Cf = tma::HaloCfg<BN, CK>;
    if (C % CK || N % BN) return cudaErrorNotSupported;
    const int nblk = 9 * (C / CK);
    const int wbytes = nblk * Cf::BBLK;
    int S = (Cf::SMEM_BUDGET - wbytes) / Cf::STAGE;
    if (S > 8) S = 8;
    if (S < 2) return cudaErrorNotSupported;
    auto enc = encoder();
    const int nsm = sm_count();
    int *err = fault_ptr();
    if (!enc || nsm <= 0 || !err) return cudaErrorNotSupported;
    CUtensorMap ma, mb, mo[2] = {};
    if (!out_maps(enc, o, B, H, W, Cf::OB, tma::HBW, mo)) return cudaErrorNotSupported;
    {
        const cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)B};
        const cuuint64_t strides[3] = {(cuuint64_t)C * 2, (cuuint64_t)W * C * 2, (cuuint64_t)H * W * C * 2};
        const cuuint32_t box[4] = {(cuuint32_t)CK, (cuuint32_t)tma::HPITCH, (cuuint32_t)(tma::HBH + 2), 1};
        const cuuint32_t es[4] = {1, 1, 1, 1};
        if (enc(&ma, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, (void *)A, dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CK == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    {
        const cuuint64_t dims[2] = {(cuuint64_t)9 * C, (cuuint64_t)N};
        const cuuint64_t strides[1] = {(cuuint64_t)9 * C * 2};
        const cuuint32_t box[2] = {(cuuint32_t)CK, (cuuint32_t)BN};
        const cuuint32_t es[2] = {1, 1};
        if (enc(&mb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void *)wmat, dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CK == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    tma::ConvGeo g;
    g.B = B;
    g.H = H;
    g.W = W;
    g.C = C;
    g.bw = tma::HBW;
    g.bh = tma::HBH;
    g.tiles_x = (W + tma::HBW - 1) / tma::HBW;
    g.tiles_y = (H + tma::HBH - 1) / tma::HBH;
    g.mtiles = B * g.tiles_x * g.tiles_y;
    g.ntiles = N / BN;
    g.tiles = g.mtiles * g.ntiles;
    g.nchunk = C / CK;
    g.flip = flip;
    g.order = whole_tiles(H, W) ? tma::ORDER_BLOCKS : tma::ORDER_TAPS;
    if (g.order == tma::ORDER_TAPS && S < g.nchunk) return cudaErrorNotSupported;
    const int smem = 1024 + wbytes + S * Cf::STAGE + 8 * tma::kOutBytes + 256;
    auto *fn = &tma::k_conv_halo<BN, CK, EPI>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    // each CTA keeps one n tile's weights: a whole number of CTAs per n tile
    const int per = nsm / g.ntiles;
    if (per < 1) return cudaErrorNotSupported;
    const int grid = (g.mtiles < per ? g.mtiles : per) * g.ntiles;
    fn<<<grid, tma::kHaloThreads, smem, s>>>(ma, mb, mo[0], mo[1], g, epi, S, err);
    return cudaGetLastError();
}

// 32 output channels: pairs of pixels (W even), halo boxes, weights resident in shared memory.
template <class EPI>
cudaError_t launch_pair(const __nv_bfloat16 *A, int B, int H, int W, int C, const __nv_bfloat16 *wmat, int flip,
                        const EPI &epi, const OutTensors &o, cudaStream_t s) {
    using Cf = tma::PairCfg;
    if (W % 2 || C % 32) return cudaErrorNotSupported;
    const int nblk = 9 * (C / 32);
    const int wbytes = nblk * Cf::BBLK;
    int S = (Cf::SMEM_BUDGET - wbytes) / Cf::STAGE;
    if (S > 8) S = 8;
    if (S < 2) return cudaErrorNotSupported;
    auto enc = encoder();
    const int nsm = sm_count();
    int *err = fault_ptr();
    if (!enc || nsm <= 0 || !err) return cudaErrorNotSupported;
    tma::ConvGeo g;
    g.B = B;
    g.H = H;
    g.W = W / 2;  // columns of two pixels
    g.C = C;
    g.bw = tma::HBW;
    g.bh = tma::HBH;
    g.tiles_x = (g.W + tma::HBW - 1) / tma::HBW;
    g.tiles_y = (H + tma::HBH - 1) / tma::HBH;
    g.mtiles = B * g.tiles_x * g.tiles_y;
    g.ntiles = 1;
    g.tiles = g.mtiles;
    g.nchunk = C / 32;
    g.flip = flip;
    g.order = !whole_tiles(H, W) ? tma::ORDER_TAPS : C % 64 ? tma::ORDER_BLOCKS : tma::ORDER_OFFSETS;
    if (g.order == tma::ORDER_OFFSETS && C > 64) return cudaErrorNotSupported;  // blocks of 64 in between
    if (g.order != tma::ORDER_BLOCKS && S < g.nchunk) return cudaErrorNotSupported;
    CUtensorMap ma, mb, mo[2] = {};
    if (!out_maps(enc, o, B, H, W, 32, 2 * tma::HBW, mo)) return cudaErrorNotSupported;
    {
        const cuuint64_t dims[4] = {(cuuint64_t)2 * C, (cuuint64_t)g.W, (cuuint64_t)H, (cuuint64_t)B};
        const cuuint64_t strides[3] = {(cuuint64_t)C * 4, (cuuint64_t)W * C * 2, (cuuint64_t)H * W * C * 2};
        const cuuint32_t box[4] = {32, (cuuint32_t)tma::HPITCH, (cuuint32_t)(tma::HBH + 2), 1};
        const cuuint32_t es[4] = {1, 1, 1, 1};
        if (enc(&ma, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, (void *)A, dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    {
        const cuuint64_t dims[2] = {(cuuint64_t)9 * C, 32};
        const cuuint64_t strides[1] = {(cuuint64_t)9 * C * 2};
        const cuuint32_t box[2] = {32, 32};
        const cuuint32_t es[2] = {1, 1};
        if (enc(&mb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void *)wmat, dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    const int smem = 1024 + wbytes + S * Cf::STAGE + 8 * tma::kOutBytes + 256;
    auto *fn = &tma::k_conv_pair<EPI>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    fn<<<g.mtiles < nsm ? g.mtiles : nsm, tma::kHaloThreads, smem, s>>>(ma, mb, mo[0], mo[1], g, epi, S, err);
    return cudaGetLastError();
}

// Wide layers: halo boxes, groups of tiles that share the weights. N in tiles of
// 128 channels, or of 64.
template <int BN, class EPI>
cudaError_t launch_group(const __nv_bfloat16 *A, int B, int H, int W, int C, const __nv_bfloat16 *wmat, int N, int flip,
                         const EPI &epi, const OutTensors &o, cudaStream_t s) {
    using Cf = tma::GroupCfg<BN>;
    if (C % 64 || N % BN) return cudaErrorNotSupported;
    auto enc = encoder();
    const int nsm = sm_count();
    int *err = fault_ptr();
    if (!enc || nsm <= 0 || !err) return cudaErrorNotSupported;
    CUtensorMap ma, mb, mo[2] = {};
    if (!out_maps(enc, o, B, H, W, Cf::OB, tma::HBW, mo)) return cudaErrorNotSupported;
    {
        const cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)B};
        const cuuint64_t strides[3] = {(cuuint64_t)C * 2, (cuuint64_t)W * C * 2, (cuuint64_t)H * W * C * 2};
        const cuuint32_t box[4] = {64, (cuuint32_t)tma::HPITCH, (cuuint32_t)(tma::HBH + 2), 1};
        const cuuint32_t es[4] = {1, 1, 1, 1};
        if (enc(&ma, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, (void *)A, dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    {
        const cuuint64_t dims[2] = {(cuuint64_t)9 * C, (cuuint64_t)N};
        const cuuint64_t strides[1] = {(cuuint64_t)9 * C * 2};
        const cuuint32_t box[2] = {64, (cuuint32_t)BN};
        const cuuint32_t es[2] = {1, 1};
        if (enc(&mb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void *)wmat, dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    tma::ConvGeo g;
    g.B = B;
    g.H = H;
    g.W = W;
    g.C = C;
    g.bw = tma::HBW;
    g.bh = tma::HBH;
    g.tiles_x = (W + tma::HBW - 1) / tma::HBW;
    g.tiles_y = (H + tma::HBH - 1) / tma::HBH;
    g.mtiles = B * g.tiles_x * g.tiles_y;
    g.ntiles = N / BN;
    g.tiles = g.mtiles * g.ntiles;
    g.nchunk = C / 64;
    g.flip = flip;
    g.order = tma::ORDER_TAPS;
    if (g.nchunk > Cf::AMAX) return cudaErrorNotSupported;  // a tile's boxes stay for all taps
    // as many tiles a group as leave every SM one
    int G = g.tiles / nsm;
    if (G > Cf::GMAX) G = Cf::GMAX;
    if (G > Cf::AMAX / g.nchunk) G = Cf::AMAX / g.nchunk;
    if (G < 1) G = 1;
    // boxes of a group and up to three (one of four or more) of the next, the rest for weights
    const int boxes = G * g.nchunk, more = g.nchunk >= 4 ? 1 : boxes < 3 ? boxes : 3;
    const int AS = boxes + more < Cf::AMAX ? boxes + more : Cf::AMAX;
    int WS = (Cf::SMEM_BUDGET - AS * Cf::A_SLOT) / Cf::W_BYTES;
    if (WS > Cf::WMAX) WS = Cf::WMAX;
    const int smem = Cf::SMEM_REST + AS * Cf::A_SLOT + WS * Cf::W_BYTES;
    const int groups = (g.mtiles + G - 1) / G * g.ntiles;
    auto *fn = &tma::k_conv_group<BN, EPI>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    fn<<<groups < nsm ? groups : nsm, tma::kHaloThreads, smem, s>>>(ma, mb, mo[0], mo[1], g, epi, G, AS, WS, err);
    return cudaGetLastError();
}

template <class EPI>
cudaError_t launch_wide(const __nv_bfloat16 *A, int B, int H, int W, int C, const __nv_bfloat16 *wmat, int N, int flip,
                        const EPI &epi, const OutTensors &o, cudaStream_t s) {
    return N % 128 == 0 ? launch_group<128>(A, B, H, W, C, wmat, N, flip, epi, o, s)
                        : launch_group<64>(A, B, H, W, C, wmat, N, flip, epi, o, s);
}

// Weight gradient (k_wgrad_tma): x [B][H][W][C] and gz [B][H][W][Cout] NHWC, dw
// [Cout][9 C] FP32 (accumulated).
cudaError_t launch_wgrad(const __nv_bfloat16 *x, int B, int H, int W, int C, const __nv_bfloat16 *gz, int Cout,
                         float *dw, cudaStream_t s) {
    const int nsm = sm_count();
    tma::WgradGeo g;
    if (nsm <= 0 || !tma::wgrad_split(g, B, H, W, C, Cout, nsm)) return cudaErrorNotSupported;
    auto enc = encoder();
    int *err = fault_ptr();
    if (!enc || !err) return cudaErrorNotSupported;
    const int bkx = g.bkx, cv = g.F * C, nv = g.F * Cout;
    auto map = [&](CUtensorMap *m, const __nv_bfloat16 *p, int ch, int cols, int rows) {
        const cuuint64_t dims[4] = {(cuuint64_t)ch, (cuuint64_t)g.W, (cuuint64_t)H, (cuuint64_t)B};
        const cuuint64_t strides[3] = {(cuuint64_t)ch * 2, (cuuint64_t)g.W * ch * 2, (cuuint64_t)H * g.W * ch * 2};
        const cuuint32_t box[4] = {64, (cuuint32_t)cols, (cuuint32_t)rows, 1};
        const cuuint32_t es[4] = {1, 1, 1, 1};
        return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, (void *)p, dims, strides, box, es,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    CUtensorMap mx, mg;
    if (!map(&mx, x, cv, bkx + 2, tma::kWgR + 2) || !map(&mg, gz, nv, bkx, tma::kWgR)) return cudaErrorInvalidValue;
    int smem = 1024 + tma::kWgXSlots * (bkx == 32 ? tma::kWgXSlot<32> : tma::kWgXSlot<16>) +
                     tma::kWgGSlots * tma::kWgR * bkx * 128 + 256;
    if (smem < 120 * 1024) smem = 120 * 1024;  // one CTA an SM: each takes all of tensor memory
    auto *fn = bkx == 32 ? &tma::k_wgrad_tma<32> : &tma::k_wgrad_tma<16>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    fn<<<g.cgroups * g.ngroups * g.ksplit * g.parts, 192, smem, s>>>(mx, mg, g, dw, err);
    return cudaGetLastError();
}

}  // namespace

namespace se2n {
namespace nn {

cudaError_t conv_wgrad(const __nv_bfloat16 *x, int B, int H, int W, int C, const __nv_bfloat16 *gz, int Cout, float *dw,
                       cudaStream_t s) {
    return launch_wgrad(x, B, H, W, C, gz, Cout, dw, s);
}

cudaError_t tc_fault(int *host_flag, bool reset) {
    cudaError_t e = cudaMemcpyFromSymbol(host_flag, g_tma_fault, sizeof(int));
    if (e == cudaSuccess && reset && *host_flag) {
        const int zero = 0;
        e = cudaMemcpyToSymbol(g_tma_fault, &zero, sizeof(int));
    }
    return e;
}

cudaError_t conv_forward(const __nv_bfloat16 *in, int B, int H, int W, int Cin, const __nv_bfloat16 *w,
                         const float *bias, int Cout, int relu, __nv_bfloat16 *out, int ldo, __nv_bfloat16 *pool,
                         cudaStream_t s) {
    const OutTensors o{{{out, Cout, ldo}, {nullptr, 0, 0}}};
    const FwdEpi epi{bias, relu, Cout, pool, W};
    if (Cout == 32) return launch_pair(in, B, H, W, Cin, w, 0, epi, o, s);
    if (Cout == 64) {
        const cudaError_t e = Cin % 64 == 0 ? launch_halo<64, 64>(in, B, H, W, Cin, w, Cout, 0, epi, o, s)
                                            : launch_halo<64, 32>(in, B, H, W, Cin, w, Cout, 0, epi, o, s);
        if (e != cudaErrorNotSupported) return e;  // more weights than shared memory holds
    }
    return launch_wide(in, B, H, W, Cin, w, Cout, 0, epi, o, s);
}

cudaError_t conv_forward_head(const __nv_bfloat16 *in, int B, int H, int W, int Cin, const __nv_bfloat16 *w,
                              const float *bias, __nv_bfloat16 *out, const HeadArgs &head, cudaStream_t s) {
    const OutTensors o{{{out, 32, 32}, {nullptr, 0, 0}}};
    const HeadEpi epi{bias, head.hw, head.hb, head.f, head.mask, head.y, out != nullptr};
    return launch_pair(in, B, H, W, Cin, w, 0, epi, o, s);
}

cudaError_t conv_dgrad(const __nv_bfloat16 *gz, int B, int H, int W, int Cout, const __nv_bfloat16 *wt, int Cin,
                       const __nv_bfloat16 *act, __nv_bfloat16 *din, __nv_bfloat16 *din2, int split, cudaStream_t s) {
    if (split % 16) return cudaErrorNotSupported;
    const DgradEpi epi{act, split};
    const OutTensors o{{{din, split, split}, {split < Cin ? din2 : nullptr, Cin - split, Cin - split}}};
    // A = gz (Cout channels, taps mirrored), B = wt [Cin][9 Cout]
    if (Cin == 32) return launch_pair(gz, B, H, W, Cout, wt, 1, epi, o, s);
    if (Cin == 96) return launch_halo<96, 32>(gz, B, H, W, Cout, wt, Cin, 1, epi, o, s);
    if (Cin == 64) {
        const cudaError_t e = Cout % 64 == 0 ? launch_halo<64, 64>(gz, B, H, W, Cout, wt, Cin, 1, epi, o, s)
                                             : launch_halo<64, 32>(gz, B, H, W, Cout, wt, Cin, 1, epi, o, s);
        if (e != cudaErrorNotSupported) return e;
    }
    return launch_wide(gz, B, H, W, Cout, wt, Cin, 1, epi, o, s);
}

}  // namespace nn
}  // namespace se2n
