// Kernels of the learned surrogate: a 4-level U-Net (32-64-128-256
// channels), BF16 weights and activations, FP32 accumulation, trained on
// (corrupted image, method output) pairs that the inpainting method itself
// generates.
//
// Activations are NHWC bf16 with the channel count a multiple of 8; a 3x3
// convolution (padding 1) is an implicit GEMM (conv_tma.cuh) with
// k = tap * C + channel, tap = (dy+1)*3 + (dx+1). Layer list and parameter
// layout are in unet.cu. Here: the first layer and everything that is not a
// convolution.
#include <cuda_bf16.h>

#include "diffuse_x2.cuh"
#include "nn.h"

using namespace se2n::nn;

namespace {

// Weights rearranged for the data gradient, K-major in the output channel:
// wt[ci][tap * Cout + co] = w[co][tap * Cin + ci], layer blockIdx.y at the same offset in
// both. One launch for all layers: a launch of a few microseconds each took 51 us of a
// backward pass.
__global__ void k_transpose_dgrad(const __nv_bfloat16 *w0, __nv_bfloat16 *wt0, const __grid_constant__ ConvLayers d) {
    const int Cout = d.cout[blockIdx.y], Cin = d.cin[blockIdx.y];
    const __nv_bfloat16 *w = w0 + d.off[blockIdx.y];
    __nv_bfloat16 *wt = wt0 + d.off[blockIdx.y];
    const int total = Cout * 9 * Cin;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        const int co = i % Cout, t = i / Cout, tap = t % 9, ci = t / 9;
        wt[i] = w[(co * 9 + tap) * Cin + ci];
    }
}

// Column sums of a [P][C] bf16 matrix into db[C] (bias gradients): each
// thread sums 8 channels (one 16-byte load) of every (256 / (C/8))-th row,
// the block combines its partial sums in shared memory, one atomic per
// channel per block.
__global__ void __launch_bounds__(256) k_colsum(const __nv_bfloat16 *g, long long P, int C, float *db) {
    __shared__ float part[256][8];
    const int groups = C / 8;                 // 4..32
    const int rows = blockDim.x / groups;     // rows per block step
    const int cg = threadIdx.x % groups, rr = threadIdx.x / groups;
    float s[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (rr < rows) {
        for (long long p = (long long)blockIdx.x * rows + rr; p < P; p += (long long)gridDim.x * rows) {
            const uint4 v = *(const uint4 *)(g + p * C + cg * 8);
            const __nv_bfloat16 *h = (const __nv_bfloat16 *)&v;
#pragma unroll
            for (int k = 0; k < 8; ++k) s[k] += __bfloat162float(h[k]);
        }
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) part[threadIdx.x][k] = s[k];
    __syncthreads();
    if (threadIdx.x < C) {
        const int c8 = threadIdx.x / 8, k = threadIdx.x % 8;
        float t = 0.0f;
        for (int r = 0; r < rows; ++r) t += part[r * groups + c8][k];
        atomicAdd(db + threadIdx.x, t);
    }
}

// Input packing: x[b][y][x][0] = f*(mask!=0), [1] = mask, [2..7] = 0.
__global__ void k_pack_input(const float *f, const uint8_t *mask, __nv_bfloat16 *x, long long P) {
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < P; p += (long long)gridDim.x * blockDim.x) {
        const float m = mask[p] ? 1.0f : 0.0f;
        __nv_bfloat16 v[8];
        v[0] = __float2bfloat16_rn(f[p] * m);
        v[1] = __float2bfloat16_rn(m);
#pragma unroll
        for (int c = 2; c < 8; ++c) v[c] = __float2bfloat16_rn(0.0f);
        *(uint4 *)(x + p * 8) = *(uint4 *)v;
    }
}

// Nearest upsampling into the first C1 channels of a wider tensor: one
// block per output row (b, y), 16 bytes per thread.
__global__ void k_upsample_into(const __nv_bfloat16 *lo, int C1, __nv_bfloat16 *out, int ldo, int H, int W) {
    const int y = blockIdx.x % H;
    const long long b = blockIdx.x / H;
    const int C8 = C1 / 8, Wl = W / 2;
    const __nv_bfloat16 *src = lo + ((b * (H / 2) + y / 2) * Wl) * C1;
    __nv_bfloat16 *dst = out + ((b * H + y) * W) * (long long)ldo;
    for (int i = threadIdx.x; i < W * C8; i += blockDim.x) {
        const int x = i / C8, c = (i - x * C8) * 8;
        *(uint4 *)(dst + (long long)x * ldo + c) = *(const uint4 *)(src + (x / 2) * C1 + c);
    }
}

// First convolution straight from the image: the input channels are
// bf16(f m) and m (the other six are zero), so each of the 32 outputs is a
// sum over 9 taps x 2 channels, done in FP32 on the CUDA cores. A block
// takes 32 x 16 pixel tiles; the tile and its 1-pixel halo of (bf16(f m), m)
// are staged in shared memory with coalesced loads, and the weights sit
// there as [tap][channel][4 outputs] float4. A thread takes four pixels of a column and half
// of the outputs, so that a 16-byte load feeds eight packed FMAs (64 images of 256 x 256:
// 137 us; 202 with one pixel and scalar FMAs). Warp-level matrix products (75 us) add in
// another order: see SumOrder in conv_tma.cuh.
constexpr int C0_TW = 32, C0_TH = 16;
__global__ void __launch_bounds__(256, 2) k_conv0(const float *f, const uint8_t *mask, const __nv_bfloat16 *w,
                                               const float *bias, __nv_bfloat16 *out, int B, int H, int W) {
    __shared__ float4 sw[9][2][8];
    __shared__ float sb[32];
    __shared__ float2 tile[C0_TH + 2][C0_TW + 2];
    for (int i = threadIdx.x; i < 9 * 2 * 8; i += blockDim.x) {
        const int tap = i / 16, ci = (i / 8) % 2, q = i % 8;
        const __nv_bfloat16 *wq = w + tap * 8 + ci;  // w[co][tap][ci], 72 per output channel
        sw[tap][ci][q] = make_float4(__bfloat162float(wq[(4 * q + 0) * 72]), __bfloat162float(wq[(4 * q + 1) * 72]),
                                     __bfloat162float(wq[(4 * q + 2) * 72]), __bfloat162float(wq[(4 * q + 3) * 72]));
    }
    if (threadIdx.x < 32) sb[threadIdx.x] = bias[threadIdx.x];
    const int tx = threadIdx.x % C0_TW, half = threadIdx.x / C0_TW % 2, ty = threadIdx.x / (2 * C0_TW);
    const int ntx = (W + C0_TW - 1) / C0_TW, nty = (H + C0_TH - 1) / C0_TH;
    const long long ntiles = (long long)B * ntx * nty;
    // the pixels of tile t that this thread stages, loaded while the tile before is computed
    constexpr int TILE = (C0_TH + 2) * (C0_TW + 2), IT = (TILE + 255) / 256;
    float pf[IT];
    uint8_t pm[IT];
    auto fetch = [&](long long t) {
        const long long b = t / ntx / nty;
        const int x0 = (int)(t % ntx) * C0_TW, y0 = (int)(t / ntx % nty) * C0_TH;
#pragma unroll
        for (int k = 0; k < IT; ++k) {
            const int i = threadIdx.x + 256 * k, ly = i / (C0_TW + 2), lx = i % (C0_TW + 2);
            const int yy = y0 + ly - 1, xx = x0 + lx - 1;
            const bool in = i < TILE && t < ntiles && yy >= 0 && yy < H && xx >= 0 && xx < W;
            const long long q = (b * H + yy) * W + xx;
            pm[k] = in ? mask[q] : 0;
            pf[k] = in ? f[q] : 0.0f;
        }
    };
    fetch(blockIdx.x);
    for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const long long b = t / ntx / nty;
        const int x0 = (int)(t % ntx) * C0_TW, y0 = (int)(t / ntx % nty) * C0_TH;
        __syncthreads();  // the previous tile is consumed (and the tables are ready)
#pragma unroll
        for (int k = 0; k < IT; ++k) {
            const int i = threadIdx.x + 256 * k;
            const float m = pm[k] ? 1.0f : 0.0f;
            if (i < TILE)
                (&tile[0][0])[i] = make_float2(__bfloat162float(__float2bfloat16_rn(pf[k] * m)), m);
        }
        __syncthreads();
        fetch(t + gridDim.x);
        // pixels (x, y .. y + 3), outputs 16 half ..; outputs co, co + 1 packed
        const int x = x0 + tx, y = y0 + 4 * ty;
        float2 u[6][3];
#pragma unroll
        for (int r = 0; r < 6; ++r)
#pragma unroll
            for (int c = 0; c < 3; ++c) u[r][c] = tile[4 * ty + r][tx + c];
        se2n::f32x2 acc[4][8];
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int q = 0; q < 8; ++q) acc[p][q] = se2n::pk2(0.0f, 0.0f);
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) {
            se2n::f32x2 v[4][2];
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                v[p][0] = se2n::dup2(u[p + tap / 3][tap % 3].x);
                v[p][1] = se2n::dup2(u[p + tap / 3][tap % 3].y);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 a = sw[tap][0][4 * half + q], c = sw[tap][1][4 * half + q];
                const se2n::f32x2 a0 = se2n::pk2(a.x, a.y), a1 = se2n::pk2(a.z, a.w);
                const se2n::f32x2 c0 = se2n::pk2(c.x, c.y), c1 = se2n::pk2(c.z, c.w);
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    acc[p][2 * q] = se2n::fma2(c0, v[p][1], se2n::fma2(a0, v[p][0], acc[p][2 * q]));
                    acc[p][2 * q + 1] = se2n::fma2(c1, v[p][1], se2n::fma2(a1, v[p][0], acc[p][2 * q + 1]));
                }
            }
        }
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            uint32_t h[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int co = 16 * half + 2 * q;
                const __nv_bfloat162 w2 = __floats2bfloat162_rn(fmaxf(se2n::lo2(acc[p][q]) + sb[co], 0.0f),
                                                                fmaxf(se2n::hi2(acc[p][q]) + sb[co + 1], 0.0f));
                h[q] = *(const uint32_t *)&w2;
            }
            // two lanes exchange 16 bytes, so that they store 32 of one pixel, then 32 of the other
            const bool odd = tx & 1;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t g = __shfl_xor_sync(0xffffffffu, odd ? h[k] : h[4 + k], 1);
                h[k] = odd ? g : h[k];
                h[4 + k] = odd ? h[4 + k] : g;
            }
            // (W is even: both pixels or none)
            if (x < W && y + p < H) {
                uint4 *dst = (uint4 *)(out + ((b * H + y + p) * W + (x & ~1)) * 32) + 2 * half + (tx & 1);
                dst[0] = make_uint4(h[0], h[1], h[2], h[3]);
                dst[4] = make_uint4(h[4], h[5], h[6], h[7]);
            }
        }
    }
}

// Gradient into an encoder output e: g_e = (pool_backward(g_pooled) + g_skip) * (e > 0),
// 8 channels (16 bytes) per thread; e has lde channels per pixel.
__global__ void k_pool_bwd_add_mask(const __nv_bfloat16 *gp, const __nv_bfloat16 *gskip, const __nv_bfloat16 *e,
                                    int lde, __nv_bfloat16 *ge, int B, int H, int W, int C) {
    const int C8 = C / 8, Ho = H / 2, Wo = W / 2;
    const long long total = (long long)B * H * W * C8;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i % C8) * 8;
        const long long pix = i / C8;
        const int x = (int)(pix % W);
        const long long t = pix / W;
        const int y = (int)(t % H);
        const long long b = t / H;
        const uint4 vp = *(const uint4 *)(gp + ((b * Ho + y / 2) * Wo + x / 2) * C + c);
        const uint4 ve = *(const uint4 *)(e + pix * lde + c);
        uint4 vs = make_uint4(0, 0, 0, 0);
        if (gskip) vs = *(const uint4 *)(gskip + pix * C + c);
        const __nv_bfloat16 *hp = (const __nv_bfloat16 *)&vp, *he = (const __nv_bfloat16 *)&ve,
                            *hs = (const __nv_bfloat16 *)&vs;
        __align__(16) __nv_bfloat16 o[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            float v = 0.25f * __bfloat162float(hp[k]);
            if (gskip) v += __bfloat162float(hs[k]);
            if (!(__bfloat162float(he[k]) > 0.0f)) v = 0.0f;
            o[k] = __float2bfloat16_rn(v);
        }
        *(uint4 *)(ge + pix * C + c) = *(const uint4 *)o;
    }
}

// Gradient into a half-resolution tensor d that was upsampled (nearest):
// g_d = (sum over the 2x2 block of g_up) * (d > 0), 8 channels per thread.
__global__ void k_up_bwd_mask(const __nv_bfloat16 *gup, const __nv_bfloat16 *d, __nv_bfloat16 *gd, int B, int Hl,
                              int Wl, int C) {
    const int C8 = C / 8, H = 2 * Hl, W = 2 * Wl;
    const long long total = (long long)B * Hl * Wl * C8;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i % C8) * 8;
        const long long pix = i / C8;
        const int x = (int)(pix % Wl);
        const long long t = pix / Wl;
        const int y = (int)(t % Hl);
        const long long b = t / Hl;
        const long long base = ((b * H + 2 * y) * W + 2 * x) * C + c;
        const uint4 q0 = *(const uint4 *)(gup + base), q1 = *(const uint4 *)(gup + base + C);
        const uint4 q2 = *(const uint4 *)(gup + base + (long long)W * C);
        const uint4 q3 = *(const uint4 *)(gup + base + (long long)W * C + C);
        const uint4 vd = *(const uint4 *)(d + pix * C + c);
        const __nv_bfloat16 *a = (const __nv_bfloat16 *)&q0, *b1 = (const __nv_bfloat16 *)&q1,
                            *c2 = (const __nv_bfloat16 *)&q2, *d3 = (const __nv_bfloat16 *)&q3,
                            *hd = (const __nv_bfloat16 *)&vd;
        __align__(16) __nv_bfloat16 o[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            float v = __bfloat162float(a[k]) + __bfloat162float(b1[k]) + __bfloat162float(c2[k]) +
                      __bfloat162float(d3[k]);
            if (!(__bfloat162float(hd[k]) > 0.0f)) v = 0.0f;
            o[k] = __float2bfloat16_rn(v);
        }
        *(uint4 *)(gd + pix * C + c) = *(const uint4 *)o;
    }
}

// Loss L = mean over pixels of (out - target)^2 and its gradient at the
// head, back into d: g_d[p][c] = g_out[p] w[c] (d > 0); also the head's
// parameter gradients. One pixel's 32 channels per thread (four 16-byte
// loads and stores); the partial sums are reduced across the warp with
// shuffles, then across the block in shared memory, one atomic each.
__global__ void __launch_bounds__(256) k_loss_head_bwd(const float *out, const float *target,
                                                       const __nv_bfloat16 *d, const float *w, __nv_bfloat16 *gd,
                                                       float *gw, float *gb, float *loss, long long P, int C,
                                                       float inv_n) {
    __shared__ float sgw[8][33];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float lg = 0.0f, lb = 0.0f;
    float lw[32], wc[32];
#pragma unroll
    for (int c = 0; c < 32; ++c) {
        lw[c] = 0.0f;
        wc[c] = w[c];
    }
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < P; p += (long long)gridDim.x * blockDim.x) {
        const float r = out[p] - target[p];
        lg += r * r;
        const float go = 2.0f * r * inv_n;
        lb += go;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint4 v = *(const uint4 *)(d + p * C + 8 * q);
            const __nv_bfloat16 *h = (const __nv_bfloat16 *)&v;
            __align__(16) __nv_bfloat16 o[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float dv = __bfloat162float(h[k]);
                lw[8 * q + k] = fmaf(go, dv, lw[8 * q + k]);
                o[k] = __float2bfloat16_rn(dv > 0.0f ? go * wc[8 * q + k] : 0.0f);
            }
            *(uint4 *)(gd + p * C + 8 * q) = *(const uint4 *)o;
        }
    }
#pragma unroll
    for (int c = 0; c < 32; ++c) {
        float v = lw[c];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) sgw[wid][c] = v;
    }
    for (int o = 16; o > 0; o >>= 1) {
        lg += __shfl_xor_sync(0xffffffffu, lg, o);
        lb += __shfl_xor_sync(0xffffffffu, lb, o);
    }
    if (lane == 0) {
        sgw[wid][32] = lb;
        atomicAdd(loss, lg * inv_n);
    }
    __syncthreads();
    if (threadIdx.x < 33) {
        float t = 0.0f;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += sgw[k][threadIdx.x];
        if (threadIdx.x < 32) atomicAdd(gw + threadIdx.x, t);
        else atomicAdd(gb, t);
    }
}

// Adam on the FP32 master parameters; refreshes the bf16 copy of the conv
// weights (bf16 index map: for i < n_bf16_span the bf16 copy mirrors p).
__global__ void k_adam(float *p, const float *g, float *m, float *v, __nv_bfloat16 *pb, long long n, float lr,
                       float b1, float b2, float eps, float c1, float c2) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float upd = lr * (mi * c1) / (sqrtf(vi * c2) + eps);
        const float pi = p[i] - upd;
        p[i] = pi;
        pb[i] = __float2bfloat16_rn(pi);
    }
}

__global__ void k_to_bf16(const float *p, __nv_bfloat16 *pb, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        pb[i] = __float2bfloat16_rn(p[i]);
}

// Per-image residual on the known pixels: r[b] = sqrt(mean over known
// pixels of (out - f)^2) (the fallback criterion of the surrogate).
__global__ void k_known_residual(const float *out, const float *f, const uint8_t *mask, int HW, float *r) {
    const int b = blockIdx.x;
    float s = 0.0f, n = 0.0f;
    for (int i = threadIdx.x; i < HW; i += blockDim.x) {
        const long long p = (long long)b * HW + i;
        if (mask[p]) {
            const float d = out[p] - f[p];
            s += d * d;
            n += 1.0f;
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        n += __shfl_xor_sync(0xffffffffu, n, o);
    }
    __shared__ float ss[32], sn[32];
    if ((threadIdx.x & 31) == 0) {
        ss[threadIdx.x >> 5] = s;
        sn[threadIdx.x >> 5] = n;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float ts = 0.0f, tn = 0.0f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            ts += ss[w];
            tn += sn[w];
        }
        r[b] = tn > 0.0f ? sqrtf(ts / tn) : 0.0f;
    }
}

int grid_for(long long n) {
    long long g = (n + 255) / 256;
    if (g > 65536) g = 65536;
    return (int)(g < 1 ? 1 : g);
}

}  // namespace

namespace se2n {
namespace nn {

cudaError_t dgrad_weights(const __nv_bfloat16 *w, __nv_bfloat16 *wt, const ConvLayers &d, cudaStream_t s) {
    k_transpose_dgrad<<<dim3(48, d.n), 256, 0, s>>>(w, wt, d);
    return cudaGetLastError();
}

cudaError_t colsum(const __nv_bfloat16 *g, long long P, int C, float *db, cudaStream_t s) {
    k_colsum<<<1024, 256, 0, s>>>(g, P, C, db);
    return cudaGetLastError();
}

cudaError_t pack_input(const float *f, const uint8_t *mask, __nv_bfloat16 *x, long long P, cudaStream_t s) {
    k_pack_input<<<grid_for(P), 256, 0, s>>>(f, mask, x, P);
    return cudaGetLastError();
}

cudaError_t upsample_into(const __nv_bfloat16 *lo, int C1, __nv_bfloat16 *out, int ldo, int B, int H, int W,
                          cudaStream_t s) {
    k_upsample_into<<<B * H, 256, 0, s>>>(lo, C1, out, ldo, H, W);
    return cudaGetLastError();
}

cudaError_t conv0_direct(const float *f, const uint8_t *mask, const __nv_bfloat16 *w, const float *bias,
                         __nv_bfloat16 *out, int B, int H, int W, cudaStream_t s) {
    // a few blocks per SM, each over many pixels: the weight table is built once per block
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    int g = grid_for((long long)B * H * W);
    if (nsm > 0 && g > 8 * nsm) g = 8 * nsm;
    k_conv0<<<g, 256, 0, s>>>(f, mask, w, bias, out, B, H, W);
    return cudaGetLastError();
}

cudaError_t pool_backward_add_mask(const __nv_bfloat16 *gp, const __nv_bfloat16 *gskip, const __nv_bfloat16 *e, int lde,
                                   __nv_bfloat16 *ge, int B, int H, int W, int C, cudaStream_t s) {
    k_pool_bwd_add_mask<<<grid_for((long long)B * H * W * C / 8), 256, 0, s>>>(gp, gskip, e, lde, ge, B, H, W, C);
    return cudaGetLastError();
}

cudaError_t up_backward_mask(const __nv_bfloat16 *gup, const __nv_bfloat16 *d, __nv_bfloat16 *gd, int B, int Hl,
                             int Wl, int C, cudaStream_t s) {
    k_up_bwd_mask<<<grid_for((long long)B * Hl * Wl * C / 8), 256, 0, s>>>(gup, d, gd, B, Hl, Wl, C);
    return cudaGetLastError();
}

cudaError_t loss_head_backward(const float *out, const float *target, const __nv_bfloat16 *d, const float *w,
                               __nv_bfloat16 *gd, float *gw, float *gb, float *loss, long long P, int C,
                               cudaStream_t s) {
    int g = grid_for(P);
    if (g > 2048) g = 2048;
    k_loss_head_bwd<<<g, 256, 0, s>>>(out, target, d, w, gd, gw, gb, loss, P, C, 1.0f / (float)P);
    return cudaGetLastError();
}

cudaError_t adam(float *p, const float *g, float *m, float *v, __nv_bfloat16 *pb, long long n, float lr, float b1,
                 float b2, float eps, int t, cudaStream_t s) {
    const float c1 = 1.0f / (1.0f - powf(b1, (float)t));
    const float c2 = 1.0f / (1.0f - powf(b2, (float)t));
    k_adam<<<grid_for(n), 256, 0, s>>>(p, g, m, v, pb, n, lr, b1, b2, eps, c1, c2);
    return cudaGetLastError();
}

cudaError_t to_bf16(const float *p, __nv_bfloat16 *pb, long long n, cudaStream_t s) {
    k_to_bf16<<<grid_for(n), 256, 0, s>>>(p, pb, n);
    return cudaGetLastError();
}

cudaError_t known_residual(const float *out, const float *f, const uint8_t *mask, int B, int HW, float *r,
                           cudaStream_t s) {
    k_known_residual<<<B, 256, 0, s>>>(out, f, mask, HW, r);
    return cudaGetLastError();
}

}  // namespace nn
}  // namespace se2n
