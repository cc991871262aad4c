// The interval as a polynomial of its operator. S Crank-Nicolson steps of one
// frequency are one linear map f(A), f(x) = ((1 + dt x / 2) / (1 - dt x / 2))^S,
// of the symmetric operator A = -diag(a_r^2) + beta L of eq. (4.2) (L: cyclic
// second difference), whose spectrum lies in [-w, 0], w = max a_r^2 + 4 beta
// (Gershgorin). f is smooth there, so the polynomial that truncates its
// Chebyshev series (Trefethen's "Approximation Theory and Approximation
// Practice", chapters 3 and 8) below FP32 resolution has a low degree: about
// 12 for T w / 2 = 3, about sqrt(2 T w ln 1e8) for large T w, whatever S is.
// Every multiplication by A is a three-point cyclic stencil on the N-vector,
// so a whole interval costs as much as that many explicit steps and needs no
// matrices: x stays in registers, the coefficients are kernel parameters.
//
// With M = A / beta, applied as (M b)_r = b_{r-1} + b_{r+1} - (2 + e_r) b_r,
// e_r = a_r^2 / beta, there are two forms (packed real and imaginary parts):
//
//   increment   x + g(A) A x with g(x) = (f(x) - 1) / x: y = M x once (the
//               constant mode of the zero frequency gives exactly 0, so it
//               comes back bit-identical, and slow modes carry rounding
//               relative to their change), then Horner's rule in M + h,
//               h = w / (2 beta) the centre of the spectrum:
//               b <- (M + h) b + q_k y, 3 packed instructions an angle and
//               degree. The coefficients in powers of (M + h) / h are those of
//               exp-like functions, all of one sign and summing to T, so
//               Horner loses nothing while T w is moderate.
//   Reinsch     f(A) x by Clenshaw's recurrence with Reinsch's differences
//               d_k = c_k x + (2 / h) M b_{k+1} + d_{k+1}, b_k = b_{k+1} + d_k
//               (Oliver, "Rounding error propagation in polynomial evaluation
//               schemes", 1979): M unshifted, so slow modes, the ones near the
//               edge 0 of the spectrum where Clenshaw's own form loses m^2 ulp,
//               keep their accuracy at large T w; 5 packed instructions.
//
// Frequencies are sorted into buckets by a bound on a_r^2 <= wx^2 + wy^2 and
// every bucket has its own w and so its own degree (its coefficients are
// padded with zeros on top, which a longer loop runs through unchanged). A
// frequency's arithmetic therefore depends on nothing but its own k and l:
// neither on the launch shape nor on its neighbours in a warp.
#pragma once

#include "diffuse_x2.cuh"
#include "poly.h"

namespace se2n {

// Copy the coefficient rows from the kernel's parameters to shared memory
// (buckets x len floats), where lanes of different buckets read them side by side.
__device__ __forceinline__ void poly_stage(float *sc, const PolyTable &t, int tid, int threads) {
    for (int i = tid; i < kPolyBuckets * t.len; i += threads) sc[i] = t.c[i / t.len][i % t.len];
}

// The bucket of a frequency and what depends on it.
struct PolyLane {
    const float *c;  // coefficients, lowest first, in shared memory
    float h;         // centre of the spectrum of -M
    int m;           // coefficients that are not padding
};
__device__ __forceinline__ PolyLane poly_lane(const float *sc, const PolyTable &t, float wx, float wy) {
    const float w2 = fmaf(wx, wx, wy * wy);
    const int b = min(kPolyBuckets - 1, (int)(w2 * (kPolyBuckets * 0.5f)));
    PolyLane p;
    p.c = sc + b * t.len;
    p.h = t.h[b];
    p.m = t.m[b];
    return p;
}

// b_{r-1} of a lane's first angle and b_{r+1} of its last, from the first and
// last angles of the P adjacent lanes that share the frequency.
template <int P>
__device__ __forceinline__ void poly_edges(f32x2 first, f32x2 last, f32x2 &lo, f32x2 &hi) {
    if constexpr (P == 1) {
        lo = last;
        hi = first;
    } else if constexpr (P == 2) {
        lo = xshfl2(last, 1);
        hi = xshfl2(first, 1);
    } else {
        const int lane = threadIdx.x & 31, base = lane & ~(P - 1);
        const int dn = base | ((lane - 1) & (P - 1)), up = base | ((lane + 1) & (P - 1));
        lo = pk2(__shfl_sync(0xffffffffu, lo2(last), dn), __shfl_sync(0xffffffffu, hi2(last), dn));
        hi = pk2(__shfl_sync(0xffffffffu, lo2(first), up), __shfl_sync(0xffffffffu, hi2(first), up));
    }
}

// Runs b <- step(b) `steps` times in place, b_r <- step(b_{r-1}, b_r, b_{r+1},
// r, c) with c the next lower coefficient, c[steps - 1] first. The two ends of
// the lane's angles go first, so that their exchange with the adjacent lanes
// runs behind the inner angles (N = 32, 1024 x 1024, T = 2: 135 us against 145
// with the exchange at the start of the step).
template <int K, int P, typename Step>
__device__ __forceinline__ void poly_steps(f32x2 (&b)[K], const float *c, int steps, Step step) {
    static_assert(K >= 3, "an inner angle");
    f32x2 lo, hi;
    poly_edges<P>(b[0], b[K - 1], lo, hi);
    float cn = c[max(steps - 1, 0)];
#pragma unroll 1
    for (int k = steps - 1; k >= 0; --k) {
        const f32x2 ck = dup2(cn);
        cn = c[max(k - 1, 0)];
        const f32x2 first = step(lo, b[0], b[1], 0, ck), last = step(b[K - 2], b[K - 1], hi, K - 1, ck);
        poly_edges<P>(first, last, lo, hi);
        f32x2 prev = b[0];
#pragma unroll
        for (int j = 1; j < K - 1; ++j) {
            const f32x2 cur = b[j];
            b[j] = step(prev, cur, b[j + 1], j, ck);
            prev = cur;
        }
        b[0] = first;
        b[K - 1] = last;
    }
}

// The increment form of one frequency group: v <- g(A) A v for the K angles of
// each of the P lanes (e[j] = a_r^2 / beta of the lane's angles). Every lane of
// the warp calls it together, as the functions below.
template <int K, int P>
__device__ __forceinline__ void poly_increment(f32x2 (&v)[K], const float (&e)[K], const PolyLane &p) {
    const int top = (int)__reduce_max_sync(0xffffffffu, (unsigned)p.m) - 1;  // highest coefficient in the warp
    f32x2 lo, hi, b[K], nd[K];
    poly_edges<P>(v[0], v[K - 1], lo, hi);
    const f32x2 ct = dup2(p.c[top]), m2 = dup2(-2.0f);
    f32x2 prev = lo;
#pragma unroll
    for (int j = 0; j < K; ++j) {
        const f32x2 cur = v[j], next = j == K - 1 ? hi : v[j + 1];
        v[j] = fma2(dup2(-e[j]), cur, fma2(m2, cur, add2(prev, next)));
        nd[j] = dup2((p.h - 2.0f) - e[j]);
        b[j] = mul2(ct, v[j]);
        prev = cur;
    }
    poly_steps<K, P>(b, p.c, top, [&](f32x2 l, f32x2 o, f32x2 r, int j, f32x2 ck) {
        return fma2(ck, v[j], fma2(nd[j], o, add2(l, r)));
    });
#pragma unroll
    for (int j = 0; j < K; ++j) v[j] = b[j];
}

// x <- f(A) x in either form.
template <int K, int P, bool REINSCH>
__device__ __forceinline__ void poly_apply(f32x2 (&x)[K], const float (&e)[K], const PolyLane &p) {
    if constexpr (!REINSCH) {
        f32x2 v[K];
#pragma unroll
        for (int j = 0; j < K; ++j) v[j] = x[j];
        poly_increment<K, P>(v, e, p);
#pragma unroll
        for (int j = 0; j < K; ++j) x[j] = add2(x[j], v[j]);
    } else {
        const int top = (int)__reduce_max_sync(0xffffffffu, (unsigned)p.m) - 1;
        f32x2 lo, hi, b[K], ne[K], d[K];
        const f32x2 ct = dup2(p.c[top]), ih = dup2(1.0f / p.h), kap = dup2(2.0f / p.h);
#pragma unroll
        for (int j = 0; j < K; ++j) {
            ne[j] = dup2(-2.0f - e[j]);
            b[j] = mul2(ct, x[j]);
            d[j] = b[j];
        }
        poly_steps<K, P>(b, p.c + 1, top - 1, [&](f32x2 l, f32x2 o, f32x2 r, int j, f32x2 ck) {
            d[j] = fma2(kap, fma2(ne[j], o, add2(l, r)), fma2(ck, x[j], d[j]));
            return add2(o, d[j]);
        });
        const f32x2 c0 = dup2(p.c[0]);
        poly_edges<P>(b[0], b[K - 1], lo, hi);
#pragma unroll
        for (int j = 0; j < K; ++j) {
            const f32x2 L = j == 0 ? lo : b[j - 1], R = j == K - 1 ? hi : b[j + 1];
            x[j] = fma2(ih, fma2(ne[j], b[j], add2(L, R)), fma2(c0, x[j], d[j]));
        }
    }
}

// Lanes a frequency in the kernels on an angle-major volume: up to 16 angles a
// lane. Twice the lanes with half the angles need half the registers but twice
// the exchanges, and their warps touch shorter runs of each plane (1024 x 1024,
// T = 2: N = 16, 32, 64 in 83, 172, 397 us against 70, 143, 301).
template <int N>
__host__ __device__ constexpr int poly_lanes() {
    return N <= 16 ? 1 : N <= 32 ? 2 : 4;
}

// One frequency of an angle-major volume vol[N][HW], fc = k Wc + l: the
// counterpart of diffuse_group_x2. Every lane of the warp calls it together;
// a lane with !active works on a valid frequency without storing.
template <int N, bool REINSCH>
__device__ __forceinline__ void poly_group(const PolyTable &t, const float *sc, const float *cs, const float *sn,
                                           float2 *vol, int H, int W, int Wc, long long HW, long long fc, bool active,
                                           int k0) {
    constexpr int P = poly_lanes<N>(), K = N / P;
    static_assert(K * P == N, "whole angles a lane");
    const int r0 = (threadIdx.x & (P - 1)) * K;
    float2 *col = vol + (long long)r0 * HW + fc;
    f32x2 x[K];
#pragma unroll
    for (int j = 0; j < K; ++j) {
        const float2 v = __ldcg(col + j * HW);
        x[j] = pk2(v.x, v.y);
    }
    const int k = (int)(fc / Wc);
    const int l = (int)(fc - (long long)k * Wc);
    const float wx = sin_2pi_frac(l, W);
    const float wy = sin_2pi_frac(k0 + k, H);
    float e[K];
#pragma unroll
    for (int j = 0; j < K; ++j) {
        const float ar = fmaf(wx, cs[r0 + j], wy * sn[r0 + j]);
        e[j] = ar * ar * t.inv_beta;
    }
    // Where every a_r is 0 the constant vectors are fixed points of the steps and of the
    // increment form, bit for bit. Reinsch's form sums its coefficients, one rounding
    // away from 1: there such a vector is left as it is in memory.
    // (A lane looks at all the angles itself: with the warp's shuffles in the branch every
    // frequency's polynomial was 4 % slower.)
    if (REINSCH && wx == 0.0f && wy == 0.0f) {
        const float2 *p = vol + fc, v0 = __ldcg(p);
        bool same = true;
#pragma unroll 1
        for (int r = 1; r < N; ++r) {
            const float2 v = __ldcg(p + r * HW);
            same = same && v.x == v0.x && v.y == v0.y;
        }
        active = active && !same;
    }
    poly_apply<K, P, REINSCH>(x, e, poly_lane(sc, t, wx, wy));
    // form the addresses again: kept across the polynomial they take 2 K registers
    asm volatile("" : "+l"(col), "+l"(HW));
    if (active) {
#pragma unroll
        for (int j = 0; j < K; ++j) col[j * HW] = make_float2(lo2(x[j]), hi2(x[j]));
    }
}

}  // namespace se2n
