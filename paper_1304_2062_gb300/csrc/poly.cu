// Coefficient tables of the interval polynomials (host) and the kernel that
// applies them to an angle-major spectrum (poly.cuh has the method).
#include "dependent.cuh"
#include "poly.cuh"

#include <math.h>
#include <string.h>

#include <climits>

namespace {

// f(x) - 1 of S steps at x in [-w, 0]
double interval_minus_one(double x, double dt, int S) {
    const double u = fmax(0.5 * dt * x, -1.0);
    return expm1(2.0 * S * atanh(u));
}

constexpr int kNodesMax = 256;

// Chebyshev coefficients of g (increment form) or f on [-w, 0] from n nodes
// into c[0 .. n/2), returns how many are above the tolerance, or -1 when the
// tail does not fall below it within n/2.
int cheb(double w, double T, double dt, int S, bool inc, int n, double *c) {
    double u[kNodesMax], v[kNodesMax], tk[kNodesMax], tp[kNodesMax];
    for (int i = 0; i < n; ++i) {
        u[i] = cos((i + 0.5) * M_PI / n);
        const double x = 0.5 * w * (u[i] - 1.0);
        const double f1 = interval_minus_one(x, dt, S);
        v[i] = inc ? (x > -1e-12 * w ? T : f1 / x) : f1 + 1.0;
        tk[i] = 1.0;
        tp[i] = u[i];  // T_{-1} = T_1
    }
    for (int k = 0; k < n / 2; ++k) {
        double s = 0.0;
        for (int i = 0; i < n; ++i) {
            s += v[i] * tk[i];
            const double next = (k == 0 ? u[i] : 2.0 * u[i] * tk[i] - tp[i]);
            tp[i] = tk[i];
            tk[i] = next;
        }
        c[k] = (k == 0 ? 1.0 : 2.0) * s / n;
    }
    // what is cut off changes f(A) x by at most 2e-8 |x| (FP32 resolves 6e-8)
    const double tol = 2e-8 / (inc ? w : 1.0);
    double tail = 0.0;
    int m = n / 2;
    while (m > 2 && tail + fabs(c[m - 1]) < tol) tail += fabs(c[--m]);
    return m > n / 2 - 2 ? -1 : m;
}

int cheb_auto(double w, double T, double dt, int S, bool inc, double *c) {
    // the degree grows as the square root of T w: start near enough nodes
    int n = 32;
    while (n < kNodesMax && n * n < 160.0 * T * w) n *= 2;
    for (; n <= kNodesMax; n *= 2) {
        const int m = cheb(w, T, dt, S, inc, n, c);
        if (m > 0) return m;
    }
    return -1;
}

}  // namespace

bool se2n_poly_make(double beta, double T, int steps, PolyTable &t) {
    const double dt = T / steps;
    if (!(dt * (2.0 + 4.0 * beta) <= 2.0) || !(T > 0.0)) return false;
    memset(&t, 0, sizeof t);
    t.inv_beta = (float)(1.0 / beta);
    // a little wider than the bucket: FP32 rounding of wx^2 + wy^2 at its edge
    auto width = [&](int b) { return (4.0 * beta + 2.0 * (b + 1) / kPolyBuckets) * (1.0 + 1e-5); };
    double c[kNodesMax / 2];
    // Horner in powers of u = (M + h) / h loses at most the sum of the
    // coefficients' sizes times w in ulp of x: about T w for these functions,
    // 24 ulp (1.4e-6 of the fastest modes, far less of the slow ones) allowed.
    // Its coefficients in M must also stay clear of the ends of FP32's range.
    bool horner = true;
    for (int b = kPolyBuckets - 1; b >= 0 && horner; --b) {  // the widest first: it decides
        const double w = width(b), h = 0.5 * w / beta;
        const int m = cheb_auto(w, T, dt, steps, true, c);
        if (m < 0 || m > 32) {
            horner = false;
            break;
        }
        // Chebyshev to powers of u: T_{k+1} = 2 u T_k - T_{k-1}
        double p[33] = {0}, t0[33] = {0}, t1[33] = {0};
        t0[0] = 1.0;
        t1[1] = 1.0;
        for (int k = 0; k < m; ++k) {
            for (int i = 0; i <= k; ++i) p[i] += c[k] * t0[i];
            double t2[33] = {0};
            for (int i = 0; i <= k + 1 && i < 32; ++i) t2[i + 1] = 2.0 * t1[i];
            for (int i = 0; i <= k; ++i) t2[i] -= t0[i];
            memcpy(t0, t1, sizeof t0);
            memcpy(t1, t2, sizeof t1);
        }
        double sum = 0.0;
        for (int i = 0; i < m; ++i) {
            sum += fabs(p[i]);
            const double q = beta * p[i] * pow(h, -i);
            if (fabs(q) < 1e-30 || fabs(q) > 1e30) horner = false;
            t.c[b][i] = (float)q;
        }
        if (sum * w > 24.0) horner = false;
        t.m[b] = m;
        t.h[b] = (float)h;
        t.len = t.len > m ? t.len : m;
    }
    if (horner) return true;
    memset(t.c, 0, sizeof t.c);
    t.reinsch = 1;
    t.len = 0;
    for (int b = 0; b < kPolyBuckets; ++b) {
        const double w = width(b);
        const int m = cheb_auto(w, T, dt, steps, false, c);
        if (m < 0 || m > kPolyMax) return false;
        for (int i = 0; i < m; ++i) t.c[b][i] = (float)c[i];
        t.m[b] = m;
        t.h[b] = (float)(0.5 * w / beta);
        t.len = t.len > m ? t.len : m;
    }
    return true;
}

int se2n_poly_cost(const PolyTable &t) { return t.reinsch ? 5 * (t.len - 1) + 2 : 3 * (t.len - 1) + 6; }

namespace se2n {

// One frequency group a thread group, K <= 16 angles a lane, all of them
// loaded before the first use; the volume is read and written once. Measured
// (events, full spectrum, 1024 x 1024, one GB300) against the step kernel it
// replaces there:
//   N = 32, T = 2 in 100 steps     122 us (4.4 TB/s), steps 1391 us
//   N = 64, T = 50 in 1000 steps   925 us, steps 29.1 ms
// At T = 2 the loads and the arithmetic of a warp (77 us of packed FP32 at its
// measured rate, 79 us of copies) follow one another, so the increment form is
// held to 128 registers, 16 warps an SM (N = 16, 32, 64: 65, 122, 261 us; 71, 140,
// 302 with 12 warps). Large T is bound by the packed FP32 pipe and Reinsch's form
// runs fastest unconstrained (949 us; 1003 with 16 warps; 925 since the addresses
// are formed again for the stores instead of kept).
constexpr int kPolyBlock = 128;

template <int N, bool REINSCH>
__global__ void __launch_bounds__(kPolyBlock, REINSCH ? 3 : 4) k_poly(const __grid_constant__ PolyArgs a) {
    __shared__ float sc[kPolyBuckets * kPolyMax];
    constexpr int P = poly_lanes<N>();
    dependent_launch();
    poly_stage(sc, a.t, threadIdx.x, kPolyBlock);
    __syncthreads();
    dependent_wait();
    const long long f = ((long long)blockIdx.x * kPolyBlock + threadIdx.x) / P;
    const bool active = f < a.HW;
    poly_group<N, REINSCH>(a.t, sc, a.cs, a.sn, a.vol, a.H, a.W, a.Wc, a.HW, active ? f : a.HW - 1, active, a.k0);
}

namespace {

template <int N>
cudaError_t launch(const PolyArgs &a, cudaStream_t s) {
    const long long blocks = (a.HW * poly_lanes<N>() + kPolyBlock - 1) / kPolyBlock;
    if (blocks > INT_MAX) return cudaErrorInvalidValue;
    return launch_dependent(a.t.reinsch ? k_poly<N, true> : k_poly<N, false>, (int)blocks, kPolyBlock, 0, s, a);
}

}  // namespace

}  // namespace se2n

cudaError_t se2n_launch_poly(int N, const PolyArgs &a, cudaStream_t s) {
    switch (N) {
        case 4: return se2n::launch<4>(a, s);
        case 8: return se2n::launch<8>(a, s);
        case 12: return se2n::launch<12>(a, s);
        case 16: return se2n::launch<16>(a, s);
        case 24: return se2n::launch<24>(a, s);
        case 30: return se2n::launch<30>(a, s);
        case 32: return se2n::launch<32>(a, s);
        case 48: return se2n::launch<48>(a, s);
        case 64: return se2n::launch<64>(a, s);
        default: return cudaErrorInvalidValue;
    }
}
