// Coefficient tables of the interval polynomials (poly.cuh has the method): plain host
// arithmetic, no CUDA.
#include "poly.h"

#include <math.h>
#include <string.h>

namespace {

// f(x) - 1 of S steps at x in [-w, 0]
double interval_minus_one(double x, double dt, int S) {
    const double u = fmax(0.5 * dt * x, -1.0);
    return expm1(2.0 * S * atanh(u));
}

constexpr int kNodesMax = 128;

// The degree of a series grows as the square root of T w (poly.cuh); half as many nodes
// again, a whole number of pairs +-u.
int nodes_for(double T, double w) {
    const int n = 2 * (int)(0.75 * sqrt(18.4 * T * w) + 10.0);
    return n < kNodesMax ? n : kNodesMax;
}

// Chebyshev series on [-w, 0], len of its coefficients known (double precision).
struct Series {
    double w;
    int len;
    double c[kNodesMax];
};

// Chebyshev coefficients of g (increment form) or f on [-w, 0] from n nodes +-u,
// u = cos((i + 1/2) pi / n), into s (3 n / 4 of them at most: beyond, what the nodes fold
// back matters). Returns how many are above the tolerance, or -1 when the tail does
// not fall below it there. The function's values come from its series on a wider
// interval where there is one (a table of eight widths needs one set of exponentials: 13 us
// of host time at T = 2, 70 at T = 50; with a set each 28 and 183).
int cheb(double w, double T, double dt, int S, bool inc, int n, const Series *wide, Series &s) {
    const int half = n / 2, most = 3 * n / 4;
    // the function's even and odd parts, which have the even and odd coefficients
    double u[kNodesMax / 2], part[2][kNodesMax / 2], tk[kNodesMax / 2], tp[kNodesMax / 2];
    for (int i = 0; i < half; ++i) u[i] = cos((i + 0.5) * M_PI / n);
    for (int z = 0; z < 2; ++z) {
        double v[kNodesMax / 2];
        if (wide) {  // Clenshaw's recurrence at all the nodes
            double y2[kNodesMax / 2], b1[kNodesMax / 2], b2[kNodesMax / 2];
            for (int i = 0; i < half; ++i) {
                y2[i] = 2.0 * (w * ((z ? -u[i] : u[i]) - 1.0) / wide->w + 1.0);
                b1[i] = b2[i] = 0.0;
            }
            for (int k = wide->len - 1; k > 0; --k)
                for (int i = 0; i < half; ++i) {
                    const double b = y2[i] * b1[i] - b2[i] + wide->c[k];
                    b2[i] = b1[i];
                    b1[i] = b;
                }
            for (int i = 0; i < half; ++i) v[i] = 0.5 * y2[i] * b1[i] - b2[i] + wide->c[0];
        } else {
            for (int i = 0; i < half; ++i) {
                const double x = 0.5 * w * ((z ? -u[i] : u[i]) - 1.0);
                const double f1 = interval_minus_one(x, dt, S);
                v[i] = inc ? (x > -1e-12 * w ? T : f1 / x) : f1 + 1.0;
            }
        }
        for (int i = 0; i < half; ++i) {
            part[0][i] = z ? part[0][i] + v[i] : v[i];
            part[1][i] = z ? part[1][i] - v[i] : v[i];
        }
    }
    for (int i = 0; i < half; ++i) {
        tk[i] = 1.0;
        tp[i] = u[i];  // T_{-1} = T_1
    }
    // what is cut off changes f(A) x by at most 2e-8 |x| (FP32 resolves 6e-8)
    const double tol = 2e-8 / (inc ? w : 1.0);
    s.w = w;
    s.len = 0;
    for (int k = 0, small = 0; k < most && small < 4; ++k) {
        const double *v = part[k & 1];
        double sum[4] = {0.0, 0.0, 0.0, 0.0};  // four chains: one would wait for every addition
        for (int i = 0; i < half; ++i) {
            sum[i & 3] += v[i] * tk[i];
            const double next = (k == 0 ? u[i] : 2.0 * u[i] * tk[i] - tp[i]);
            tp[i] = tk[i];
            tk[i] = next;
        }
        s.c[k] = (k == 0 ? 1.0 : 2.0) * ((sum[0] + sum[1]) + (sum[2] + sum[3])) / n;
        // both parities have come down far below the tolerance: so have all that follow
        small = fabs(s.c[k]) < 1e-6 * tol ? small + 1 : 0;
        s.len = k + 1;
    }
    double tail = 0.0;
    int m = s.len;
    while (m > 2 && tail + fabs(s.c[m - 1]) < tol) tail += fabs(s.c[--m]);
    return m > s.len - 2 ? -1 : m;
}

int cheb_auto(double w, double T, double dt, int S, bool inc, const Series *wide, Series &s) {
    for (int n = nodes_for(T, w);; n = n + n / 2 < kNodesMax ? (n + n / 2) & ~1 : kNodesMax) {
        const int m = cheb(w, T, dt, S, inc, n, wide, s);
        if (m > 0 || n == kNodesMax) return m;
    }
}

}  // namespace

bool se2n_poly_make(double beta, double T, int steps, PolyTable &t) {
    const double dt = T / steps;
    if (!(dt * (2.0 + 4.0 * beta) <= 2.0) || !(T > 0.0)) return false;
    // the kernels work with a_r^2 / beta times the spectrum, which has to stay in FP32's range
    if (!(beta >= 1e-12)) return false;
    memset(&t, 0, sizeof t);
    t.inv_beta = (float)(1.0 / beta);
    // a little wider than the bucket: FP32 rounding of wx^2 + wy^2 at its edge
    auto width = [&](int b) { return (4.0 * beta + 2.0 * (b + 1) / kPolyBuckets) * (1.0 + 1e-5); };
    Series wide, own;
    // Horner in powers of u = (M + h) / h loses at most the sum of the
    // coefficients' sizes times w in ulp of x: about T w for these functions,
    // 24 ulp (1.4e-6 of the fastest modes, far less of the slow ones) allowed.
    // Its coefficients in M must also stay clear of the ends of FP32's range.
    bool horner = true;
    for (int b = kPolyBuckets - 1; b >= 0 && horner; --b) {  // the widest first: it decides
        const double w = width(b), h = 0.5 * w / beta;
        Series &s = b == kPolyBuckets - 1 ? wide : own;
        const int m = cheb_auto(w, T, dt, steps, true, b == kPolyBuckets - 1 ? nullptr : &wide, s);
        if (m < 0 || m > 32) {
            horner = false;
            break;
        }
        // Chebyshev to powers of u: T_{k+1} = 2 u T_k - T_{k-1}
        double p[33] = {0}, t0[33] = {0}, t1[33] = {0};
        t0[0] = 1.0;
        t1[1] = 1.0;
        for (int k = 0; k < m; ++k) {
            for (int i = 0; i <= k; ++i) p[i] += s.c[k] * t0[i];
            double t2[33] = {0};
            for (int i = 0; i <= k + 1 && i < 32; ++i) t2[i + 1] = 2.0 * t1[i];
            for (int i = 0; i <= k; ++i) t2[i] -= t0[i];
            memcpy(t0, t1, sizeof t0);
            memcpy(t1, t2, sizeof t1);
        }
        double sum = 0.0, power = beta;
        for (int i = 0; i < m; ++i) {
            sum += fabs(p[i]);
            const double q = p[i] * power;  // beta h^-i
            power /= h;
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
    for (int b = kPolyBuckets - 1; b >= 0; --b) {
        const double w = width(b);
        Series &s = b == kPolyBuckets - 1 ? wide : own;
        const int m = cheb_auto(w, T, dt, steps, false, b == kPolyBuckets - 1 ? nullptr : &wide, s);
        if (m < 0 || m > kPolyMax) return false;
        for (int i = 0; i < m; ++i) t.c[b][i] = (float)s.c[i];
        t.m[b] = m;
        t.h[b] = (float)(0.5 * w / beta);
        t.len = t.len > m ? t.len : m;
    }
    return true;
}

int se2n_poly_cost(const PolyTable &t) { return t.reinsch ? 5 * (t.len - 1) + 2 : 3 * (t.len - 1) + 6; }
