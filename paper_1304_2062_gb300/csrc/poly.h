// Host side of the interval polynomials (poly.cuh): the coefficient tables.
#pragma once

constexpr int kPolyBuckets = 8;
constexpr int kPolyMax = 64;  // coefficients a bucket

// Coefficients of one interval's polynomial, a kernel parameter (2.1 KB).
// Bucket b holds the frequencies with wx^2 + wy^2 in [b, b + 1) * 2 / buckets.
struct PolyTable {
    int reinsch;             // 0: increment form (Horner), 1: Reinsch's recurrence
    int len;                 // row length in use: max over the buckets of m
    float inv_beta;
    int m[kPolyBuckets];     // coefficients of the bucket (>= 2), the rest of its row is zero
    float h[kPolyBuckets];   // centre of the spectrum of -A / beta
    float c[kPolyBuckets][kPolyMax];
};

// Fill t for S steps of dt = T / S. False where the polynomial form does not
// apply: beta below 1e-12, a Crank-Nicolson factor may be negative (dt (2 + 4 beta) > 2, where
// f oscillates up to -1 and is no longer smooth), or more than kPolyMax
// coefficients would be needed.
bool se2n_poly_make(double beta, double T, int steps, PolyTable &t);
// Packed instructions an angle of the widest bucket (the cost estimate).
int se2n_poly_cost(const PolyTable &t);
