// How a weight gradient (k_wgrad_tma, conv_tma.cuh) is split over CTAs: plain host
// arithmetic, and what the kernel shares of it.
#pragma once

#ifdef __CUDACC__
#define SE2N_HD __host__ __device__ __forceinline__
#else
#define SE2N_HD inline
#endif

namespace se2n {
namespace nn {
namespace tma {

constexpr int kWgR = 8;  // image rows of a pixel block

struct WgradGeo {
    int B, H, W;        // of the tensors as read (W columns of F pixels)
    int C, Cout;        // channels of the layer
    int F;              // pixels a column
    int bkx;            // columns of a pixel block
    int xblocks, yblocks, kblocks;
    int cgroups, ngroups;  // 64-channel groups of In and gz as read
    int ksplit, per;    // pixel ranges a (channel group, channel group), blocks of each but the last
    int len;            // pixel blocks a sum at most
    int tiles;          // of a unit a CTA takes at most
    int parts;          // CTAs that share a unit's tiles, at most (the others return)
};

// Column offsets s0 .. s1 of a unit: -1 needs In's last pixel and gz's first one, 1 the
// reverse (c0 / C is 0 and every group holds all there is when F = 1).
SE2N_HD void wgrad_offsets(const WgradGeo &g, int c0, int n0, int &s0, int &s1) {
    s0 = g.F == 1 || ((c0 + 63) / g.C >= g.F - 1 && n0 / g.Cout == 0) ? -1 : 0;
    s1 = g.F == 1 || (c0 / g.C == 0 && (n0 + 63) / g.Cout >= g.F - 1) ? 1 : 0;
}
// Its tiles: (dy -1 | 0) of each offset, dy 1 of two offsets each.
SE2N_HD int wgrad_tiles(int s0, int s1) {
    const int ns = s1 - s0 + 1;
    return ns + (ns + 1) / 2;
}

// Terms of the longest sum a weight gradient was made of before its boxes held whole
// rows of blocks: runs of up to 64 pixels of a row, in as many ranges as give two units an
// SM of tiles of 128 (tap, channel) rows.
inline int wgrad_terms(int B, int H, int W, int C, int sms) {
    const int run = W < 64 ? W : 64, runs = B * H * ((W + run - 1) / run), mtiles = (9 * C + 127) / 128;
    int ranges = (2 * sms + mtiles - 1) / mtiles;
    if (ranges > runs) ranges = runs;
    return (runs + ranges - 1) / ranges * run;
}

// The layer of W pixels a row read as columns, and its split. The tensor core's sums
// truncate, so a sum loses bits in proportion to its length: it ends after as many blocks as
// make it wgrad_terms() long (a column of F pixels adds one term to each sum) or after
// one, is added to dW, and the next begins. Shorter ones move the result the
// other way (3.7e-9 a term), so ranges are at most a quarter and a thousand terms shorter.
// Within that the split is what takes the fewest cycles by the kernel's bounds, the boxes'
// rows (2.7 cycles each), the products (80 each) and the additions to dW, over whole waves
// of CTAs.
inline bool wgrad_split(WgradGeo &g, int B, int H, int W, int C, int Cout, int sms) {
    g.B = B;
    g.H = H;
    g.C = C;
    g.Cout = Cout;
    g.F = C % 64 == 0 && Cout % 64 == 0 ? 1 : C % 32 == 0 ? 2 : 8;
    if ((g.F * C) % 64 || Cout % 32 || W % g.F || sms < 1) return false;
    g.W = W / g.F;
    g.bkx = g.W > 16 ? 32 : 16;
    g.xblocks = (g.W + g.bkx - 1) / g.bkx;
    g.yblocks = (H + kWgR - 1) / kWgR;
    g.kblocks = B * g.xblocks * g.yblocks;
    g.cgroups = g.F * C / 64;
    g.ngroups = g.F * Cout / 64;
    int most = wgrad_terms(B, H, W, C, sms) / (kWgR * g.bkx);
    if (most > g.kblocks) most = g.kblocks;
    if (most < 1) most = 1;
    g.len = most;
    const int terms = kWgR * g.bkx;
    int least = most - 1024 / terms;
    if (least < (3 * most + 3) / 4) least = (3 * most + 3) / 4;
    const double rows = 2.7 * ((kWgR + 2) * (g.bkx + 2) + terms);
    double best = 0.0;
    for (int parts = g.F == 8 ? 1 : 3; parts >= 1; --parts) {
        const int tiles = (5 + parts - 1) / parts;
        int ctas = 0, widest = 0;  // a range
        for (int gr = 0; gr < g.cgroups * g.ngroups; ++gr) {
            int s0, s1;
            wgrad_offsets(g, gr % g.cgroups * 64, gr / g.cgroups * 64, s0, s1);
            const int t = wgrad_tiles(s0, s1);
            ctas += (t + tiles - 1) / tiles;
            if (t > widest) widest = t;
        }
        if (widest > tiles) widest = tiles;
        const double products = 80.0 * kWgR * (g.bkx / 16) * widest, block = rows > products ? rows : products;
        for (int waves = 1; waves <= 8; ++waves) {
            int per = waves * sms / ctas;  // ranges, then blocks a range
            per = per < 1 ? g.kblocks : (g.kblocks + per - 1) / per;
            if (per < least) per = least;
            const int ranges = (g.kblocks + per - 1) / per, sums = (per + g.len - 1) / g.len;
            const double cycles = (double)(((long long)ranges * ctas + sms - 1) / sms) *
                                  (per * block + sums * (1000.0 + 2000.0 * widest));
            if (best == 0.0 || cycles < best) {
                best = cycles;
                g.parts = parts;
                g.tiles = tiles;
                g.ksplit = ranges;
                g.per = per;
            }
        }
    }
    return true;
}

}  // namespace tma
}  // namespace nn
}  // namespace se2n
