// The kernel that applies an interval polynomial to an angle-major spectrum
// (poly.cuh has the method, poly_table.cu makes the coefficients).
#include "dependent.cuh"
#include "poly.cuh"

#include <climits>

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
