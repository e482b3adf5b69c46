// The Hessian-vector product of the two optimisers' kernels, from one sample
// group's stored perturbations.
#pragma once
#include "hr_device.cuh"

namespace hr {

// H p = 1/M sum_m loss_m w_m, w_mk = (tau_mk (tau_m . p) / s^4 - p_k / s^2) n^2/S(tau_m),
// into q[n] (shared, one writer per element): FP64 weights rounded to FP32, their
// products with the losses in Kahan sums in order of m.  p [n] in shared memory;
// every thread of the block calls it; it ends with a barrier.
//
// Only the sums have an order, so the products are formed by all threads, a tile of
// rows at a time (odd pitch: no bank conflicts over rows), and one thread per
// element adds them up.  With one thread per element forming its own, the published
// optimiser's kernel (two dims, 256 perturbations) took 71 us, now 16; the Newton-CG
// one (ten products of 64 dims and 32 perturbations) 93 us, now 89: bound by FP64,
// two lanes a cycle and SM, and by the chains of sums and divisions between.
struct HvpTile {
    static constexpr int kDoubles = 3072, kRows = 512;
    double t[kDoubles];            // [rows][n | 1] perturbations, then the products (floats)
    double tp[kRows], iS[kRows];   // tau . p and n^2 / S by row
    float loss[kRows];
    double p2[64];                 // p / s^2
};

// `beside` is called by the last warp while the first ones form the tau . p.
template <class F>
__device__ __forceinline__ void hvp_product(HvpTile& S, const float* __restrict__ tau, const float* __restrict__ invS,
                                            const float* __restrict__ loss, int M, int n, const double* p, double is2,
                                            double is4, double* q, F beside) {
    const int ld = n | 1, tile = min(HvpTile::kRows, HvpTile::kDoubles / ld);
    // i / n = (i recip) >> 20 for the tile's i < rows n <= kDoubles: recip n - 2^20 < n <= 64, so the
    // quotient is exact while i 63 < 2^20, and i recip <= rows (2^20 + n) stays within 32 bits
    const uint32_t recip = (uint32_t)(((1u << 20) + (uint32_t)n - 1u) / (uint32_t)n);
    static_assert(HvpTile::kDoubles * 63 < (1 << 20) && HvpTile::kRows < (1 << 11), "division by n");
    Kahan acc;
    if (threadIdx.x < n) S.p2[threadIdx.x] = p[threadIdx.x] * is2;
    for (int m0 = 0; m0 < M; m0 += tile) {
        const int rows = min(tile, M - m0);
        for (int i = threadIdx.x; i < rows * n; i += blockDim.x) {
            const int r = (int)(((uint32_t)i * recip) >> 20), k = i - r * n;
            S.t[r * ld + k] = (double)tau[(size_t)m0 * n + i];
        }
        for (int r = threadIdx.x; r < rows; r += blockDim.x) {
            S.iS[r] = (double)invS[m0 + r];
            S.loss[r] = loss[m0 + r];
        }
        __syncthreads();
        for (int r = threadIdx.x; r < rows; r += blockDim.x) {
            double s = 0.0;
            for (int k = 0; k < n; ++k) s += S.t[r * ld + k] * p[k];
            S.tp[r] = s;
        }
        if (m0 == 0 && threadIdx.x >= blockDim.x - 32) beside();
        __syncthreads();
        for (int i = threadIdx.x; i < rows * n; i += blockDim.x) {
            const int r = (int)(((uint32_t)i * recip) >> 20), k = i - r * n;
            double* x = &S.t[r * ld + k];
            const double w = (*x * S.tp[r] * is4 - S.p2[k]) * S.iS[r];
            *reinterpret_cast<float*>(x) = __fmul_rn((float)w, S.loss[r]);
        }
        __syncthreads();
        if (threadIdx.x < n)
            for (int r = 0; r < rows; ++r) acc.add(*reinterpret_cast<const float*>(&S.t[r * ld + threadIdx.x]));
        __syncthreads();
    }
    if (threadIdx.x < n) q[threadIdx.x] = ((double)acc.s - (double)acc.c) / (double)M;
    __syncthreads();
}

}  // namespace hr
