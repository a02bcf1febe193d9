// grape_filter.cu - Gaussian filtering of the controls and its chain rule
// (App. A of the paper, after Motzoi et al.).
//
// N piecewise-constant controls u[j][k] of length Dt are smoothed into M
// subpixel amplitudes s[n][k] of length dt, the slices the propagation then
// runs on:  s[n][k] = sum_j T_k[n][j] u[j][k]  with the error-function
// transfer matrix  T_k[n][j] = (erf(w0_k (n dt - j Dt)/2) - erf(w0_k (n dt -
// (j+1) Dt)/2)) / 2  (0-based n, j).  The gradient with respect to the
// controls is the transposed sum  g_u[j][k] = sum_n T_k[n][j] g_s[n][k].
//
// T is computed on the fly in FP64 (CUDA's erf).  erf(x) rounds to +-1
// exactly for |x| > 5.93, so an entry is exactly zero once both arguments
// pass kSat = 6.5 on the same side: each output sums only the band of terms
// that can be non-zero, and equals the dense sum up to those exact zeros and
// the order of the terms.
//
// What bounds it: about 60 dependent FP64 operations per erf, at 2 lanes per
// cycle and SM.  One thread per output walked its band one erf after the
// other (66 terms of two erf in the adjoint): 580 us for both maps at 200
// controls x 2000 subpixels x 3 controls.  Now a half-warp (apply) or a warp
// (adjoint) shares an output's band, a lane takes the erf of one edge from
// its neighbour instead of computing it twice (apply), and controls of equal
// bandwidth share the matrix entries: 27 us, launches included.
#include "grape_internal.h"

#include <cmath>

namespace {

constexpr double kSat = 6.5;
constexpr int kEdge = 16;                        // lanes per output of the apply kernel

// number of controls from k on that share control k's bandwidth
__device__ __forceinline__ int equal_run(const FilterArgs &a, int k) {
    int e = k + 1;
    while (e < a.R && a.w0[e] == a.w0[k]) ++e;
    return e - k;
}

// s[n][k]: the half-warp's lane l takes term j0 + l (E of its left edge; the
// right edge's E comes from lane l + 1, so 15 terms per pass)
__global__ void __launch_bounds__(256) filter_apply_kernel(const FilterArgs a) {
    const int lane = threadIdx.x & (kEdge - 1);
    const long long n_ = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / kEdge;
    const int n = (int)min(n_, (long long)a.M - 1);      // (idle half-warps repeat the last output)
    const double t = n * a.dt;
    for (int k = 0; k < a.R;) {
        const int run = equal_run(a, k);
        const double w = a.w0[k];
        const double reach = 2.0 * kSat / w;     // |t - edge| beyond which erf saturates
        const int j0 = max(0, (int)floor((t - reach) / a.Dt) - 1);
        const int j1 = min(a.N - 1, (int)ceil((t + reach) / a.Dt));
        double acc[GRAPE_MAXR];
#pragma unroll
        for (int q = 0; q < GRAPE_MAXR; ++q) acc[q] = 0.0;
        // the two halves of the warp may need different numbers of passes
        const int mine = (j1 - j0 + kEdge - 1) / (kEdge - 1);
        const int passes = max(mine, __shfl_xor_sync(0xffffffffu, mine, kEdge));
        for (int b = 0; b < passes; ++b) {
            const int j = j0 + b * (kEdge - 1) + lane;
            const double e = erf(0.5 * w * (t - j * a.Dt));
            const double right = __shfl_down_sync(0xffffffffu, e, 1, kEdge);
            if (lane == kEdge - 1 || j > j1) continue;
            const double T = 0.5 * (e - right);
#pragma unroll
            for (int q = 0; q < GRAPE_MAXR; ++q)
                if (q < run) acc[q] = fma(T, a.in[(size_t)j * a.R + k + q], acc[q]);
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < GRAPE_MAXR; ++q) {
            if (q >= run) break;
#pragma unroll
            for (int sh = kEdge / 2; sh > 0; sh >>= 1) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], sh, kEdge);
            if (lane == 0 && n_ < a.M) a.out[(size_t)n * a.R + k + q] = acc[q];
        }
        k += run;
    }
}

// g_u[j][k]: the warp's lanes take the subpixels n0 + lane, n0 + 32 + lane, ...
__global__ void __launch_bounds__(128) filter_adjoint_kernel(const FilterArgs a) {
    const int lane = threadIdx.x & 31;
    const long long j_ = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (j_ >= a.N) return;                       // whole warps
    const int j = (int)j_;
    for (int k = 0; k < a.R;) {
        const int run = equal_run(a, k);
        const double w = a.w0[k];
        const double reach = 2.0 * kSat / w;
        const int n0 = max(0, (int)floor((j * a.Dt - reach) / a.dt) - 1);
        const int n1 = min(a.M - 1, (int)ceil(((j + 1) * a.Dt + reach) / a.dt) + 1);
        double acc[GRAPE_MAXR];
#pragma unroll
        for (int q = 0; q < GRAPE_MAXR; ++q) acc[q] = 0.0;
        for (int n = n0 + lane; n <= n1; n += 32) {
            const double t = n * a.dt;
            const double T = 0.5 * (erf(0.5 * w * (t - j * a.Dt)) - erf(0.5 * w * (t - (j + 1) * a.Dt)));
#pragma unroll
            for (int q = 0; q < GRAPE_MAXR; ++q)
                if (q < run) acc[q] = fma(T, a.in[(size_t)n * a.R + k + q], acc[q]);
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < GRAPE_MAXR; ++q) {
            if (q >= run) break;
#pragma unroll
            for (int sh = 16; sh > 0; sh >>= 1) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], sh);
            if (lane == 0) a.out[(size_t)j * a.R + k + q] = acc[q];
        }
        k += run;
    }
}

}  // namespace

cudaError_t grape_launch_filter(const FilterArgs &a, bool adjoint, cudaStream_t s) {
    if (adjoint) {
        const unsigned blocks = (unsigned)(((long long)a.N * 32 + 127) / 128);
        filter_adjoint_kernel<<<blocks, 128, 0, s>>>(a);
    } else {
        const unsigned blocks = (unsigned)(((long long)a.M * kEdge + 255) / 256);
        filter_apply_kernel<<<blocks, 256, 0, s>>>(a);
    }
    return cudaGetLastError();
}
