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
// bandwidth share the matrix entries: 27 us, launches included.  Where there
// are outputs enough to fill the chip and their bands are short, idle lanes
// would cost what they save, and fewer lanes share an output (`lanes` below).
#include "grape_internal.h"

#include <algorithm>
#include <cmath>
#include <initializer_list>

namespace {

constexpr double kSat = 6.5;

// number of controls from k on that share control k's bandwidth
__device__ __forceinline__ int equal_run(const FilterArgs &a, int k) {
    int e = k + 1;
    while (e < a.R && a.w0[e] == a.w0[k]) ++e;
    return e - k;
}

// s[n][k]: lane l of the output's group of kEdge takes term j0 + l (E of its
// left edge; the right edge's E comes from lane l + 1, so kEdge - 1 terms per
// pass); a lane by itself walks the edges
template <int kEdge>
__global__ void __launch_bounds__(256) filter_apply_kernel(const FilterArgs a) {
    const int lane = threadIdx.x & (kEdge - 1);
    const long long n_ = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / kEdge;
    const int n = (int)min(n_, (long long)a.M - 1);      // (idle groups repeat the last output)
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
        if constexpr (kEdge == 1) {
            double e = erf(0.5 * w * (t - j0 * a.Dt));
            for (int j = j0; j <= j1; ++j) {
                const double right = erf(0.5 * w * (t - (j + 1) * a.Dt)), T = 0.5 * (e - right);
#pragma unroll
                for (int q = 0; q < GRAPE_MAXR; ++q)
                    if (q < run) acc[q] = fma(T, a.in[(size_t)j * a.R + k + q], acc[q]);
                e = right;
            }
        } else {
            // the groups of the warp may need different numbers of passes
            int passes = (j1 - j0 + kEdge - 1) / (kEdge - 1);
#pragma unroll
            for (int sh = kEdge; sh < 32; sh *= 2) passes = max(passes, __shfl_xor_sync(0xffffffffu, passes, sh));
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

// g_u[j][k]: the lanes of the output's group of G take the subpixels n0 + lane,
// n0 + G + lane, ...
template <int G>
__global__ void __launch_bounds__(128) filter_adjoint_kernel(const FilterArgs a) {
    const int lane = threadIdx.x & (G - 1);
    const long long j_ = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / G;
    const int j = (int)min(j_, (long long)a.N - 1);      // (idle groups repeat the last output)
    for (int k = 0; k < a.R;) {
        const int run = equal_run(a, k);
        const double w = a.w0[k];
        const double reach = 2.0 * kSat / w;
        const int n0 = max(0, (int)floor((j * a.Dt - reach) / a.dt) - 1);
        const int n1 = min(a.M - 1, (int)ceil(((j + 1) * a.Dt + reach) / a.dt) + 1);
        double acc[GRAPE_MAXR];
#pragma unroll
        for (int q = 0; q < GRAPE_MAXR; ++q) acc[q] = 0.0;
        for (int n = n0 + lane; n <= n1; n += G) {
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
            for (int sh = G / 2; sh > 0; sh >>= 1) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], sh, G);
            if (lane == 0 && j_ < a.N) a.out[(size_t)j * a.R + k + q] = acc[q];
        }
        k += run;
    }
}

// Lanes per output.  A pass of a group is one chain of FP64 latency while there
// are at most 2.5 warps per SM, and the pipe's time for its lanes, idle ones
// included, beyond; so a launch costs passes(G) max(2.5, outputs G / (32 x 152
// SMs)).  The widest group is the cheapest for few outputs and long bands; a
// narrower one is taken where it costs less than `gain` of the widest (a wide
// group reads its terms together, so a predicted third is worth nothing:
// 80 000 subpixels to 20 000 controls in bands of 41, 0.300 ms on 32 lanes, 0.319
// on one).  Measured, widest group against the rule, one control, 10^5 outputs:
// apply, bands of 4 terms, 0.286 -> 0.073 ms (16 -> 1 lane); adjoint, bands of 6,
// 0.853 -> 0.149 ms (32 -> 1; one thread per output and an erf per edge and
// control before the groups: 0.097 and 0.140 ms, with eight controls 0.654 and
// 0.950 against 0.073 and 0.150).
int lanes(const FilterArgs &a, bool adjoint, std::initializer_list<int> widths, double gain) {
    const double n_out = adjoint ? a.N : a.M;
    double first = 0.0, best = 0.0;
    int g = 0;
    for (const int w : widths) {
        double passes = 0.0;
        for (int k = 0; k < a.R; ++k) {
            if (k > 0 && a.w0[k] == a.w0[k - 1]) continue;
            const double reach = 2.0 * kSat / a.w0[k];
            const double terms = adjoint ? std::min((double)a.M, std::ceil((a.Dt + 2.0 * reach) / a.dt) + 4.0)
                                         : std::min((double)a.N, std::ceil(2.0 * reach / a.Dt) + 3.0);
            passes += !adjoint && w == 1 ? terms + 1.0 : std::ceil(terms / (adjoint ? w : w - 1));
        }
        const double cost = passes * std::max(2.5, n_out * w / (32.0 * 152.0));
        if (g == 0) first = best = cost, g = w;
        else if (cost < gain * first && cost <= best) best = cost, g = w;   // (a tie: no idle lanes)
    }
    return g;
}

template <int G>
void launch_apply(const FilterArgs &a, cudaStream_t s) {
    filter_apply_kernel<G><<<(unsigned)(((long long)a.M * G + 255) / 256), 256, 0, s>>>(a);
}
template <int G>
void launch_adjoint(const FilterArgs &a, cudaStream_t s) {
    filter_adjoint_kernel<G><<<(unsigned)(((long long)a.N * G + 127) / 128), 128, 0, s>>>(a);
}

}  // namespace

cudaError_t grape_launch_filter(const FilterArgs &a, bool adjoint, cudaStream_t s) {
    if (adjoint) {
        switch (lanes(a, true, {32, 16, 8, 4, 2, 1}, 0.63)) {
            case 32: launch_adjoint<32>(a, s); break;
            case 16: launch_adjoint<16>(a, s); break;
            case 8: launch_adjoint<8>(a, s); break;
            case 4: launch_adjoint<4>(a, s); break;
            case 2: launch_adjoint<2>(a, s); break;
            default: launch_adjoint<1>(a, s);
        }
    } else {
        switch (lanes(a, false, {16, 8, 4, 1}, 0.75)) {
            case 16: launch_apply<16>(a, s); break;
            case 8: launch_apply<8>(a, s); break;
            case 4: launch_apply<4>(a, s); break;
            default: launch_apply<1>(a, s);
        }
    }
    return cudaGetLastError();
}
