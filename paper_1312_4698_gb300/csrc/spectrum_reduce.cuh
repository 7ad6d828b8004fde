// Last launch of the Fourier steps: I[k] = scale / n_good times the sum of the partial rows, in a fixed
// order.  A thread of row y adds rows y, y + 8, ..., then the 8 sums are added in order of y: a thread per
// energy walking all rows waits for each in turn (the direct FP64 step of 7350 trajectories, 14 samples,
// 46 energies, 919 rows: 280 -> 216 us).
#pragma once

#include <cstdint>

namespace scivr {
namespace {

constexpr int kRedX = 32, kRedY = 8;

__global__ void __launch_bounds__(kRedX *kRedY) k_reduce_rows(const double *__restrict__ part, int n_rows, int n_E,
                                                              const int64_t *__restrict__ n_good, double scale,
                                                              double *__restrict__ I_out)
{
    __shared__ double sums[kRedY][kRedX];
    const int k = blockIdx.x * kRedX + threadIdx.x;
    double s = 0.0;
    if (k < n_E) {
#pragma unroll 8
        for (int m = threadIdx.y; m < n_rows; m += kRedY) s += part[(int64_t)m * n_E + k];
    }
    sums[threadIdx.y][threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.y != 0 || k >= n_E) return;
    s = 0.0;
#pragma unroll
    for (int y = 0; y < kRedY; ++y) s += sums[y][threadIdx.x];
    I_out[k] = n_good[0] > 0 ? s * (scale / (double)n_good[0]) : 0.0;
}

inline cudaError_t launch_reduce_rows(const double *part, int n_rows, int n_E, const int64_t *n_good, double scale,
                                      double *I_out, cudaStream_t s)
{
    k_reduce_rows<<<(n_E + kRedX - 1) / kRedX, dim3(kRedX, kRedY), 0, s>>>(part, n_rows, n_E, n_good, scale, I_out);
    return cudaGetLastError();
}

}  // namespace
}  // namespace scivr
