// fp64_ops.cuh's functions beside CUDA's own, one argument (or pair) a thread.
#include "fp64_ops.cuh"

__global__ void k_probe(const double *x, const double *y, double *out, int n)
{
    __shared__ double2 tab[64];
    for (int i = threadIdx.x; i < 64; i += blockDim.x) tab[i] = scivr::kExp2Table[i];
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = scivr::exp_t(x[i], tab);
    out[n + i] = exp(x[i]);
    out[2 * n + i] = scivr::recip(x[i]);
    out[3 * n + i] = 1.0 / x[i];
    // the larger part to a magnitude in [1, 2), as the callers do
    const double a = x[i], b = y[i];
    const int e = max(scivr::mag_key(a), scivr::mag_key(b)) >> 20;
    if (e >= 64 && e <= 1980) {
        const double sc = __hiloint2double((2046 - e) << 20, 0);
        out[4 * n + i] = scivr::arg_normal(a * sc, b * sc, (float)(a * sc), (float)(b * sc));
    } else {
        out[4 * n + i] = atan2(b, a);
    }
    out[5 * n + i] = atan2(b, a);
}

extern "C" int probe(const double *x, const double *y, double *out, int n)
{
    double *d = nullptr;
    cudaError_t e = cudaMalloc(&d, sizeof(double) * 8 * (size_t)n);
    if (e == cudaSuccess) e = cudaMemcpy(d, x, sizeof(double) * n, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(d + n, y, sizeof(double) * n, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        k_probe<<<(n + 127) / 128, 128>>>(d, d + n, d + 2 * n, n);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(out, d + 2 * n, sizeof(double) * 6 * n, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)e;
}
