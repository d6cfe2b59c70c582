// The sums of squares of csrc/gf_squares.cuh over the rows of a host array, in the screening copies' way:
// a warp a row, up to 32 values a lane between two flushes.
#include "gf_squares.cuh"

static __global__ void k_rows(const float *x, long long n, int d, double *out) {
    const int lane = threadIdx.x & 31;
    const long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= n) return;
    SquareSum sum;
    for (int j0 = 0; j0 < d; j0 += 1024) {
        for (int j = j0 + lane; j < min(d, j0 + 1024); j += 32) sum.add(x[i * d + j]);
        sum.flush();
    }
    const double total = sum.warp_total();
    if (lane == 0) out[i] = total;
}

extern "C" int square_sums(const float *x, long long n, int d, double *out) {
    float *dx = nullptr;
    double *dout = nullptr;
    cudaError_t e = cudaMalloc(&dx, (size_t)n * d * 4);
    if (e == cudaSuccess) e = cudaMalloc(&dout, (size_t)n * 8);
    if (e == cudaSuccess) e = cudaMemcpy(dx, x, (size_t)n * d * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        k_rows<<<(unsigned)((n + 7) / 8), 256>>>(dx, n, d, dout);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(out, dout, (size_t)n * 8, cudaMemcpyDeviceToHost);
    cudaFree(dx);
    cudaFree(dout);
    return (int)e;
}
