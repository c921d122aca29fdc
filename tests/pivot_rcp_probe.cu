// pivot_rcp and bad_pivot over an array, for the test beside it (host arrays of n elements).
#include "pivot.cuh"

static __global__ void probe(const double* x, double* y, int* bad, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    y[i] = ndsi::pivot_rcp(x[i]);
    bad[i] = ndsi::bad_pivot(x[i]) ? 1 : 0;
}

extern "C" int pivot_probe(const double* x, double* y, int* bad, int n) {
    double *dx = nullptr, *dy = nullptr;
    int* db = nullptr;
    cudaError_t e = cudaMalloc(&dx, sizeof(double) * n);
    if (e == cudaSuccess) e = cudaMalloc(&dy, sizeof(double) * n);
    if (e == cudaSuccess) e = cudaMalloc(&db, sizeof(int) * n);
    if (e == cudaSuccess) e = cudaMemcpy(dx, x, sizeof(double) * n, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        probe<<<(n + 255) / 256, 256>>>(dx, dy, db, n);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(y, dy, sizeof(double) * n, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(bad, db, sizeof(int) * n, cudaMemcpyDeviceToHost);
    cudaFree(dx);
    cudaFree(dy);
    cudaFree(db);
    return static_cast<int>(e);
}
