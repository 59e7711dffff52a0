// rsqrt_f64 (csrc/nb_rsqrt.cuh) of every double of a file, written to another:
// rsqrt_f64_check in out. Built and called by tests/test_gpu_rsqrt.py.
#include <cstdio>
#include <vector>

#include <cuda_runtime.h>

#include "nb_rsqrt.cuh"

__global__ void rsqrt_kernel(const double *x, double *y, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = nb::rsqrt_f64(x[i]);
}

int main(int argc, char **argv)
{
    if (argc != 3) return 2;
    std::vector<double> v;
    FILE *f = fopen(argv[1], "rb");
    if (!f) return 2;
    for (double x; fread(&x, sizeof x, 1, f) == 1;) v.push_back(x);
    fclose(f);
    const int n = (int)v.size();
    const size_t bytes = n * sizeof(double);
    double *x = nullptr, *y = nullptr;
    if (n < 1 || cudaMalloc(&x, bytes) != cudaSuccess || cudaMalloc(&y, bytes) != cudaSuccess) return 3;
    if (cudaMemcpy(x, v.data(), bytes, cudaMemcpyHostToDevice) != cudaSuccess) return 3;
    rsqrt_kernel<<<(n + 255) / 256, 256>>>(x, y, n);
    if (cudaMemcpy(v.data(), y, bytes, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
    f = fopen(argv[2], "wb");
    if (!f || fwrite(v.data(), sizeof(double), n, f) != (size_t)n || fclose(f) != 0) return 2;
    cudaFree(x);
    cudaFree(y);
    return 0;
}
