// Test program for the FP64 helpers of md_kernels.cuh: reads n doubles from
// argv[1], evaluates rcp_newton(x) and cut_float(x) (as a double) on the GPU and
// writes the two results per value to argv[2].  Built and run by
// tests/test_ds_arithmetic.py.
#include <cstdio>
#include <vector>

#include "md_kernels.cuh"

__global__ void k_fp64(const double *in, double *out, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n)
        return;
    out[2 * i] = mdk::rcp_newton(in[i]);
    out[2 * i + 1] = (double)mdk::cut_float(in[i]);
}

int main(int argc, char **argv)
{
    if (argc != 3)
        return 2;
    FILE *f = fopen(argv[1], "rb");
    if (!f)
        return 3;
    int n = 0;
    if (fread(&n, sizeof n, 1, f) != 1 || n <= 0)
        return 4;
    std::vector<double> h(n), o(2 * (size_t)n);
    if (fread(h.data(), sizeof(double), n, f) != (size_t)n)
        return 5;
    fclose(f);
    double *din = nullptr, *dout = nullptr;
    if (cudaMalloc(&din, sizeof(double) * n) != cudaSuccess || cudaMalloc(&dout, sizeof(double) * 2 * n) != cudaSuccess)
        return 6;
    cudaMemcpy(din, h.data(), sizeof(double) * n, cudaMemcpyHostToDevice);
    k_fp64<<<(n + 255) / 256, 256>>>(din, dout, n);
    if (cudaMemcpy(o.data(), dout, sizeof(double) * 2 * n, cudaMemcpyDeviceToHost) != cudaSuccess)
        return 7;
    cudaFree(din);
    cudaFree(dout);
    FILE *g = fopen(argv[2], "wb");
    if (!g || fwrite(o.data(), sizeof(double), o.size(), g) != o.size())
        return 8;
    fclose(g);
    return 0;
}
