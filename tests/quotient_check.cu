// Prints scalar_quotient(a, b) of csrc/sellsolve.cuh and the device's a / b for
// the pairs of a file: count (int64), then count doubles a and count doubles b;
// writes count doubles of each result to the second file.
#include <cstdint>
#include <cstdio>
#include <vector>

#include "sellsolve.cuh"

__global__ void quotients(int64_t n, const double *a, const double *b, double *q, double *d) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    q[i] = gbcg::scalar_quotient(a[i], b[i]);
    d[i] = a[i] / b[i];
}

int main(int argc, char **argv) {
    if (argc < 3) return 2;
    FILE *f = std::fopen(argv[1], "rb");
    int64_t n = 0;
    if (!f || std::fread(&n, 8, 1, f) != 1 || n < 1) return 3;
    std::vector<double> v(2 * (size_t)n);
    if (std::fread(v.data(), 8, v.size(), f) != v.size()) return 4;
    std::fclose(f);
    double *in = nullptr, *out = nullptr;
    if (cudaMalloc(&in, 8 * v.size()) != cudaSuccess || cudaMalloc(&out, 8 * v.size()) != cudaSuccess) return 5;
    if (cudaMemcpy(in, v.data(), 8 * v.size(), cudaMemcpyHostToDevice) != cudaSuccess) return 6;
    quotients<<<(unsigned)((n + 255) / 256), 256>>>(n, in, in + n, out, out + n);
    if (cudaMemcpy(v.data(), out, 8 * v.size(), cudaMemcpyDeviceToHost) != cudaSuccess) return 7;
    f = std::fopen(argv[2], "wb");
    if (!f || std::fwrite(v.data(), 8, v.size(), f) != v.size()) return 8;
    std::fclose(f);
    cudaFree(in);
    cudaFree(out);
    return 0;
}
