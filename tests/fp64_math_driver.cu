// Test driver of fp64_math.cuh: one function over arrays (the power's plan from b[0]: p,
// negative for L).
//   in  file: int32 op, n; float64 a[n], b[n]
//   out file: float64 x[n], y[n] (y: the second result, where the function has one)
#include <cmath>
#include <cstdio>
#include <vector>

#include "fp64_math.cuh"

__global__ void run(int op, int n, const double* a, const double* b, double* x, double* y, tp::RootPow rp) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double u = 0.0, v = 0.0;
    if (op == 0) u = tp::rcp64(a[i]), v = 1.0 / a[i];
    if (op == 1) u = tp::div64(a[i], b[i], tp::rcp64(b[i])), v = a[i] / b[i];
    if (op == 2) u = tp::sqrt64(a[i], &v);
    if (op == 3) u = tp::third64(a[i]), v = a[i] / 3.0;
    if (op == 4) u = tp::root_pow(a[i], rp, &v);
    if (op == 5) u = pow(a[i], -rp.a), v = rp.a;
    x[i] = u;
    y[i] = v;
}

int main(int argc, char** argv) {
    if (argc != 3) return 2;
    FILE* f = std::fopen(argv[1], "rb");
    int hdr[2];
    if (!f || std::fread(hdr, 4, 2, f) != 2) return 2;
    const size_t n = hdr[1];
    std::vector<double> h(2 * n);
    if (std::fread(h.data(), 8, 2 * n, f) != 2 * n) return 2;
    std::fclose(f);
    double* d = nullptr;
    if (cudaMalloc(&d, 32 * n) != cudaSuccess ||
        cudaMemcpy(d, h.data(), 16 * n, cudaMemcpyHostToDevice) != cudaSuccess)
        return 3;
    run<<<(unsigned)((n + 127) / 128), 128>>>(hdr[0], (int)n, d, d + n, d + 2 * n, d + 3 * n,
                                            tp::root_plan(std::fabs(h[n]), h[n] < 0.0));
    if (cudaGetLastError() != cudaSuccess ||
        cudaMemcpy(h.data(), d + 2 * n, 16 * n, cudaMemcpyDeviceToHost) != cudaSuccess)
        return 3;
    f = std::fopen(argv[2], "wb");
    if (!f || std::fwrite(h.data(), 8, 2 * n, f) != 2 * n) return 2;
    std::fclose(f);
    return 0;
}
