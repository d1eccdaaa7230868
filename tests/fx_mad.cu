// Prints how many of 64 multiply-adds (csrc/fx.cuh, mad_wide) are wrong where the low
// word of the sum is the value of a factor, so that the compiler may hold both in one
// register.
#include <cstdio>

#include "fx.cuh"

using namespace dgmg;

__global__ void k_mad(const int *x, const int *y, long long *out, long long *ref) {
    const int i = threadIdx.x, a = x[i], b = y[i];
    const long long c = (long long)(unsigned)a;
    out[i] = mad_wide(a, b, c);
    out[32 + i] = mad_wide(b, a, c);
    ref[i] = ref[32 + i] = c + (long long)a * b;
}

int main() {
    int *x, *y;
    long long *out, *ref;
    if (cudaMallocManaged(&x, 32 * sizeof(int)) != cudaSuccess || cudaMallocManaged(&y, 32 * sizeof(int)) != cudaSuccess ||
        cudaMallocManaged(&out, 64 * sizeof(long long)) != cudaSuccess ||
        cudaMallocManaged(&ref, 64 * sizeof(long long)) != cudaSuccess)
        return 2;
    for (int i = 0; i < 32; ++i) {
        x[i] = 0x40000001 + 12345 * i;
        y[i] = -0x20000003 + 777 * i;
    }
    k_mad<<<1, 32>>>(x, y, out, ref);
    if (cudaDeviceSynchronize() != cudaSuccess) return 2;
    int bad = 0;
    for (int i = 0; i < 64; ++i) bad += out[i] != ref[i];
    std::printf("%d\n", bad);
    return 0;
}
