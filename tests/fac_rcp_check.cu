// The FP64 line kernels' reciprocal against CUDA's 1 / x on the GPU: prints "worst K", the largest
// difference in units in the last place over 2^20 values x = +-m 2^e, m in [1, 2), e in [-60, 60].  Built and
// run by tests/test_gpu_tile_edges.py.
#include "../paper_2006_07583_gb300/csrc/adi_factored.cu"
#include <cstdio>

__global__ void check(long long *worst) {
    unsigned long long s = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x + 1;
    long long w = 0;
    for (int i = 0; i < 16; ++i) {
        s = s * 6364136223846793005ULL + 1442695040888963407ULL;  // a linear congruential generator (Knuth)
        const unsigned long long e = 1023 - 60 + (s >> 33) % 121, sign = (s >> 62) & 1;
        const double x = __longlong_as_double((long long)((sign << 63) | (e << 52) | ((s * 2862933555777941757ULL) >> 12)));
        const long long a = __double_as_longlong(adi::fac_rcp(x)), b = __double_as_longlong(1.0 / x);
        const long long d = a > b ? a - b : b - a;
        w = d > w ? d : w;
    }
    atomicMax((unsigned long long *)worst, (unsigned long long)w);
}

int main() {
    long long *d, h = -1;
    if (cudaMalloc(&d, sizeof(h)) != cudaSuccess || cudaMemset(d, 0, sizeof(h)) != cudaSuccess) return 1;
    check<<<256, 256>>>(d);
    if (cudaMemcpy(&h, d, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    printf("worst %lld\n", h);
    return 0;
}
