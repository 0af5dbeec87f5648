// The FP64 block inverse of the CFD line kernel (fac_inv) against one division and four products, bit for bit, over
// 2^18 blocks of ordinary entries and blocks whose determinant overflows or is zero: prints "differ K".  Built
// and run on the GPU by tests/test_gpu_line_precision.py.
#include "../paper_2006_07583_gb300/csrc/adi_factored.cu"
#include <cstdio>

__global__ void check(int *differ) {
    unsigned long long s = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x + 1;
    auto next = [&] {  // a linear congruential generator (Knuth); values in (-4, 4)
        s = s * 6364136223846793005ULL + 1442695040888963407ULL;
        return ((double)(s >> 11) * 0x1p-53 - 0.5) * 8.0;
    };
    int n = 0;
    for (int i = 0; i < 4; ++i) {
        double S[2][2], R[2][2];
        const double scale = i == 2 ? 0x1p600 : 1.0;
        for (int p = 0; p < 2; ++p)
            for (int q = 0; q < 2; ++q) S[p][q] = scale * next();
        if (i == 3) { S[1][0] = S[0][0]; S[1][1] = S[0][1]; }
        adi::fac_inv<double, 2>(S, R);
        const double id = 1.0 / (S[0][0] * S[1][1] - S[0][1] * S[1][0]);
        const double W[2][2] = {{S[1][1] * id, -S[0][1] * id}, {-S[1][0] * id, S[0][0] * id}};
        for (int p = 0; p < 2; ++p)
            for (int q = 0; q < 2; ++q) n += !(R[p][q] == W[p][q] || (isnan(R[p][q]) && isnan(W[p][q])));
    }
    if (n) atomicAdd(differ, n);
}

int main() {
    int *d, h = -1;
    if (cudaMalloc(&d, sizeof(h)) != cudaSuccess || cudaMemset(d, 0, sizeof(h)) != cudaSuccess) return 1;
    check<<<256, 256>>>(d);
    if (cudaMemcpy(&h, d, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    printf("differ %d\n", h);
    return 0;
}
