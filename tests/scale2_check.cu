// scale2_check.cu -- PrecF64::scale2 (kg_arith.cuh) against the multiplication it stands for, bit for
// bit, on a table of doubles given as bit patterns on standard input and on random bit patterns.
// Input: lines "<hex bits of x> <exponent of p2>".  Output: one line per mismatch, then
// "checked <n> mismatches <m> nonzero <k>", k the results that are not zero.
#include <cstdio>
#include <cstring>
#include <vector>

#include "kg_arith.cuh"

__global__ void k_scale(const unsigned long long* x, const int* e, unsigned long long* got, unsigned long long* want, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double v = __longlong_as_double((long long)x[i]), p2 = ldexp(1.0, e[i]);
    got[i] = (unsigned long long)__double_as_longlong(kg::PrecF64::scale2(v, p2));
    want[i] = (unsigned long long)__double_as_longlong(__dmul_rn(v, p2));
}

int main() {
    std::vector<unsigned long long> x;
    std::vector<int> e;
    unsigned long long b;
    int p;
    while (std::scanf("%llx %d", &b, &p) == 2) {
        x.push_back(b);
        e.push_back(p);
    }
    unsigned long long s = 0x9E3779B97F4A7C15ull;   // xorshift64: every exponent field turns up
    for (int i = 0; i < 1 << 20; i++) {
        s ^= s << 13;
        s ^= s >> 7;
        s ^= s << 17;
        x.push_back(s);
        e.push_back(i % 3 == 0 ? -1 : -(12 + i % 16));   // one half, and 1/N^3 of the grids
    }
    const int n = (int)x.size();
    unsigned long long *dx, *dg, *dw;
    int* de;
    if (cudaMalloc((void**)&dx, 8 * (size_t)n) || cudaMalloc((void**)&dg, 8 * (size_t)n) ||
        cudaMalloc((void**)&dw, 8 * (size_t)n) || cudaMalloc((void**)&de, 4 * (size_t)n))
        return 2;
    cudaMemcpy(dx, x.data(), 8 * (size_t)n, cudaMemcpyHostToDevice);
    cudaMemcpy(de, e.data(), 4 * (size_t)n, cudaMemcpyHostToDevice);
    k_scale<<<(n + 255) / 256, 256>>>(dx, de, dg, dw, n);
    std::vector<unsigned long long> got(n), want(n);
    cudaMemcpy(got.data(), dg, 8 * (size_t)n, cudaMemcpyDeviceToHost);
    if (cudaMemcpy(want.data(), dw, 8 * (size_t)n, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
    int bad = 0, nonzero = 0;
    for (int i = 0; i < n; i++) {
        nonzero += (want[i] << 1) != 0;
        if (got[i] != want[i] && bad++ < 20) std::printf("x %016llx 2^%d: %016llx, not %016llx\n", x[i], e[i], got[i], want[i]);
    }
    std::printf("checked %d mismatches %d nonzero %d\n", n, bad, nonzero);
    return 0;
}
