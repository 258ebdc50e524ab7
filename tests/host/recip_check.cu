// Newton's reciprocal (csrc/body.cuh) against the division, over mantissas at random and
// at both ends, every exponent on either side of the line from which the
// division itself is used, and all that is not a normal number.  Prints OK if no
// result is more than one unit in the last place from 1 / p.
#include <cstdint>
#include <cstdio>
#include <vector>

#include "body.cuh"

__global__ void k_check(const double* __restrict__ p, int n, int* __restrict__ far, int* __restrict__ where) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double a = fast_recip(p[i]), b = 1.0 / p[i];
    const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
    const bool same = x == y || (a != a && b != b) || (x - y <= 1 && y - x <= 1);
    if (!same) {
        atomicAdd(far, 1);
        atomicMax(where, i);
    }
}

int main() {
    std::vector<double> p;
    uint64_t s = 0x9E3779B97F4A7C15ull;
    auto next = [&] {                                  // splitmix64
        uint64_t z = (s += 0x9E3779B97F4A7C15ull);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return z ^ (z >> 31);
    };
    auto add = [&](uint64_t e, uint64_t m) {
        for (uint64_t sign : {0ull, 1ull}) {
            const uint64_t b = sign << 63 | e << 52 | (m & 0xFFFFFFFFFFFFFull);
            double d;
            memcpy(&d, &b, sizeof(d));
            p.push_back(d);
        }
    };
    for (uint64_t e = 0; e < 2048; ++e) {
        for (uint64_t m : {0ull, 1ull, 2ull, 0xFFFFFFFFFFFFFull, 0xFFFFFFFFFFFFEull, 0x8000000000000ull, 0x7FFFFFFFFFFFFull})
            add(e, m);
        for (int k = 0; k < 200; ++k) add(e, next());
    }
    for (int k = 0; k < 4000000; ++k) add(1023, next());
    for (uint64_t m = 0; m < (1u << 20); ++m) add(1000, m << 32);          // every leading half, low bits clear and set
    for (uint64_t m = 0; m < (1u << 20); ++m) add(1040, m << 32 | 0xFFFFFFFFull);
    const int n = (int)p.size();
    double* d = nullptr;
    int* out = nullptr;
    int got[2] = {-1, -1};
    if (cudaMalloc(&d, (size_t)n * sizeof(double)) != cudaSuccess || cudaMalloc(&out, 2 * sizeof(int)) != cudaSuccess) return 2;
    cudaMemcpy(d, p.data(), (size_t)n * sizeof(double), cudaMemcpyHostToDevice);
    cudaMemset(out, 0, 2 * sizeof(int));
    k_check<<<(n + 255) / 256, 256>>>(d, n, out, out + 1);
    if (cudaMemcpy(got, out, sizeof(got), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    if (got[0]) {
        std::printf("%d of %d are further than one unit from the division, one of them 1 / %.17g\n", got[0], n, p[got[1]]);
        return 1;
    }
    std::printf("OK\n");
    return 0;
}
