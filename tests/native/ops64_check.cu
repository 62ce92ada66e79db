// Compares the FP64 division and square root of ops64.cuh with the compiler's
// on the GPU: random mantissas over a range of scales, operands beside powers
// of two and exact quotients and squares, zeros, subnormals, infinities.
// Prints the number of operands tried and of results that differ (both NaN
// counts as equal).
#include <stdio.h>

#include "ops64.cuh"

using namespace swadj::d64;

__device__ unsigned long long mix(unsigned long long x) {   // splitmix64 (Steele et al. 2014)
    x += 0x9e3779b97f4a7c15ULL;
    x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ULL;
    x = (x ^ (x >> 27)) * 0x94d049bb133111ebULL;
    return x ^ (x >> 31);
}

// mode 0: any mantissa; 1: few bits; 2: all ones but few; 3: any bit pattern
__device__ double draw(unsigned long long r, int mode) {
    const unsigned long long e = 1023 - 300 + (r >> 52) % 600;
    unsigned long long m = mix(r) & 0xfffffffffffffULL;
    if (mode == 1) m &= 0xfULL << (r % 49);
    if (mode == 2) m |= 0xfffffffffffffULL << (r % 49);
    if (mode == 3) return __longlong_as_double((long long)mix(r + 7));
    m &= 0xfffffffffffffULL;
    return __longlong_as_double((long long)((e << 52) | m | (mix(r + 3) & 1ULL) << 63));
}

__device__ bool same(double a, double b) { return a == b || (a != a && b != b); }

__global__ void check(unsigned long long n, unsigned long long *bad) {
    unsigned long long nb = 0;
    for (unsigned long long k = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; k < n;
         k += (unsigned long long)gridDim.x * blockDim.x) {
        const int mode = (int)(k & 3);
        double a = draw(mix(2 * k), mode), b = draw(mix(2 * k + 1), mode);
        if ((k >> 2) % 16 == 0) {   // a quotient at or beside a representable one
            a = __dmul_rn(a, b);
            if ((k >> 6) & 1) a = __longlong_as_double(__double_as_longlong(a) + 1);
        }
        if ((k >> 2) % 97 == 0) a = 0.0;
        if (!same(div(a, recip(b)), a / b)) nb++;
        if ((k >> 2) % 16 == 0) b = __dmul_rn(b, b);
        if (mode != 3) b = fabs(b);
        if (!same(root(b), sqrt(b))) nb++;
    }
    if (nb) atomicAdd(bad, nb);
}

int main() {
    const unsigned long long n = 1ULL << 27;
    unsigned long long *bad = nullptr, host = 0;
    if (cudaMalloc(&bad, 8) != cudaSuccess) return 2;
    cudaMemset(bad, 0, 8);
    check<<<1216, 128>>>(n, bad);
    if (cudaMemcpy(&host, bad, 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    printf("%llu operands, %llu differ\n", 2 * n, host);
    cudaFree(bad);
    return host == 0 ? 0 : 1;
}
