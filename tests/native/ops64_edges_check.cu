// Compares the FP64 division and square root of ops64.cuh with the compiler's
// on the GPU, bit for bit (the sign of a zero too; any NaN equals any other),
// where the integer path hands over to the compiler's operation: quotients
// about the smallest normal number and about the largest, operands at either
// end of the normal numbers, subnormal operands, zeros of both signs,
// infinities and NaN.  Prints the number tried and of results that differ.
#include <stdio.h>

#include "ops64.cuh"

using namespace swadj::d64;

__device__ unsigned long long mix(unsigned long long x) {   // splitmix64 (Steele et al. 2014)
    x += 0x9e3779b97f4a7c15ULL;
    x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ULL;
    x = (x ^ (x >> 27)) * 0x94d049bb133111ebULL;
    return x ^ (x >> 31);
}

// exponent field e (0: subnormal or zero, 2047: infinity or NaN), random sign
// and mantissa, some mantissas of few bits or none
__device__ double make(int e, unsigned long long r) {
    unsigned long long m = mix(r) & 0xfffffffffffffULL;
    if ((r & 7) == 0) m = 0;
    if ((r & 7) == 1) m &= 0xfULL << ((r >> 8) % 49);
    if ((r & 7) == 2) m = 0xfffffffffffffULL - (m & 3);
    return __longlong_as_double((long long)((unsigned long long)e << 52 | m |
                                            (mix(r + 1) & 1) << 63));
}
__device__ int clip(int e) { return e < 0 ? 0 : e > 2047 ? 2047 : e; }

__device__ bool same(double a, double b) {
    return __double_as_longlong(a) == __double_as_longlong(b) || (a != a && b != b);
}

__global__ void check(unsigned long long n, unsigned long long *bad) {
    unsigned long long nb = 0;
    for (unsigned long long k = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; k < n;
         k += (unsigned long long)gridDim.x * blockDim.x) {
        const unsigned long long r = mix(k);
        const int any = (int)((r >> 8) % 2048), off = (int)((r >> 20) % 9) - 4;
        const int end = (r >> 24) & 1 ? 2047 - (int)((r >> 25) % 4) : (int)((r >> 25) % 4);
        int ea = any, eb = (int)((r >> 32) % 2048);
        switch (k % 6) {
            case 0: ea = clip(eb - 1022 + off); break;   // about the smallest normal quotient
            case 1: ea = clip(eb + 1023 + off); break;   // about the largest
            case 2: ea = end; break;
            case 3: eb = end; break;
            case 4: ea = 0; break;
            case 5: eb = 0; break;
        }
        double a = make(ea, mix(r)), b = make(eb, mix(r + 5));
        if (k % 11 == 0) a = (r >> 40) & 1 ? -0.0 : 0.0;
        if (k % 13 == 0) b = (r >> 41) & 1 ? -0.0 : 0.0;
        if (!same(div(a, recip(b)), a / b)) nb++;
        const double x = make(end, r);
        if (!same(root(x), sqrt(x))) nb++;
        if (!same(root(b), sqrt(b))) nb++;
    }
    if (nb) atomicAdd(bad, nb);
}

int main() {
    const unsigned long long n = 1ULL << 26;
    unsigned long long *bad = nullptr, host = 0;
    if (cudaMalloc(&bad, 8) != cudaSuccess) return 2;
    cudaMemset(bad, 0, 8);
    check<<<1216, 128>>>(n, bad);
    if (cudaMemcpy(&host, bad, 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    printf("%llu operands, %llu differ\n", 3 * n, host);
    cudaFree(bad);
    return host == 0 ? 0 : 1;
}
