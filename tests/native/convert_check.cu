// Compares the conversion from double to float of ops64.cuh with the
// hardware's on the GPU, bit for bit: doubles at every float, half way to the
// next and one bit beside either, and of any bit pattern.  Prints the number
// tried and of results that differ (both NaN counts as equal).
#include <stdio.h>

#include "ops64.cuh"

using namespace swadj::d64;

__device__ unsigned long long mix(unsigned long long x) {   // splitmix64 (Steele et al. 2014)
    x += 0x9e3779b97f4a7c15ULL;
    x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ULL;
    x = (x ^ (x >> 27)) * 0x94d049bb133111ebULL;
    return x ^ (x >> 31);
}
__device__ bool same(float a, float b) {
    return __float_as_uint(a) == __float_as_uint(b) || (a != a && b != b);
}

__global__ void check(unsigned long long *bad) {
    unsigned long long nb = 0;
    for (unsigned long long k = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
         k < (1ULL << 32); k += (unsigned long long)gridDim.x * blockDim.x) {
        const float f = __uint_as_float((unsigned)k);
        const double d = (double)f;
        const unsigned long long r = mix(k);
        unsigned long long b = (unsigned long long)__double_as_longlong(d);
        if (r & 1) b += 0x10000000ULL;
        b += (long long)((r >> 1) % 3) - 1;
        const double x = __longlong_as_double((long long)b);
        if (!same(to_float(x), (float)x)) nb++;
        const double y = __longlong_as_double((long long)mix(r));
        if (!same(to_float(y), (float)y)) nb++;
    }
    if (nb) atomicAdd(bad, nb);
}

int main() {
    unsigned long long *bad = nullptr, host = 0;
    if (cudaMalloc(&bad, 8) != cudaSuccess) return 2;
    cudaMemset(bad, 0, 8);
    check<<<1216, 128>>>(bad);
    if (cudaMemcpy(&host, bad, 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    printf("%llu values, %llu differ\n", 2ULL << 32, host);
    cudaFree(bad);
    return host == 0 ? 0 : 1;
}
