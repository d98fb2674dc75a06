// GPU check of the tracker's double reciprocal (itm_track.cu, rcp_double) against
// the IEEE division 1.0 / a: at most one ulp apart over the range of its float
// start, (2^-100, 2^100), equal outside it. Its error is half an ulp plus less
// than 2^-38 ulp: the start is off by less than 2^-22, the two iterations square
// that to 2^-88, and a step's inner rounding is 2^-53 of a term below 2^-44.
// Prints the largest distance inside in ulps, how many differ outside, and how
// many differ at all in a million.
#include <cstdio>

#include "itm_track.cu"

namespace itm {
namespace {

__device__ double value(unsigned long long i, bool &inside)
{
    // splitmix64 (Steele, Lea, Flood 2014)
    unsigned long long z = i * 0x9e3779b97f4a7c15ull;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    z ^= z >> 31;
    // every exponent in turn; mantissas random, and next to powers of two
    const int e = (int)(i % 240) - 120;
    unsigned long long m = z & 0xfffffffffffffull;
    if (i % 7 == 0) m = z & 0xfull;
    if (i % 7 == 1) m = 0xffffffffffff0ull | (z & 0xfull);
    const double a = __longlong_as_double((long long)(((unsigned long long)(1023 + e) << 52) | m));
    const float f = (float)a;
    inside = f > 0x1p-100f && f < 0x1p100f;
    return a;
}

__global__ void check(unsigned long long n, unsigned long long *out)
{
    const unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    bool inside;
    const double a = value(i, inside);
    const long long x = __double_as_longlong(rcp_double(a)), y = __double_as_longlong(1.0 / a);
    const unsigned long long d = (unsigned long long)(x > y ? x - y : y - x);
    if (inside) atomicMax(&out[0], d);
    else if (d) atomicAdd(&out[1], 1ull);
    if (d) atomicAdd(&out[2], 1ull);
}

}  // namespace
}  // namespace itm

int main()
{
    unsigned long long *out = nullptr, h[3] = {9, 9, 9};
    if (cudaMalloc(&out, sizeof(h)) != cudaSuccess) return 2;
    cudaMemset(out, 0, sizeof(h));
    const unsigned long long n = 1ull << 30;
    itm::check<<<(unsigned)(n / 256), 256>>>(n, out);
    if (cudaDeviceSynchronize() != cudaSuccess) return 3;
    cudaMemcpy(h, out, sizeof(h), cudaMemcpyDeviceToHost);
    printf("%llu %llu %llu\n", h[0], h[1], h[2] * 1000000ull / n);
    return 0;
}
