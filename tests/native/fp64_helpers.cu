// The FP64 helpers against the plain operations: widen, narrow, twice and from_index bit
// for bit (random values, rounding ties, subnormals, the boundaries of FP32, infinities and
// NaN), rcp_series against the division.
#include <cstdio>

#include "pibm_internal.cuh"

using namespace pibm;

namespace {

enum { NARROW, TWICE, WIDEN, INDEX, RCP, KINDS };

__device__ unsigned long long bits(double v) { return (unsigned long long)__double_as_longlong(v); }
__device__ bool same(double a, double b) { return bits(a) == bits(b) || (isnan(a) && isnan(b)); }
__device__ bool same(float a, float b) {
  return __float_as_uint(a) == __float_as_uint(b) || (isnan(a) && isnan(b));
}
__device__ unsigned long long mix(unsigned long long x) {  // splitmix64
  x += 0x9e3779b97f4a7c15ull;
  x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
  x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
  return x ^ (x >> 31);
}

__device__ void one(double v, unsigned long long* bad) {
  if (!same(narrow(v), (float)v)) atomicAdd(&bad[NARROW], 1ull);
  if (!same(twice(v), v + v)) atomicAdd(&bad[TWICE], 1ull);
}
__device__ void one(float v, unsigned long long* bad) {
  if (!same(widen(v), (double)v)) atomicAdd(&bad[WIDEN], 1ull);
}
// 2^-1000 <= d <= 2^1000: next to the division's result at most
__device__ void reciprocal(double d, unsigned long long* bad) {
  const long long off = (long long)(bits(rcp_series(d)) - bits(1.0 / d));
  if (off < -1 || off > 1) atomicAdd(&bad[RCP], 1ull);
}

__global__ void k_random(unsigned long long n, unsigned long long* bad) {
  const unsigned long long step = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
       i += step) {
    const unsigned long long r = mix(i), keep = r & 0x800fffffffffffffull;
    one(__longlong_as_double((long long)r), bad);
    // exponents about FP32's range; then with mantissas on FP32's grid, half a step
    // beyond it (ties) and one bit beside those
    const unsigned long long e = ((r >> 52 & 0x7ff) % 400 + 800) << 52;
    one(__longlong_as_double((long long)(keep | e)), bad);
    const unsigned long long tie = (r >> 8 & 1 ? 0x10000000ull : 0ull) | (r >> 9 & 1);
    one(__longlong_as_double((long long)((keep & ~0x1fffffffull) | e | tie)), bad);
    one(__uint_as_float((unsigned)(r >> 16)), bad);
    const int c = (int)(r & 0x7fffffff) >> (r >> 40 & 31);
    if (!same(from_index(c), (double)c)) atomicAdd(&bad[INDEX], 1ull);
    const unsigned long long mant = r & 0x000fffffffffffffull;
    // densities, masses (1 +- 1/2^k, 2^-23 .. 2^8), and the whole range
    reciprocal(1.0 + (double)(long long)(r << 1) * exp2(-64.0 - (double)(r & 31)), bad);
    reciprocal(__longlong_as_double((long long)(mant | (1000 + (r >> 52 & 31)) << 52)), bad);
    reciprocal(__longlong_as_double((long long)(mant | (24 + (r >> 52 & 2047) % 2000) << 52)), bad);
  }
}

__global__ void k_special(unsigned long long* bad) {
  const unsigned long long v[] = {
      0ull, 1ull, 0x000fffffffffffffull, 0x0010000000000000ull,  // 0, FP64 subnormals
      0x36a0000000000000ull, 0x3690000000000000ull, 0x3690000000000001ull,  // 2^-149, half of it
      0x380fffffffffffffull, 0x3810000000000000ull, 0x3810000000000001ull,  // 2^-126
      0x380fffffdfffffffull, 0x380fffffe0000000ull, 0x380ffffff0000000ull,
      0x47efffffe0000000ull, 0x47efffffefffffffull, 0x47effffff0000000ull,  // FLT_MAX, to infinity
      0x47f0000000000000ull, 0x7fdfffffffffffffull, 0x7fe0000000000000ull,
      0x7fefffffffffffffull, 0x7ff0000000000000ull, 0x7ff8000000000000ull, 0x7ff0000000000001ull};
  for (unsigned long long b : v)
    for (int s = 0; s < 2; ++s)
      one(__longlong_as_double((long long)(b | (unsigned long long)s << 63)), bad);
  const unsigned f[] = {0u,          1u,          0x007fffffu, 0x00800000u, 0x00800001u,
                        0x3f800000u, 0x7f7fffffu, 0x7f800000u, 0x7fc00000u, 0x7f800001u};
  for (unsigned b : f)
    for (int s = 0; s < 2; ++s) one(__uint_as_float(b | (unsigned)s << 31), bad);
  const int c[] = {0, 1, 2, 3, 0x3fffffff, 0x40000000, 0x7ffffffe, 0x7fffffff};
  for (int i : c)
    if (!same(from_index(i), (double)i)) atomicAdd(&bad[INDEX], 1ull);
  for (int e = -1000; e <= 1000; ++e) reciprocal(exp2((double)e), bad);
}

}  // namespace

int main() {
  unsigned long long *dev = nullptr, bad[KINDS] = {};
  cudaMalloc(&dev, sizeof(bad));
  cudaMemset(dev, 0, sizeof(bad));
  k_random<<<608, 256>>>(100000000ull, dev);
  k_special<<<1, 1>>>(dev);
  const cudaError_t e = cudaMemcpy(bad, dev, sizeof(bad), cudaMemcpyDeviceToHost);
  cudaFree(dev);
  printf("%s: narrow %llu twice %llu widen %llu from_index %llu rcp_series %llu\n",
         cudaGetErrorString(e), bad[NARROW], bad[TWICE], bad[WIDEN], bad[INDEX], bad[RCP]);
  for (unsigned long long b : bad)
    if (b || e != cudaSuccess) return 1;
  return 0;
}
