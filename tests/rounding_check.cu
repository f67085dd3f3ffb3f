// sqrt_rn and recip_rn (spfd_internal.cuh) against the correctly rounded
// sqrt() and division, bit for bit, on 2^25 values: random bit patterns,
// values near powers of two, squares and their neighbours, small integers,
// and the special values.  Prints the number of mismatches.
#include <cstdio>

#include "spfd_internal.cuh"

__device__ unsigned long long mix(unsigned long long z) {  // splitmix64
  z += 0x9e3779b97f4a7c15ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

__global__ void check(unsigned long long n, unsigned long long *bad) {
  const unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const unsigned long long r = mix(i);
  double x = __longlong_as_double((long long)r);
  switch (i & 7) {
    case 1: x = 1.0 + (double)(r % 4096) * 0x1p-52; break;
    case 2: x = 2.0 - (double)(r % 4096 + 1) * 0x1p-52; break;
    case 3: x = (double)(r % (1u << 26)); x *= x; break;
    case 4: x = (double)(r % (1u << 26)); x = nextafter(x * x, (r >> 40) & 1 ? 1e300 : 0.0); break;
    case 5: x = (double)(r % 100000); break;
    case 6: x = scalbn(1.0 + (double)(r >> 12) * 0x1p-52, (int)(r % 2098) - 1074); break;
    default: break;
  }
  if (i < 8) {
    const double s[8] = {0.0, -0.0, 1.0 / 0.0, -1.0 / 0.0, 0.0 / 0.0, 4.9e-324, 2.2e-308, 1.7e308};
    x = s[i];
  }
  auto same = [](double a, double b) {
    return __double_as_longlong(a) == __double_as_longlong(b) || (isnan(a) && isnan(b));
  };
  if (!same(spfd::recip_rn(x), 1.0 / x)) atomicAdd(&bad[0], 1ull);
  if (!same(spfd::sqrt_rn(x), sqrt(x))) atomicAdd(&bad[1], 1ull);
}

int main() {
  unsigned long long *bad = nullptr, h[2] = {1, 1};
  const unsigned long long n = 1ull << 25;
  if (cudaMalloc(&bad, sizeof h) != cudaSuccess) return 2;
  cudaMemset(bad, 0, sizeof h);
  check<<<(unsigned)((n + 255) / 256), 256>>>(n, bad);
  if (cudaMemcpy(h, bad, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
  printf("recip %llu sqrt %llu\n", h[0], h[1]);
  return 0;
}
