// GPU harness of the lattice kernel's reciprocal and quotient
// (vlb_lattice_body.cuh) against the language's correctly rounded division, bit
// by bit: in FP32 every divisor of [1, 2) (quotients of a random dividend), in
// both types pseudo-random operands over the exponents 2^-60 .. 2^60, and in
// FP64 over 2^-500 .. 2^500.  Prints the number of results that differ.
#include <cstdio>
#include <vector>

#include "vlb_lattice_body.cuh"

__device__ __forceinline__ unsigned long long mix(unsigned long long x) {  // SplitMix64
  x += 0x9e3779b97f4a7c15ull;
  x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
  x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
  return x ^ (x >> 31);
}
// A number of random sign and mantissa with an exponent of -range .. range.
template <class C>
__device__ C number(unsigned long long r, int range) {
  const C m = C(1) + C(r >> 11) * C(1.0 / 9007199254740992.0);
  const int e = (int)(mix(r) % (2 * range + 1)) - range;
  return ldexp(r & 1 ? -m : m, e);
}
template <class C>
__global__ void count(int n, int range, bool every, unsigned long long* differ) {
  unsigned long long d = 0;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    const C a = number<C>(mix(2 * (unsigned long long)k), range);
    const C b = every ? C(__uint_as_float(0x3f800000u + (unsigned)k)) : number<C>(mix(2 * (unsigned long long)k + 1), range);
    d += vlb::reciprocal(b) != C(1) / b;
    d += vlb::quotient(a, b) != a / b;
    d += vlb::quotient(b, b) != C(1);
  }
  if (d) atomicAdd(differ, d);
}

int main() {
  unsigned long long* differ;
  if (cudaMallocManaged(&differ, sizeof(*differ)) != cudaSuccess) return 1;
  *differ = 0;
  count<float><<<608, 256>>>(1 << 23, 20, true, differ);
  count<float><<<608, 256>>>(1 << 26, 60, false, differ);
  count<double><<<608, 256>>>(1 << 24, 60, false, differ);
  count<double><<<608, 256>>>(1 << 24, 500, false, differ);
  if (cudaDeviceSynchronize() != cudaSuccess) return 1;
  std::printf("%llu\n", *differ);
  return 0;
}
