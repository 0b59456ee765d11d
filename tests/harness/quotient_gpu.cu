// GPU harness of the lattice kernel's reciprocal and quotient
// (vlb_lattice_body.cuh): for FP32 and FP64, the largest error in units of the
// result's last place over a = 1, b = every FP32 number of [0.5, 2) (FP64: the
// same with random low bits), and over pseudo-random a, b of 2^-40 .. 2^40.
#include <cmath>
#include <cstdio>
#include <vector>

#include "vlb_lattice_body.cuh"

template <class C>
__global__ void evaluate(const C* a, const C* b, C* r, C* q, int n) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    r[k] = vlb::reciprocal(b[k]);
    q[k] = vlb::quotient(a[k], b[k]);
  }
}

template <class C>
static double ulps(C got, long double exact) {
  const C e = (C)exact;
  const C next = std::nextafter(std::fabs(e), (C)INFINITY);
  return (double)(std::fabs((long double)got - exact) / ((long double)next - (long double)std::fabs(e)));
}

template <class C>
static int run(const char* name) {
  unsigned long long s = 88172645463325252ull;
  auto rnd = [&]() { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s; };
  auto unit = [&]() { return (double)(rnd() >> 11) * 0x1p-53; };
  std::vector<C> a, b;
  for (unsigned bits = 0x3f000000u; bits < 0x40000000u; bits += 7) {  // 0.5 .. 2
    float f;
    __builtin_memcpy(&f, &bits, 4);
    a.push_back((C)1);
    b.push_back((C)(sizeof(C) == 8 ? (double)f * (1.0 + 0x1p-24 * unit()) : f));
  }
  for (int k = 0; k < 2000000; ++k) {
    a.push_back((C)std::ldexp(1.0 + unit(), (int)(rnd() % 81) - 40));
    b.push_back((C)std::ldexp(rnd() & 1 ? 1.0 + unit() : -1.0 - unit(), (int)(rnd() % 81) - 40));
  }
  const int n = (int)a.size();
  std::vector<C> r(n), q(n);
  C *da, *db, *dr, *dq;
  if (cudaMalloc(&da, n * sizeof(C)) || cudaMalloc(&db, n * sizeof(C)) || cudaMalloc(&dr, n * sizeof(C)) ||
      cudaMalloc(&dq, n * sizeof(C)))
    return 1;
  cudaMemcpy(da, a.data(), n * sizeof(C), cudaMemcpyHostToDevice);
  cudaMemcpy(db, b.data(), n * sizeof(C), cudaMemcpyHostToDevice);
  evaluate<C><<<304, 256>>>(da, db, dr, dq, n);
  cudaMemcpy(r.data(), dr, n * sizeof(C), cudaMemcpyDeviceToHost);
  if (cudaMemcpy(q.data(), dq, n * sizeof(C), cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
  double er = 0.0, eq = 0.0;
  for (int k = 0; k < n; ++k) {
    er = std::fmax(er, ulps(r[k], 1.0L / (long double)b[k]));
    eq = std::fmax(eq, ulps(q[k], (long double)a[k] / (long double)b[k]));
  }
  std::printf("%s %.6f %.6f\n", name, er, eq);
  return 0;
}

int main() { return run<float>("fp32") || run<double>("fp64"); }
