// Device program for tests/test_division_gpu.py: counts the quotients and
// reciprocals (k_device.cuh) that differ from the division, and the widened
// FP32 numbers that differ from the conversion, over random significands and
// exponents, operands near 1, divisors whose significands are nearly ones
// alone, zeros, subnormal, infinite and extreme operands.
#include <cstdio>

#include "k_device.cuh"

__device__ unsigned long long mix(unsigned long long x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}
__device__ bool same(double a, double b) {
  return __double_as_longlong(a) == __double_as_longlong(b) || (a != a && b != b);
}

__global__ void probe(unsigned long long* bad, int mode) {
  const unsigned long long id = blockIdx.x * 256ull + threadIdx.x;
  for (int i = 0; i < 1024; ++i) {
    const unsigned long long s = mix(id * 1024 + i), u = mix(s ^ 0x1234567);
    double a = __longlong_as_double((long long)((s >> 12) | 0x3FF0000000000000ull));
    double b = __longlong_as_double((long long)((u >> 12) | 0x3FF0000000000000ull));
    if (mode == 1) {
      a = 1.0 + ldexp(a - 1.0, -(int)(u % 60));
      b = 1.0 + ldexp(b - 1.0, -(int)(s % 60));
    } else if (mode == 2) {
      a = ldexp(a, (int)(u % 400) - 200);
      b = ldexp(b, (int)(s % 400) - 200);
    } else if (mode == 3) {
      b = __longlong_as_double((long long)(0x3FFFFFFFFFFFFFFFull - (u & 63)));
      if (s & 1) a = 1.0;
    } else if (mode == 4) {
      a = __longlong_as_double((long long)s);      // any bits
      b = __longlong_as_double((long long)u);
      if (i % 64 == 0) a = 0.0;
      if (i % 64 == 1) b = 0.0;
    }
    if (!same(crash::quotient(a, b), a / b)) atomicAdd(bad + 2 * mode, 1ull);
    if (!same(crash::reciprocal(b), 1.0 / b)) atomicAdd(bad + 2 * mode + 1, 1ull);
    float f = __uint_as_float((unsigned)s);
    if (i % 4 == 0) f = __uint_as_float((unsigned)s & 0x80FFFFFFu);     // zero, subnormal, smallest normal
    if (!same(crash::wide(f), (double)f)) atomicAdd(bad + 10, 1ull);
  }
}

int main() {
  unsigned long long *d = nullptr, h[11];
  if (cudaMalloc(&d, sizeof h) != cudaSuccess || cudaMemset(d, 0, sizeof h) != cudaSuccess) return 1;
  for (int mode = 0; mode < 5; ++mode) probe<<<512, 256>>>(d, mode);
  if (cudaMemcpy(h, d, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
  for (unsigned long long v : h) std::printf("%llu\n", v);
  return 0;
}
