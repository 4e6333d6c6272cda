// Host program for tests/test_direction_f32.py: draws attempts (random words,
// points at the unit circle, points near the origin) and prints, for each
// kind, how many there were, how many the integer form left to FP64, and how
// many it answered otherwise than the FP64 formula rounded to FP32.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <random>

#include "k_device.cuh"

int main() {
  std::mt19937_64 r(20240607);
  for (int kind = 0; kind < 4; ++kind) {
    const long n = 4000000;
    long open = 0, wrong = 0;
    for (long i = 0; i < n; ++i) {
      uint64_t a = r(), b = r();
      if (kind == 1) {          // within a few units of the circle v1^2 + v2^2 = 1
        const double v1 = 2.0 * ((double)(r() >> 11) * 0x1p-53) - 1.0, v2 = std::sqrt(1.0 - v1 * v1);
        a = (uint64_t)((int64_t)std::ldexp(v1, 52) + (1ll << 52)) << 11;
        b = (uint64_t)((int64_t)std::ldexp(v2, 52) - 8000 + (int64_t)(r() % 16001) + (1ll << 52)) << 11;
      } else if (kind == 2) {   // near the origin, down to it
        a = (uint64_t)((1ll << 52) + (int64_t)(r() % (1ull << (r() % 40)))) << 11;
        b = (uint64_t)((1ll << 52) - (int64_t)(r() % (1ull << (r() % 40)))) << 11;
      } else if (kind == 3) {   // the ends of the range
        a = r() % 2 ? r() % 8192 : ~(r() % 8192);
        b = (uint64_t)((1ll << 52) + (int64_t)(r() % 4096) - 2048) << 11;
      }
      float v1, v2, s;
      const int ok = crash::iso_attempt_f32((uint32_t)a, (uint32_t)(a >> 32), (uint32_t)b, (uint32_t)(b >> 32), v1, v2, s);
      if (ok < 0) { ++open; continue; }
      volatile double u1 = 2.0 * ((double)(a >> 11) * 0x1p-53) - 1.0, u2 = 2.0 * ((double)(b >> 11) * 0x1p-53) - 1.0;
      volatile double p = u1 * u1, q = u2 * u2;
      const volatile double S = p + q;
      const int want = S < 1.0 && S != 0.0;
      if (ok != want || (ok && ((float)u1 != v1 || (float)u2 != v2 || (float)S != s))) ++wrong;
    }
    std::printf("%d %ld %ld %ld\n", kind, n, open, wrong);
  }
  return 0;
}
