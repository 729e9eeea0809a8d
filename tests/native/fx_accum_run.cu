// Host run of the iterate's update (fxaccum.cuh) on pseudo-random sites: per update the
// scale and the 24 FP32 components of the correction, then exponent and integers of x, in
// hexadecimal, for the test that computes the sums exactly.
#include <cstdint>
#include <cstdio>
#include <cstring>

#include "../../paper_1108_2473_gb300/csrc/fxaccum.cuh"

int main() {
  uint64_t r = 0x9E3779B97F4A7C15ull;
  auto rnd = [&]() {
    r ^= r << 13; r ^= r >> 7; r ^= r << 17;
    return r;
  };
  for (int site = 0; site < 300; ++site) {
    long long x[24] = {0};
    int E = 0;
    double scale = 1.0 + (double)(rnd() >> 12) * 0x1p-52;
    if (site % 3 == 1) scale *= 1e-200;
    if (site % 3 == 2) scale *= 1e200;
    for (int n = 0; n < 10; ++n) {
      float e[24];
      for (int k = 0; k < 24; ++k) {
        e[k] = (float)((double)(int64_t)rnd() * 0x1p-63);
        if (rnd() % 4 == 0) e[k] *= 1e-3f;  // (components of other exponents)
        if (rnd() % 16 == 0) e[k] = 0.f;
      }
      if (site % 50 == 7 && n > 0)
        for (int k = 0; k < 24; ++k) e[k] = 0.f;
      E = lqcd::fx_accum_site(e, lqcd::fx_scale(scale), E, x);
      uint64_t w;
      std::memcpy(&w, &scale, 8);
      std::printf("%d %llx", n, (unsigned long long)w);
      for (int k = 0; k < 24; ++k) {
        uint32_t u;
        std::memcpy(&u, &e[k], 4);
        std::printf(" %x", u);
      }
      std::printf(" %d", E);
      for (int k = 0; k < 24; ++k) std::printf(" %lld", x[k]);
      std::printf("\n");
      scale *= site % 2 ? 1e-6 : 0.7;  // as in a refinement, or of like size
    }
  }
  return 0;
}
