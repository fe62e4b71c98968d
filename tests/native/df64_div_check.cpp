// div_markstein against the FP32 division, bit for bit.
#include <cstdio>
#include <cstring>
#include <random>

#include "df64.cuh"

static float from_bits(uint32_t b) {
  float f;
  memcpy(&f, &b, 4);
  return f;
}

int main() {
  std::mt19937_64 rng(7);
  long bad = 0, n = 0;
  auto check = [&](float a, float b) {
    const float q = sdmd::div_markstein(a, b), d = a / b;
    ++n;
    if (memcmp(&q, &d, 4) != 0) ++bad;
  };
  for (long i = 0; i < 20000000; ++i) {
    const uint64_t r = rng();
    const uint32_t ma = (uint32_t)r & 0x807fffffu, mb = (uint32_t)(r >> 32) & 0x007fffffu;
    const uint64_t e = rng();
    const uint32_t eb = 32 + (uint32_t)e % 190;                 // b and 1 / b normal
    const uint32_t ea = 1 + (uint32_t)(e >> 32) % 253;
    const float a = from_bits(ma | (ea << 23)), b = from_bits(mb | (eb << 23));
    const double q = (double)a / (double)b;
    if (q > 3e38 || q < -3e38) continue;
    check(a, b);
  }
  // significands with long runs of ones or zeros, the hard cases of the proof
  for (uint32_t ma = 0; ma < 4096; ++ma)
    for (uint32_t mb = 0; mb < 1024; ++mb) {
      const uint32_t a0 = (ma & 2048) ? 0x7fffffu - (ma & 2047) : (ma & 2047);
      const uint32_t b0 = (mb & 512) ? 0x7fffffu - (mb & 511) : (mb & 511);
      check(from_bits(a0 | (120u << 23)), from_bits(b0 | (127u << 23)));
    }
  check(0.f, 3.f);
  check(1e-40f, 3.f);
  check(1e-30f, 1e10f);
  printf("%ld %ld\n", n, bad);
  return bad != 0;
}
