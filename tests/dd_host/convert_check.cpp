// Host build of rb_dd.cuh: its integer split of a double into a float pair against
// the compiler's conversions, bit for bit; prints the number of values compared and
// of differences.
#include <cstdio>
#include <cstring>
#include <random>

#include "rb_dd.cuh"

static uint32_t fbits(float x) {
  uint32_t u;
  std::memcpy(&u, &x, sizeof(u));
  return u;
}
static long n = 0, bad = 0;
static void check(uint64_t u) {
  double x;
  std::memcpy(&x, &u, sizeof(x));
  const volatile float h = (float)x;
  const volatile float l = (float)(x - (double)h);
  const rb::ffx::dd d = rb::ffx::from_double_int(x);
  const bool nan = x != x, lnan = l != l;  // NaN payloads are not compared
  ++n;
  if (!(nan ? d.h != d.h : fbits(d.h) == fbits(h))) ++bad;
  else if (!(lnan ? d.l != d.l : fbits(d.l) == fbits(l))) ++bad;
}

int main() {
  std::mt19937_64 g(1);
  // every exponent: random mantissas, and the ties and ends of the 29 dropped bits
  const uint64_t low[] = {0, 1, 0x0FFFFFFF, 0x10000000, 0x10000001, 0x1FFFFFFF};
  const uint64_t high[] = {0, 1, 2, 0x3FFFFF, 0x400000, 0x7FFFFE, 0x7FFFFF};
  for (uint64_t e = 0; e < 2048; ++e)
    for (uint64_t s = 0; s < 2; ++s) {
      const uint64_t top = s << 63 | e << 52;
      for (uint64_t h : high)
        for (uint64_t l : low) check(top | h << 29 | l);
      for (int i = 0; i < 200; ++i) check(top | (g() >> 12));
    }
  std::printf("%ld %ld\n", n, bad);
  return 0;
}
