// Host-side check of the integer float <-> double conversions against the
// language's: exponents and mantissas at the edges of every range, halfway
// cases, and random bits.
#include <cmath>
#include <cstdio>
#include <cstring>

#include "../../paper_0810_5365_gb300/csrc/wd_common.cuh"

using namespace wd;

static unsigned long long bits(double d) { unsigned long long b; memcpy(&b, &d, 8); return b; }
static unsigned bits(float f) { unsigned b; memcpy(&b, &f, 4); return b; }
static bool bad = false;

static void narrow_one(unsigned long long b) {
  cx<double> d[2] = {{1.0, 0.0}, {-2.5, 3.0}};
  memcpy(&d[1].r, &b, 8);
  cx<float> got[2];
  convert(got, d);
  const float want = (float)d[1].r;
  if (std::isnan(want) ? !std::isnan(got[1].r) : bits(want) != bits(got[1].r)) {
    if (!bad) printf("FAIL to float %016llx: %08x, want %08x\n", b, bits(got[1].r), bits(want));
    bad = true;
  }
}
static void widen_one(unsigned b) {
  cx<float> f[2] = {{1.0f, 0.0f}, {-2.5f, 3.0f}};
  memcpy(&f[1].i, &b, 4);
  cx<double> got[2];
  convert(got, f);
  const double want = (double)f[1].i;
  if (std::isnan(want) ? !std::isnan(got[1].i) : bits(want) != bits(got[1].i)) {
    if (!bad) printf("FAIL to double %08x\n", b);
    bad = true;
  }
}

int main() {
  long long n = 0;
  const unsigned long long low[] = {0, 1, 0x0fffffff, 0x10000000, 0x10000001, 0x1fffffff, 0x20000000, 0x2fffffff,
                                    0x30000000, 0x30000001, 0x3fffffffull};
  for (unsigned long long e = 0; e < 2048; e++)
    for (unsigned long long top : {0ull, 1ull, 2ull, 0x3ffffeull, 0x3fffffull, 0x200000ull})
      for (unsigned long long l : low)
        for (unsigned long long s : {0ull, 1ull}) narrow_one(s << 63 | e << 52 | ((top << 30 | l) & 0xfffffffffffffull)), n++;
  for (unsigned b = 0; b < 0xffffffffu - 4099; b += 4099) widen_one(b), n++;
  for (unsigned e = 0; e < 256; e++)
    for (unsigned m : {0u, 1u, 0x400000u, 0x7fffffu})
      for (unsigned s : {0u, 1u}) widen_one(s << 31 | e << 23 | m), n++;
  unsigned long long x = 0x9E3779B97F4A7C15ull;
  for (int k = 0; k < 4000000; k++) {
    x ^= x << 13; x ^= x >> 7; x ^= x << 17;
    narrow_one(x), n++;
    narrow_one((x & 0x8fffffffffffffffull) | 0x3000000000000000ull), n++;  // around 1
  }
  if (bad) return 1;
  printf("OK %lld\n", n);
  return 0;
}
