// Host run of the block fixed-point number conversions (fx.cuh) against long double.
// Prints one line per check: name, checked values, differing ones.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <random>

#include "fx.cuh"

static double from_bits(unsigned long long b) {
  double x;
  memcpy(&x, &b, 8);
  return x;
}
static unsigned long long to_bits(double x) {
  unsigned long long b;
  memcpy(&b, &x, 8);
  return b;
}

// v 2^e over every exponent that a line can carry; a long double holds a 63-bit v exactly, and its
// conversion rounds once, to nearest with ties to even, subnormal results included
static void integers_to_float64() {
  std::mt19937_64 g(1);
  long long n = 0, bad = 0;
  for (int e = -1150; e <= 1024; ++e)
    for (int i = 0; i < 200; ++i) {
      long long v = (long long)(g() >> 1) >> (i % 63);
      if (i >= 100) {  // at and next to a tie of every result width
        const int w = 1 + (int)(g() % 62);
        v = (1ll << w) | (1ll << (g() % w));
        v += (long long)(g() % 3) - 1;
      }
      if (g() & 1) v = -v;
      const double want = (double)ldexpl((long double)v, e);
      n += 1;
      bad += to_bits(want) != fx_to_bits(v, e);
    }
  printf("integers_to_float64 %lld %lld\n", n, bad);
}

// float64 -> integer in units of 2^(E - 1081): exact at E equal to the number's own exponent, else
// rounded to the nearest unit
static void float64_to_integers() {
  std::mt19937_64 g(2);
  long long n = 0, bad = 0;
  for (int ex = 0; ex < 2047; ++ex)
    for (int i = 0; i < 100; ++i) {
      const unsigned long long b = (g() & 0x800FFFFFFFFFFFFFull) | (unsigned long long)ex << 52;
      const int up = i < 10 ? 0 : (int)(g() % 70);
      const int E = (ex ? ex : 1) + up;
      if (E > 2046) continue;
      const long long v = fx_from_bits(b, E);
      const long double x = ldexpl((long double)from_bits(b), 1081 - E);
      n += 1;
      bad += fabsl((long double)v - x) > 0.5L || (v < 0 ? -v : v) >= (1ll << 59) + (up ? 1 : 0);
    }
  printf("float64_to_integers %lld %lld\n", n, bad);
}

int main() {
  integers_to_float64();
  float64_to_integers();
  return 0;
}
