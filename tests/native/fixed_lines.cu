// Host run of the block fixed-point arithmetic of the float64 FFT lines (fx.cuh, the butterflies of
// fft.cuh) against long double.  Prints one line per check: of the conversions the name, checked values
// and differing ones; of a transformed line "line", length, plan variant, inverse, kind and the
// RMS error over the RMS of the result.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <complex>
#include <random>
#include <vector>

#include "fft.cuh"

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

typedef long double ld;
typedef std::complex<long double> cld;

// radix plans of a line (stage 0 has span 1), as the library numbers them
static std::vector<int> radices(int N, int variant) {
  std::vector<int> R;
  while (variant < 2 && N % 8 == 0) R.push_back(8), N /= 8;
  while (N % 4 == 0) R.push_back(4), N /= 4;
  while (N % 2 == 0) R.push_back(2), N /= 2;
  while (N % 3 == 0) R.push_back(3), N /= 3;
  if (variant & 1) std::reverse(R.begin(), R.end());
  if (R.empty()) R.push_back(1);
  return R;
}

// DFT of x, sign +1 or -1, by its smallest factor
static void reference(const cld *x, int stride, int N, int sign, const std::vector<cld> &w, cld *out) {
  if (N == 1) {
    out[0] = x[0];
    return;
  }
  const int r = N % 2 == 0 ? 2 : 3, M = N / r, n0 = (int)w.size();
  std::vector<cld> sub(N);
  for (int q = 0; q < r; ++q) reference(x + q * stride, stride * r, M, sign, w, sub.data() + q * M);
  for (int k = 0; k < N; ++k) {
    cld s = 0;
    for (int q = 0; q < r; ++q) {
      const cld t = w[(long long)q * k % N * (n0 / N)];
      s += sub[q * M + k % M] * (sign < 0 ? t : std::conj(t));
    }
    out[k] = s;
  }
}

// stage of radix R over span Ns, in place, as fft_stage_r
static void stage(cpx<fx> *x, int N, int R, int Ns, bool inv, const int4 *tw, int sh) {
  for (int q = 0; q < N / R; ++q) {
    const int g = q / Ns, j = q % Ns, e0 = g * Ns * R + j, step = N / (Ns * R);
    cpx<fx> v[8];
    for (int r = 0; r < R; ++r) v[r] = x[e0 + r * Ns];
    if (inv && j)
      for (int r = 1; r < R; ++r) v[r] = cmul_conj(v[r], tw[r * j * step]);
    const int dir = inv ? 1 : -1;
    if (R == 8) dft8(v, dir);
    if (R == 4) dft4(v, dir);
    if (R == 3) dft3(v, dir);
    if (R == 2) dft2(v);
    if (!inv && j)
      for (int r = 1; r < R; ++r) v[r] = cmul(v[r], tw[r * j * step]);
    for (int r = 0; r < R; ++r) {
      v[r].x.v = fx_round_shift(v[r].x.v, sh);
      v[r].y.v = fx_round_shift(v[r].y.v, sh);
      x[e0 + r * Ns] = v[r];
    }
  }
}

static const char *const kKinds[] = {"noise", "constant", "alternating", "wave", "peak", "peak_over_noise", "decades"};

static void lines(int N) {
  const ld pi = acosl(-1.0L);
  std::vector<cld> w(N);
  std::vector<int4> tw(N);
  auto halves = [](ld x, int &hi, int &lo) {  // as the library's tables
    long long q = llrintl(x * 0x1p62L);
    if ((int)q == INT32_MIN) q += 1;
    hi = (int)((q + 0x80000000ll) >> 32);
    lo = (int)q;
  };
  for (int k = 0; k < N; ++k) {
    w[k] = cld(cosl(2 * pi * k / N), -sinl(2 * pi * k / N));
    halves(w[k].real(), tw[k].x, tw[k].y);
    halves(w[k].imag(), tw[k].z, tw[k].w);
  }
  std::mt19937_64 g(N);
  std::normal_distribution<double> nd;
  const double top = 1.0 - 0x1p-53;  // largest mantissa: components just below 2^59
  for (int kind = 0; kind < 7; ++kind)
    for (int inv = 0; inv < 2; ++inv) {
      std::vector<cld> in(N), ref(N);
      const int k0 = 1 + (int)(g() % N);
      for (int i = 0; i < N; ++i) {
        double a = nd(g), b = nd(g);
        if (kind == 1) a = b = top;
        if (kind == 2) a = b = i & 1 ? -top : top;
        if (kind == 3) {
          const cld u = w[(long long)k0 * i % N] * cld(M_SQRT1_2, M_SQRT1_2);
          a = (double)u.real();
          b = (double)u.imag();
        }
        if (kind == 4) a = i == N / 3 ? 0.7e-7 : 0.0, b = 0.0;
        if (kind == 5) a = i == N / 3 ? top : 1e-3 * a, b *= 1e-3;
        if (kind == 6) a *= pow(10.0, -15.0 * (double)(g() >> 11) * 0x1p-53), b *= 1e-9;
        in[i] = cld(a, b);
      }
      reference(in.data(), 1, N, inv ? 1 : -1, w, ref.data());
      ld norm = 0;
      for (const cld &z : ref) norm += std::norm(z);
      for (int variant = 0; variant < 4; ++variant) {
        const std::vector<int> R = radices(N, variant);
        if (variant > 0 && R == radices(N, variant & 2 ? variant - 2 : 0)) continue;
        const int S = (int)R.size();
        std::vector<int> Ns(S), rev(N);
        for (int s = 0, n = 1; s < S; n *= R[s++]) Ns[s] = n;
        for (int p = 0; p < N; ++p) {  // digit reversal: position -> index
          int idx = 0, mul = 1, len = N, rest = p;
          for (int s = S - 1; s >= 0; --s) {
            len /= R[s];
            idx += rest / len * mul;
            rest %= len;
            mul *= R[s];
          }
          rev[p] = idx;
        }
        int E = 1;
        for (const cld &z : in)
          for (double c : {(double)z.real(), (double)z.imag()}) E = std::max(E, (int)(to_bits(c) >> 52) & 2047);
        std::vector<cpx<fx>> f(N);
        unsigned long long sum = 0;
        for (int p = 0; p < N; ++p) {
          const cld z = inv ? in[rev[p]] : in[p];
          f[p].x.v = fx_from_bits(to_bits((double)z.real()), E);
          f[p].y.v = fx_from_bits(to_bits((double)z.imag()), E);
          sum += (unsigned long long)(llabs(f[p].x.v) + llabs(f[p].y.v)) >> 16;
        }
        const int lsum = 80 - __builtin_clzll(sum + N);
        const unsigned long long meta = fx_schedule(R.data(), S, inv, lsum, E);
        for (int i = 0; i < S; ++i) {
          const int s = inv ? i : S - 1 - i;
          stage(f.data(), N, R[s], Ns[s], inv, tw.data(), fx_shift(meta, s));
        }
        ld err = 0;
        for (int p = 0; p < N; ++p) {
          const cld got(from_bits(fx_to_bits(f[p].x.v, fx_exp(meta))), from_bits(fx_to_bits(f[p].y.v, fx_exp(meta))));
          err += std::norm(got - ref[inv ? p : rev[p]]);
        }
        printf("line %d %d %d %s %.3Le\n", N, variant, inv, kKinds[kind], norm > 0 ? sqrtl(err / norm) : err);
      }
    }
}

// the compile-time plan is variant 0
static void plans() {
  const int ct[] = {48, 64, 96, 128, 192, 256, 384, 512, 768, 1024};
  long long bad = 0;
  for (int N : ct) {
    const StagePlan p = stage_plan(N);
    bad += std::vector<int>(p.R, p.R + p.S) != radices(N, 0);
  }
  printf("plans %d %lld\n", 10, bad);
}

int main() {
  integers_to_float64();
  float64_to_integers();
  plans();
  for (int N = 2; N <= 4096; ++N) {
    int rest = N;
    while (rest % 2 == 0) rest /= 2;
    while (rest % 3 == 0) rest /= 3;
    if (rest == 1) lines(N);
  }
  return 0;
}
