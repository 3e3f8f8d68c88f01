// 64-bit block fixed point for the float64 FFT lines.
//
// sm_103a issues a float64 warp instruction every 16 cycles an SM, 64 times slower than
// float32 or integer ones, so a radix-8 butterfly in float64 (84 operations) takes 1300 cycles
// of the SM.  The same butterfly on 64-bit integers takes 2 instructions an addition and 3 wide
// multiply-adds a product, about 460 instructions at full rate (130 cycles).
//
// A line of N complex values shares one exponent.  Components start below 2^59 and every stage
// is followed by a right shift, rounded, just large enough that the next stage cannot
// overflow.  The bound on the modulus is the smaller of (radix) * (the bound before it) and the
// line's sum of |re| + |im|, which bounds every partial sum of a transform: a line that holds a
// single peak is never shifted, a dense one loses the bits that its sums gain.  The error
// is about one unit of 2^-59 of the bound, float64's is log2(N) roundings of 2^-53 of the values.
//
// Rotations: 2^-62 units (Q62) split in two balanced halves, value = hi 2^32 + lo with lo a
// signed 32-bit number, so that signed wide multiply-adds form every partial product; the lo
// lo product, below one unit of the result, is left out.
#pragma once
#include <stdint.h>

struct fx {
  long long v;
};
__host__ __device__ __forceinline__ fx operator+(fx a, fx b) { return {a.v + b.v}; }
__host__ __device__ __forceinline__ fx operator-(fx a, fx b) { return {a.v - b.v}; }
__host__ __device__ __forceinline__ fx operator-(fx a) { return {-a.v}; }

__host__ __device__ __forceinline__ int fx_lo(long long a) { return (int)a; }
// high half such that a = fx_hi(a) 2^32 + fx_lo(a)
__host__ __device__ __forceinline__ int fx_hi(long long a) { return (int)(a >> 32) + (int)((unsigned)(int)a >> 31); }
__host__ __device__ __forceinline__ long long fx_wide(int a, int b) { return (long long)a * b; }

// a * h for a constant in 2^-63 units (0 < h < 1)
__host__ __device__ __forceinline__ fx fx_scale63(fx a, int hh, int hl) {
  const int ah = fx_hi(a.v), al = fx_lo(a.v);
  const long long mid = (1ll << 30) + fx_wide(al, hh) + fx_wide(ah, hl);
  const long long hi = fx_wide(ah, hh) * 2 + (mid >> 31);
  return {hi};
}
// sqrt(1/2) and sqrt(3)/2 in 2^-63 units
constexpr long long kFxRsqrt2 = 0x5A827999FCEF3242ll;
constexpr long long kFxSqrt3h = 0x6ED9EBA16132A9CFll;
__host__ __device__ __forceinline__ fx fx_mul_rsqrt2(fx a) {
  return fx_scale63(a, (int)((kFxRsqrt2 + 0x80000000ll) >> 32), (int)(unsigned)(kFxRsqrt2 & 0xFFFFFFFFll));
}
__host__ __device__ __forceinline__ fx fx_mul_sqrt3h(fx a) {
  return fx_scale63(a, (int)((kFxSqrt3h + 0x80000000ll) >> 32), (int)(unsigned)(kFxSqrt3h & 0xFFFFFFFFll));
}

// Rotation by w = (c + i d), halves (c_hi, c_lo, d_hi, d_lo) of Q62 numbers; conj: by c - i d.
// Each middle sum stays below 2^62.8 for moduli up to 2^62.5 (Cauchy-Schwarz over the pair).
__host__ __device__ __forceinline__ void fx_rotate(long long ax, long long ay, int4 w, bool conj, long long &ox,
                                                   long long &oy) {
  const int xh = fx_hi(ax), xl = fx_lo(ax), yh = fx_hi(ay), yl = fx_lo(ay);
  const int ph = conj ? w.z : -w.z, pl = conj ? w.w : -w.w;  // the tables hold no -2^31
  const int qh = conj ? -w.z : w.z, ql = conj ? -w.w : w.w;
  const long long half = 1ll << 29;
  const long long mx = half + fx_wide(xl, w.x) + fx_wide(xh, w.y) + fx_wide(yl, ph) + fx_wide(yh, pl);
  const long long my = half + fx_wide(yl, w.x) + fx_wide(yh, w.y) + fx_wide(xl, qh) + fx_wide(xh, ql);
  ox = (fx_wide(xh, w.x) + fx_wide(yh, ph)) * 4 + (mx >> 30);
  oy = (fx_wide(yh, w.x) + fx_wide(xh, qh)) * 4 + (my >> 30);
}

// float64 bits -> integer in units of 2^(E - 1081), E >= the number's biased exponent (1..2046):
// below 2^59 in magnitude, rounded to the nearest
__host__ __device__ __forceinline__ long long fx_from_bits(unsigned long long b, int E) {
  const int ex = (int)(b >> 52) & 2047;
  const long long m = (long long)((b & 0xFFFFFFFFFFFFFull) | (ex ? 1ull << 52 : 0ull)) << 6;
  int d = E - (ex ? ex : 1);
  d = d > 62 ? 62 : d;
  const long long r = (m + ((1ll << d) >> 1)) >> d;
  return (long long)b < 0 ? -r : r;
}

// magnitude of a result outside the normal range, from its 64 leading bits m and biased exponent less
// one be (fx_to_bits): a subnormal number in units of 2^-1074 (a full last unit carries into the
// normal range), zero or infinity.  Kept out of line: it would cost the loops that store the lines
// registers.
#ifdef __CUDA_ARCH__
static __noinline__ __device__
#else
static inline
#endif
unsigned long long fx_end_bits(unsigned long long m, int be) {
  if (be > 0) return 0x7FF0000000000000ull;
  const int sh = 11 - be;
  if (sh > 64) return 0ull;
  const unsigned long long q = sh < 64 ? m >> sh : 0ull;
  const unsigned long long rest = m << (64 - sh);  // against a half, 2^63
  return q + (rest > 0x8000000000000000ull || (rest == 0x8000000000000000ull && (q & 1u)) ? 1ull : 0ull);
}

// v 2^e as float64 bits, rounded once to nearest, ties to even, also into the subnormal range;
// infinity from the midpoint above the largest finite number on
__host__ __device__ __forceinline__ unsigned long long fx_to_bits(long long v, int e) {
  const unsigned long long sign = (unsigned long long)v & 0x8000000000000000ull;
  unsigned long long m = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  if (m == 0) return 0ull;
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)m);
#else
  const int lz = __builtin_clzll(m);
#endif
  m <<= lz;
  const int be = e + 63 - lz + 1022;  // biased exponent less one: the leading bit adds it back
  if ((unsigned)be > 2045u) return sign | fx_end_bits(m, be);
  const unsigned long long q = m >> 11;
  const unsigned long long rest = m & 2047u;
  const unsigned long long up = rest + (q & 1u) > 1024u ? 1ull : 0ull;
  return sign | (((unsigned long long)be << 52) + q + up);
}

// ---- per-line state: shift of stage s in bits 3 s, exponent of the result in bits 48..63 --
constexpr int kFxNonFinite = 32767;
__host__ __device__ __forceinline__ int fx_exp(unsigned long long meta) { return (int)((long long)meta >> 48); }
__host__ __device__ __forceinline__ int fx_shift(unsigned long long meta, int s) { return (int)(meta >> (3 * s)) & 7; }
__host__ __device__ __forceinline__ long long fx_round_shift(long long v, int sh) {
  return (v + ((1ll << sh) >> 1)) >> sh;
}

// Largest admissible bound, in half bits of the modulus: 2^62.5.  The bound of the sum is
// held half a bit lower, since |re| + |im| of a partial sum enters the rotations by 45 degrees.
constexpr int kFxLimit = 125;

// Shifts of a transform whose stages have radices R[0..S-1], run in order S-1..0 (forward) or
// 0..S-1 (inverse), for a line whose components are below 2^59 and whose sum of |re| + |im| is
// below 2^lsum.  E is the biased exponent that the components were aligned to.
__host__ __device__ __forceinline__ unsigned long long fx_schedule(const int *R, int S, bool inverse, int lsum, int E) {
  int bound = 119, sum = 2 * lsum + 1, total = 0;
  unsigned long long meta = 0;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int i = 0; i < S; ++i) {
    const int s = inverse ? i : S - 1 - i;
    const int r = R[s];
    bound += r == 8 ? 6 : (r >= 3 ? 4 : (r == 2 ? 2 : 0));
    if (bound > sum) bound = sum;
    if (i + 1 < S) {
      const int rn = R[inverse ? s + 1 : s - 1];
      int next = bound + (rn == 8 ? 6 : (rn >= 3 ? 4 : (rn == 2 ? 2 : 0)));
      if (next > sum) next = sum;
      const int sh = next > kFxLimit ? (next - kFxLimit + 1) >> 1 : 0;
      meta |= (unsigned long long)sh << (3 * s);
      bound -= 2 * sh;
      sum -= 2 * sh;
      total += sh;
    }
  }
  const int ex = E >= 2047 ? kFxNonFinite : E - 1081 + total;
  return meta | ((unsigned long long)(unsigned short)(short)ex << 48);
}
