// BiCGStab finalisation (Sec. 3.2): the deterministic sum of per-block partials and the
// scalar updates that follow each apply of an iteration and its vector update.  The same
// device functions serve the single-block finaliser kernels (kernels_pw.cu) and the last
// block of the kernel that produced the partials (fft_passes.cuh, k_kxr), which finalises
// in place of a separate launch.
#pragma once
#include "rve_kern.cuh"

// 128-bit integer sum over the lanes of a warp (modulo 2^128)
__device__ __forceinline__ __int128 warp_add128(__int128 acc) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long lo = __shfl_xor_sync(0xffffffffu, (unsigned long long)acc, o);
    const unsigned long long hi = __shfl_xor_sync(0xffffffffu, (unsigned long long)((unsigned __int128)acc >> 64), o);
    acc = (__int128)((unsigned __int128)acc + (((unsigned __int128)hi << 64) | lo));
  }
  return acc;
}
__device__ __forceinline__ int clz128(unsigned __int128 mag) {
  const unsigned long long top = (unsigned long long)(mag >> 64);
  return top ? __clzll(top) : 64 + __clzll((unsigned long long)mag);
}
// the leading 64 of 128 bits, the rest as a sticky bit (lz leading zeros, below 128)
__device__ __forceinline__ unsigned long long leading128(unsigned __int128 mag, int lz) {
  mag <<= lz;
  return (unsigned long long)(mag >> 64) | ((unsigned long long)mag ? 1ull : 0ull);
}
// Significant bits that a sum of up to 2^20 terms needs where bits below its unit were cut: fewer than
// 2 G + 64 units are lost (one a term, one a lane and batch), a sixteenth of the last place of a
// sum of this many bits.
constexpr int kSumBits = 79;

// The sum of finite terms that cancel below those bits, from a first window on: with a unit 53 bits
// below the last place of the largest term nothing overflows; from there the sum is known to 2 G + 64 units,
// so it fits a window of 128 bits whose unit lies up to 103 bits lower, and what is above the window
// cancels modulo 2^128.  Repeated until the sum has its bits, or the unit is the last place of the
// smallest term, where nothing is cut.  Also rounds results outside the normal range.  Rare, and kept short
// (no unrolling) and out of line: the finalisers are chains of code that run once, and inlined or
// unrolled this costs a 64^3 BiCGStab iteration 3 to 8 us of 108.
template <bool CG>
__device__ __noinline__ double warp_sum_cancelled(const double *p, int G) {
  const int lane = threadIdx.x & 31;
  int emax = 1, emin = 2046;
#pragma unroll 1
  for (int i = lane; i < G; i += 32) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(CG ? __ldcg(p + i) : p[i]);
    const int ex = max((int)(b >> 52) & 2047, 1);
    emax = max(emax, ex);
    if (b << 1) emin = min(emin, ex);
  }
  emax = __reduce_max_sync(0xffffffffu, emax);
  emin = __reduce_min_sync(0xffffffffu, emin);
  int unit = emax - 1075 - 53;
#pragma unroll 1
  for (;;) {
    unsigned __int128 s = 0;
#pragma unroll 1
    for (int i = lane; i < G; i += 32) {
      const unsigned long long b = (unsigned long long)__double_as_longlong(CG ? __ldcg(p + i) : p[i]);
      const int ex = (int)(b >> 52) & 2047;
      const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (ex ? 1ull << 52 : 0ull);
      const int sh = (ex ? ex : 1) - 1075 - unit;
      const unsigned __int128 t =
          sh >= 0 ? (sh < 128 ? (unsigned __int128)m << sh : 0) : (unsigned __int128)(sh > -64 ? m >> -sh : 0ull);
      s += (b >> 63) ? 0 - t : t;
    }
    const __int128 acc = warp_add128((__int128)s);
    const unsigned __int128 mag = (unsigned __int128)(acc < 0 ? -acc : acc);
    const int lz = clz128(mag);
    if (acc == 0 && unit <= emin - 1075) return 0.0;
    if (unit <= emin - 1075 || 128 - lz >= kSumBits) {
      const double r = scalbn(__ull2double_rn(leading128(mag, lz)), 64 - lz + unit);
      return acc < 0 ? -r : r;
    }
    unit = max(unit - (125 - max(128 - lz, 22)), emin - 1075);
  }
}

// Sum of G float64 partials by one warp, to 9/16 of a unit in the last place whatever cancels
// (rounded once where no bit was cut): each value becomes a 128-bit integer in units of 2^-53 ulp of
// the largest exponent seen (53 mantissa bits, 53 below them, room for 2^20 terms above), and
// integers add exactly in any order.  Bits below the unit are cut; if fewer bits of the sum are left
// than that allows, warp_sum_cancelled takes over.  A compensated float64 sum needs five operations
// a value and seven a tree level on a pipe that takes a warp instruction every 16 cycles (the
// block-wide one took 4.2 us a quantity, 33 us of a 512^2 BiCGStab iteration's seven sums); integer
// adds run at full rate, a warp a quantity.  Non-finite values fall back to a float64 sum, which
// propagates them.  CG: the partials were written by other blocks of the running kernel, so they
// are read past L1 (ld.global.cg).
template <bool CG>
__device__ __forceinline__ double warp_sum(const double *p, int G) {
  constexpr int U = 8;  // values per lane in flight
  const int lane = threadIdx.x & 31;
  __int128 acc = 0;
  int E = 1;
  bool finite = true;
  for (int base = 0; base < G; base += 32 * U) {
    unsigned long long b[U];
    int e = 1;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = base + 32 * u + lane;
      b[u] = i < G ? (unsigned long long)__double_as_longlong(CG ? __ldcg(p + i) : p[i]) : 0ull;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) e = max(e, (int)(b[u] >> 52) & 2047);
    e = __reduce_max_sync(0xffffffffu, e);
    finite = finite && e < 2047;
    if (e > E) {
      acc = e - E < 127 ? acc >> (e - E) : 0;
      E = e;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int ex = (int)(b[u] >> 52) & 2047;
      const unsigned long long m = (b[u] & 0xFFFFFFFFFFFFFull) | (ex ? 1ull << 52 : 0ull);
      const int sh = E - (ex ? ex : 1);
      const __int128 t = sh < 106 ? ((__int128)m << 53) >> sh : 0;
      acc += (b[u] >> 63) ? -t : t;
    }
  }
  if (!finite) {
    double s = 0.0;
    for (int i = lane; i < G; i += 32) s += CG ? __ldcg(p + i) : p[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
  }
  acc = warp_add128(acc);
  const unsigned __int128 mag = (unsigned __int128)(acc < 0 ? -acc : acc);
  const int lz = clz128(mag);
  // rounded by integers: a conversion and scalbn are a chain on the float64 pipe.  be: biased exponent less
  // one, as in fx_to_bits; at E <= 54 the unit is at most 2^-1074 and nothing was cut
  const int be = 64 - lz + (E - 1075 - 53) + 63 + 1022;
  if (__builtin_expect((128 - lz < kSumBits && E > 54) || (unsigned)be > 2045u, 0))
    return E == 1 && lz == 128 ? 0.0 : warp_sum_cancelled<CG>(p, G);
  const unsigned long long lead = leading128(mag, lz);
  const unsigned long long q = lead >> 11;
  const unsigned long long b = ((unsigned long long)be << 52) + q + ((lead & 2047u) + (q & 1u) > 1024u ? 1ull : 0ull);
  return __longlong_as_double((long long)(b | (acc < 0 ? 1ull << 63 : 0ull)));
}

// NQ sums of G partials each (quantity q at part + q G), one warp a quantity; every thread of the
// block receives them.
template <int NQ, bool CG>
__device__ __forceinline__ void block_sums(const double *part, int G, double (&out)[NQ]) {
  __shared__ double res[NQ];
  for (int q = threadIdx.x >> 5; q < NQ; q += blockDim.x >> 5) {
    const double s = warp_sum<CG>(part + (size_t)q * G, G);
    if ((threadIdx.x & 31) == 0) res[q] = s;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NQ; ++q) out[q] = res[q];
  __syncthreads();
}

// Last-block detection over the blocks of one group member (nblocks of them): every block
// publishes its partials (the caller wrote them), fences, and counts itself in; the block that
// brings the count to nblocks returns true (uniformly for its threads) and resets the counter
// for the next launch.  The counter starts at 0 (zeroed when the handle is created).
__device__ __forceinline__ bool last_block_arrives(unsigned int *ctr, unsigned int nblocks) {
  __shared__ int last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned int prev = atomicAdd(ctr, 1u);
    last = prev == nblocks - 1 ? 1 : 0;
    if (last) *ctr = 0u;
  }
  __syncthreads();
  return last != 0;
}

// after apply(p -> v): vE = s3 sum(w dphi), alpha = rho / (rhat, v), sE = rE - alpha vE.
// part: G partials of sum w dphi, then G of (rhat, v).
template <bool CG>
__device__ __forceinline__ void fin_alpha(KrylovScalars *ks, const double *part, int G) {
  double sum[2];
  block_sums<2, CG>(part, G, sum);
  const double wdp = sum[0], rv = sum[1];
  if (threadIdx.x == 0) {
    ks->vE = ks->strain ? ks->pE : ks->s3 * wdp;
    const double rvt = rv + ks->rhE * ks->vE;
    if (rvt == 0.0) {
      ks->done = 1;
      ks->status = 2;
      return;
    }
    ks->alpha = ks->rho / rvt;
    ks->sE = ks->rE - ks->alpha * ks->vE;
    ks->alpha_f = (float)ks->alpha;
    ks->sE_f = (float)(ks->sE * ks->escale);
  }
}

// alpha update of a float32 chunk iteration: as fin_alpha, and the pending vector update of
// the previous iteration, which the x-forward pass just applied, is cleared.
template <bool CG>
__device__ __forceinline__ void fin_alpha_clear(KrylovScalars *ks, const double *part, int G) {
  fin_alpha<CG>(ks, part, G);
  if (threadIdx.x == 0) ks->pending = 0;
}

// after apply(s -> t): tE, omega = (t, s) / (t, t); xE, rE updates.
// part: G partials of sum w dphi, G of (t, s), G of (t, t).
template <bool CG>
__device__ __forceinline__ void fin_omega(KrylovScalars *ks, const double *part, int G) {
  double sum[3];
  block_sums<3, CG>(part, G, sum);
  const double wdp = sum[0], ts = sum[1], tt = sum[2];
  if (threadIdx.x == 0) {
    ks->tE = ks->strain ? ks->sE : ks->s3 * wdp;
    const double tst = ts + ks->tE * ks->sE;
    const double ttt = tt + ks->tE * ks->tE;
    ks->omega = ttt > 0.0 ? tst / ttt : 0.0;
    ks->omega_f = (float)ks->omega;
    ks->xE += ks->alpha * ks->pE + ks->omega * ks->sE;
    ks->rE = ks->sE - ks->omega * ks->tE;
  }
}

// after x += alpha p + omega s, r = s - omega t: convergence test and the next iteration's
// beta (rho_{k+1} from the fused dot).  part: G partials of |r|^2, then G of (rhat, r).
template <bool CG>
__device__ __forceinline__ void fin_conv(KrylovScalars *ks, const double *part, int G) {
  double sum[2];
  block_sums<2, CG>(part, G, sum);
  const double rr = sum[0], rhr = sum[1];
  if (threadIdx.x == 0) {
    ks->iters += 1;
    const double rn2 = rr + ks->rE * ks->rE;
    ks->rn2 = rn2;
    if (rn2 <= fmax(ks->tol2 * ks->bn2, ks->atol2)) {
      ks->done = 1;
      ks->status = 0;
      return;
    }
    if (ks->omega == 0.0) {
      ks->done = 1;
      ks->status = 2;
      return;
    }
    if (ks->iters >= ks->maxit) {
      ks->done = 1;
      ks->status = 1;
      return;
    }
    const double rho_new = ks->fault_rho0 ? 0.0 : rhr + ks->rhE * ks->rE;
    if (rho_new == 0.0) {
      ks->done = 1;
      ks->status = 2;
      return;
    }
    ks->beta = (rho_new / ks->rho) * (ks->alpha / ks->omega);
    ks->rho = rho_new;
    ks->pE = ks->rE + ks->beta * (ks->pE - ks->omega * ks->vE);
    ks->beta_f = (float)ks->beta;
    ks->pE_f = (float)(ks->pE * ks->escale);
  }
}

// after apply(s -> t) in a float32 chunk: the omega update of fin_omega and the convergence
// test of fin_conv in one step, before r = s - omega t exists as a vector.  With the field
// dots of this apply's epilogue (part: G partials each of sum w dphi, (t, s), (t, t),
// (rhat, s), (rhat, t), (s, s)) the field parts of |r|^2 and (rhat, r) are
//   |r|^2 = (s, s) - 2 omega (t, s) + omega^2 (t, t),   (rhat, r) = (rhat, s) - omega (rhat, t)
// (the float32 run's convergence threshold is far above their rounding).  The vector update
// is left pending; the next x-forward pass or the chunk's closing k_kx_finish applies it.
template <bool CG>
__device__ __forceinline__ void fin_omega_conv(KrylovScalars *ks, const double *part, int G) {
  double sum[6];
  block_sums<6, CG>(part, G, sum);
  const double wdp = sum[0], ts = sum[1], tt = sum[2], rs = sum[3], rt = sum[4], ss = sum[5];
  if (threadIdx.x == 0) {
    ks->tE = ks->strain ? ks->sE : ks->s3 * wdp;
    const double tst = ts + ks->tE * ks->sE;
    const double ttt = tt + ks->tE * ks->tE;
    const double om = ttt > 0.0 ? tst / ttt : 0.0;
    ks->omega = om;
    ks->omega_f = (float)om;
    ks->xE += ks->alpha * ks->pE + om * ks->sE;
    ks->rE = ks->sE - om * ks->tE;
    ks->pending = 1;
    const double rr = fmax(ss - 2.0 * om * ts + om * om * tt, 0.0);
    const double rhr = rs - om * rt;
    ks->iters += 1;
    const double rn2 = rr + ks->rE * ks->rE;
    ks->rn2 = rn2;
    if (rn2 <= fmax(ks->tol2 * ks->bn2, ks->atol2)) {
      ks->done = 1;
      ks->status = 0;
      return;
    }
    if (om == 0.0) {
      ks->done = 1;
      ks->status = 2;
      return;
    }
    if (ks->iters >= ks->maxit) {
      ks->done = 1;
      ks->status = 1;
      return;
    }
    const double rho_new = ks->fault_rho0 ? 0.0 : rhr + ks->rhE * ks->rE;
    if (rho_new == 0.0) {
      ks->done = 1;
      ks->status = 2;
      return;
    }
    ks->beta = (rho_new / ks->rho) * (ks->alpha / om);
    ks->rho = rho_new;
    ks->pE = ks->rE + ks->beta * (ks->pE - om * ks->vE);
    ks->beta_f = (float)ks->beta;
    ks->pE_f = (float)(ks->pE * ks->escale);
  }
}

// the update of ApplyArgs::fin by the member's last block
__device__ __forceinline__ void finalise(int fin, KrylovScalars *ks, const double *part, int G) {
  if (fin == 1) fin_alpha<true>(ks, part, G);
  else if (fin == 2) fin_omega<true>(ks, part, G);
  else if (fin == 5) fin_alpha_clear<true>(ks, part, G);
  else fin_omega_conv<true>(ks, part, G);
}
