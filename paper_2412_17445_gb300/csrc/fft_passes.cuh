#pragma once
// FFT pass kernels of the operator apply (Eq. CrackLength_linearization) and the helpers
// they share with the residual passes (Eq. System_CrackLength).
//
// Every pass kernel takes the line length of its own axis as the template parameter NL:
// NL > 0 is a compile-time length, so index arithmetic, loop trip counts and the stage
// sequence fold to constants; NL = 0 reads the length from the runtime plan.  Both run the
// same stage sequence.  Instantiated in kernels_fft.cu (NL = 0, plus the residual kernels)
// and kernels_fft_<N>.cu (one compile-time length each, compiled in parallel).
//
// Layout: real fields are channel-major [ch][z][y][x]; the spectral scratch holds half
// spectra [ch][z][y][kx] with hx = nx/2 + 1 (kx natural order).  In 3D the y-forward pass
// leaves ky in digit-reversed order, which is exactly the input order the y-inverse pass
// needs (see fft.cuh), so no permutation is ever applied to whole fields.
//
// Passes of one apply:
//   2D: x-forward (+prologue) -> y fused (forward, projection / Laplacian, inverse)
//       -> x-inverse (+epilogue)                                      3 kernels
//   3D: x-forward -> y-forward -> z fused -> y-inverse -> x-inverse   5 kernels
// Two real rows are transformed together as one complex row (z = a + i b) and separated
// by Hermitian symmetry, so every FFT in the x passes is a full-length complex FFT.
#include <type_traits>

#include "rve_kern.cuh"
#include "krylov_fin.cuh"

namespace {

constexpr double kInvSqrt2 = 0.70710678118654752440;

__device__ __forceinline__ FDiv make_fdiv(unsigned d) {
  FDiv f;
  f.d = d;
  f.m = d > 1 ? (0xFFFFFFFFu / d) + 1u : 0u;
  return f;
}

// ---- spectral multiply ------------------------------------------------------------------
// Galerkin projection of a Mandel tensor at one frequency (Eq. GFourier, symmetric reading):
//   (G : tau)_ij = (tau n)_i n_j + n_i (tau n)_j - (n . tau . n) n_i n_j,
// with n the unit direction of the rotated scheme's modified frequency (Willot).  In terms of the
// unnormalised direction m and i = 1 / |m|^2, with v = tau m and u = v - (i / 2) (m . v) m:
//   (G : tau)_ij = i (m_i u_j + u_i m_j)
// which needs one reciprocal and no root, and 14 (2D) or 25 (3D) operations a real tensor:
// the float64 column pass has 48 float64 operations a frequency in 2D, 100 with unit vectors.
template <typename T, int D>
struct ProjDir {
  T m[D];      // direction (Mandel shear entries: tau_ij = t / sqrt 2)
  T c[D];      // 2 i scale m
  T half_inv;  // i / 2; everything is 0 where m vanishes
};

template <typename T, int D>
__device__ __forceinline__ void willot_dir(const AxisTab<T> &tb, const int *k, T scale, ProjDir<T, D> &p, T &xi2) {
  T sn[D], cs[D];
  xi2 = 0;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    sn[a] = tb.sn[a][k[a]];
    cs[a] = tb.cs[a][k[a]];
    xi2 += tb.xi2[a][k[a]];
  }
  T nn = 0;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    T v = sn[a];
#pragma unroll
    for (int b = 0; b < D; ++b)
      if (b != a) v *= cs[b];
    p.m[a] = v;
    nn += v * v;
  }
  T inv = 0;
  if (nn > (T)0) {
    if constexpr (sizeof(T) == 8) inv = recip_nr(nn);
    else inv = (T)1 / nn;
  }
  p.half_inv = (T)0.5 * inv;
  const T f = (T)2 * inv * scale;
#pragma unroll
  for (int a = 0; a < D; ++a) p.c[a] = f * p.m[a];
}

template <typename T, int M>
__device__ __forceinline__ void project_mandel(T *t, const ProjDir<T, M == 3 ? 2 : 3> &p) {
  const T r = (T)kInvSqrt2;
  if constexpr (M == 3) {
    const T txy = t[2] * r;
    T u0 = t[0] * p.m[0] + txy * p.m[1];
    T u1 = txy * p.m[0] + t[1] * p.m[1];
    const T s = (p.m[0] * u0 + p.m[1] * u1) * p.half_inv;
    u0 -= s * p.m[0];
    u1 -= s * p.m[1];
    t[0] = p.c[0] * u0;
    t[1] = p.c[1] * u1;
    t[2] = r * (p.c[1] * u0 + p.c[0] * u1);
  } else {
    const T tyz = t[3] * r, txz = t[4] * r, txy = t[5] * r;
    T u0 = t[0] * p.m[0] + txy * p.m[1] + txz * p.m[2];
    T u1 = txy * p.m[0] + t[1] * p.m[1] + tyz * p.m[2];
    T u2 = txz * p.m[0] + tyz * p.m[1] + t[2] * p.m[2];
    const T s = (p.m[0] * u0 + p.m[1] * u1 + p.m[2] * u2) * p.half_inv;
    u0 -= s * p.m[0];
    u1 -= s * p.m[1];
    u2 -= s * p.m[2];
    t[0] = p.c[0] * u0;
    t[1] = p.c[1] * u1;
    t[2] = p.c[2] * u2;
    t[3] = r * (p.c[2] * u1 + p.c[1] * u2);
    t[4] = r * (p.c[2] * u0 + p.c[0] * u2);
    t[5] = r * (p.c[1] * u0 + p.c[0] * u1);
  }
}

// ---- float64 lines in block fixed point (fx.cuh) ----------------------------------------
// Lines lie in shared memory as ((lc Np + smap(e)) << lw) + w (lc < Lc groups of 2^lw adjacent
// lines, Np slots a line); the state of line (lc, w) is meta[(lc << lw) + w], after the lines.
// The float64 lines are replaced in place by integers: one sweep finds each line's largest
// exponent, a second aligns the values to it and sums their magnitudes.  nw / Lc warps share a
// group where there are fewer groups than warps, else a warp takes whole groups.  Starts
// and ends with a barrier.
__device__ __forceinline__ unsigned long long *fx_meta(cpx<double> *sm, int Lc, int lw, int Np) {
  return reinterpret_cast<unsigned long long *>(sm + ((Lc * Np) << lw));
}

template <int NL>
__device__ __forceinline__ void fx_load_lines(cpx<double> *sm, int Lc, int lw, int Np, const FftPlan &pl, bool inverse) {
  __shared__ unsigned long long acc[32][16];
  const int N = NL > 0 ? NL : pl.N;
  unsigned long long *meta = fx_meta(sm, Lc, lw, Np);
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int W = 1 << lw, w = lane & (W - 1);
  // warps per group; one where its lanes take at most four elements of the group each (sharing a group
  // costs three barriers)
  const int spl = Lc < nw && (N << lw) > 128 ? nw / Lc : 1;
  const int step = (32 >> lw) * spl;
  const unsigned long long *raw = reinterpret_cast<const unsigned long long *>(sm);
  longlong2 *out = reinterpret_cast<longlong2 *>(sm);
  __syncthreads();
  const int part = wi % spl;
  for (int lc = wi / spl;; lc += nw / spl) {
    const bool on = lc < Lc;
    if (!on && spl == 1) break;
    const int e0 = (lane >> lw) + part * (32 >> lw);
    const int base = lc * Np;
    unsigned mx = 0;
    if (on) {
#pragma unroll 4
      for (int e = e0; e < N; e += step) {
        const int o = ((base + smap<NL>(e)) << lw) + w;
        const ulonglong2 z = reinterpret_cast<const ulonglong2 *>(raw)[o];
        mx = max(mx, max((unsigned)(z.x >> 32) & 0x7FFFFFFFu, (unsigned)(z.y >> 32) & 0x7FFFFFFFu));
      }
      for (int o = W; o < 32; o <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if (spl > 1) {
      if (on && lane < W) acc[wi][w] = mx;
      __syncthreads();
      if (on)
        for (int k = 0; k < spl; ++k) mx = max(mx, (unsigned)acc[wi - part + k][w]);
    }
    const int E = max((int)(mx >> 20), 1);
    unsigned long long sum = 0;
    if (on) {
#pragma unroll 4
      for (int e = e0; e < N; e += step) {
        const int o = ((base + smap<NL>(e)) << lw) + w;
        const ulonglong2 z = reinterpret_cast<const ulonglong2 *>(raw)[o];
        const long long a = fx_from_bits(z.x, E), b = fx_from_bits(z.y, E);
        out[o] = make_longlong2(a, b);
        sum += (unsigned long long)((a < 0 ? -a : a) + (b < 0 ? -b : b)) >> 16;
      }
      for (int o = W; o < 32; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    }
    if (spl > 1) {
      __syncthreads();  // the maxima have been read
      if (on && lane < W) acc[wi][w] = sum;
      __syncthreads();
      if (on && part == 0)
        for (int k = 1; k < spl; ++k) sum += acc[wi + k][w];
    }
    if (on && part == 0 && lane < W) {
      const int lsum = 80 - __clzll((long long)(sum + N));
      unsigned long long state;
      if constexpr (NL > 0) {
        constexpr StagePlan P = stage_plan(NL);
        state = inverse ? fx_schedule(P.R, P.S, true, lsum, E) : fx_schedule(P.R, P.S, false, lsum, E);
      } else {
        state = fx_schedule(pl.R, pl.S, inverse, lsum, E);
      }
      meta[(lc << lw) + w] = state;
    }
    if (spl > 1) break;  // every group has its warps
  }
  __syncthreads();
}

// one value of a transformed line in type T: of integers scaled by the line's exponent
template <typename T>
__device__ __forceinline__ cpx<T> line_value(cpx<T> z, const unsigned long long *meta, int line) {
  if constexpr (sizeof(T) == 8) {
    const int e = fx_exp(meta[line]);
    if (e == kFxNonFinite) {  // a NaN or an infinity anywhere in a line reaches all of its values
      const T nan = __longlong_as_double(0x7FF8000000000000ll);
      return {nan, nan};
    }
    return {__longlong_as_double((long long)fx_to_bits(__double_as_longlong(z.x), e)),
            __longlong_as_double((long long)fx_to_bits(__double_as_longlong(z.y), e))};
  } else {
    return z;
  }
}

// Transforms of Lc 2^lw lines in shared memory; float64 lines enter as float64 and leave as
// fixed point (read through line_value).
template <typename T, int NL, bool INV, int LW, bool MERGE = false>
__device__ __forceinline__ void fft_lines(cpx<T> *sm, int Lc, int lw, const FftPlan &pl) {
  constexpr bool fixed = sizeof(T) == 8;
  const int Np = line_slots<NL>(pl.Np);
  const unsigned long long *meta = nullptr;
  if constexpr (fixed) {
    fx_load_lines<NL>(sm, Lc, lw, Np, pl, INV);
    meta = fx_meta(sm, Lc, lw, Np);
  } else {
    __syncthreads();
  }
  using V = std::conditional_t<fixed, fx, T>;
  cpx<V> *lines = reinterpret_cast<cpx<V> *>(sm);
  if constexpr (NL > 0) {
    const auto *tw = (const typename FftTypes<V>::Tw *)pl.tw;
    if constexpr (INV && MERGE) {
      // float32 x-inverse pass in 3D: adjacent small stages merged (ct_stage_io).  In 2D the 20
      // registers more cost resident blocks (four 512^2: 72.5 us against 70), the forward passes
      // have none left for it.
      constexpr int S = stage_plan(NL).S;
      auto smr = [&](int lc, int e, int) -> cpx<V> & { return lines[lc * NL + smap<NL>(e)]; };
      auto get = [&](int lc, int e, int w) { return smr(lc, e, w); };
      auto put = [&](int lc, int e, int w, cpx<V> v) { smr(lc, e, w) = v; };
      ct_dit_io<V, NL, S - 1, S>(Lc, 0, tw, get, smr, put);
      __syncthreads();
    } else if constexpr (INV) {
      fft_dit_ct<V, NL, LW>(lines, Lc, lw, tw, meta);
    } else {
      fft_dif_ct<V, NL, LW>(lines, Lc, lw, tw, meta);
    }
  } else {
    // lw > 0: consecutive threads take consecutive lines (contiguous addresses); lw = 0: the
    // lines are Np apart, a multiple of the bank count for power-of-two N, so consecutive
    // threads take consecutive butterflies of one line instead
    const int W = 1 << lw;
    LineLayout ly;
    ly.L = Lc << lw;
    ly.dL = make_fdiv(Lc << lw);
    ly.lw = W;
    ly.dlw = make_fdiv(W);
    ly.lsA = Np << lw;
    ly.lsB = 1;
    ly.es = W;
    ly.line_fastest = lw > 0;
    if constexpr (INV) fft_dit<V>(lines, ly, pl, meta);
    else fft_dif<V>(lines, ly, pl, meta);
  }
}

// ---- x-forward tail: DIF over the packed row pairs, then Hermitian unpack + store -------
// tr = 0: half spectra stored row-major [ch][row][kx] (coalesced along kx);
// tr = 1: stored transposed [ch][kx][row] for the fused 2D column pass (k_col_fused2d).
// With tr the threads walk the digit-reversed positions of each line (conflict-free shared
// reads; the partner N - k of position p lies at a nearly contiguous position) and write
// the two rows of a pair as one 16-byte store.
template <typename T, int NL>
__device__ __forceinline__ void xfwd_tail(cpx<T> *sm, int c, int P, int row0, const Geo &g, const FftPlan &pl,
                          cpx<T> *spec, int tr = 0) {
  const int nx = NL > 0 ? NL : g.nx, hx = nx / 2 + 1, Np = line_slots<NL>(pl.Np);
  fft_lines<T, NL, false, 0>(sm, c * P, 0, pl);
  [[maybe_unused]] const unsigned long long *meta = nullptr;
  if constexpr (sizeof(T) == 8) meta = fx_meta(sm, c * P, 0, Np);
  const int cs = g.rows * hx;
  const FDiv dhx = make_fdiv(hx), dP = make_fdiv(P);
  if (sizeof(T) == 4 && tr) {
    const int totp = c * P * nx;
    const FDiv dnx = make_fdiv(nx);
    for (int i = threadIdx.x; i < totp; i += blockDim.x) {
      const int l = NL > 0 ? i / NL : (int)fdiv(i, dnx);
      const int p = i - l * nx;
      int k;
      if constexpr (NL > 0) k = digit_rev_ct<NL>(p);
      else k = pl.rev[p];
      if (2 * k > nx) continue;
      const int kn = k == 0 ? 0 : nx - k;
      int pn;
      if constexpr (NL > 0) pn = digit_unrev_ct<NL>(kn);
      else pn = pl.unrev[kn];
      const int ch = (int)fdiv(l, dP), pr = l - ch * P;
      const cpx<T> zk = sm[l * Np + smap<NL>(p)];
      const cpx<T> zn = sm[l * Np + smap<NL>(pn)];
      const cpx<T> A = {(zk.x + zn.x) * (T)0.5, (zk.y - zn.y) * (T)0.5};
      const cpx<T> B = {(zk.y + zn.y) * (T)0.5, (zn.x - zk.x) * (T)0.5};
      const int r0 = row0 + 2 * pr;
      cpx<T> *dst = spec + ch * cs + k * g.rows + r0;
      if (r0 + 1 < g.rows) {
        if constexpr (sizeof(T) == 4) {
          *reinterpret_cast<float4 *>(dst) = make_float4(A.x, A.y, B.x, B.y);
        } else {
          dst[0] = A;
          dst[1] = B;
        }
      } else if (r0 < g.rows) {
        dst[0] = A;
      }
    }
    return;
  }
  const int tot = c * P * hx;
  // the positions and values of U entries are read before the first is stored (a store to the
  // scratch would hold back the table reads of the next entry)
  constexpr int U = sizeof(T) == 4 ? 4 : 2;
  for (int base = 0; base < tot; base += U * (int)blockDim.x) {
    cpx<T> zk[U], zn[U];
    int pk[U], pn[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = min(base + u * (int)blockDim.x + (int)threadIdx.x, tot - 1);
      const int l = NL > 0 ? i / (NL / 2 + 1) : (int)fdiv(i, dhx);
      const int k = i - l * hx;
      pk[u] = l * Np + smap<NL>(__ldg(pl.unrev + k));
      pn[u] = l * Np + smap<NL>(__ldg(pl.unrev + (k == 0 ? 0 : nx - k)));
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      zk[u] = sm[pk[u]];
      zn[u] = sm[pn[u]];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = base + u * (int)blockDim.x + (int)threadIdx.x;
      if (i >= tot) break;
      const int l = NL > 0 ? i / (NL / 2 + 1) : (int)fdiv(i, dhx);
      const int k = i - l * hx;
      const int ch = (int)fdiv(l, dP), pr = l - ch * P;
      cpx<T> A, B;
      if constexpr (sizeof(T) == 8) {
        // halves of sums of integers
        const long long kx = __double_as_longlong(zk[u].x) >> 1, ky = __double_as_longlong(zk[u].y) >> 1;
        const long long mx = __double_as_longlong(zn[u].x) >> 1, my = __double_as_longlong(zn[u].y) >> 1;
        A = line_value<T>({__longlong_as_double(kx + mx), __longlong_as_double(ky - my)}, meta, l);
        B = line_value<T>({__longlong_as_double(ky + my), __longlong_as_double(mx - kx)}, meta, l);
      } else {
        A = {(zk[u].x + zn[u].x) * (T)0.5, (zk[u].y - zn[u].y) * (T)0.5};
        B = {(zk[u].y + zn[u].y) * (T)0.5, (zn[u].x - zk[u].x) * (T)0.5};
      }
      const int r0 = row0 + 2 * pr, r1 = r0 + 1;
      if (r0 < g.rows) spec[ch * cs + r0 * hx + k] = A;
      if (r1 < g.rows) spec[ch * cs + r1 * hx + k] = B;
    }
  }
}

// ---- x-inverse head: load row pairs of half spectra, rebuild full lines, DIT inverse ----
template <typename T, int NL, bool MERGE = false>
__device__ __forceinline__ void xinv_head(cpx<T> *sm, int c, int P, int row0, const Geo &g, const FftPlan &pl,
                          const cpx<T> *spec, int tr = 0) {
  const int nx = NL > 0 ? NL : g.nx, hx = nx / 2 + 1, Np = line_slots<NL>(pl.Np);
  const int cs = g.rows * hx;
  const int tot = c * P * hx;
  const FDiv dhx = make_fdiv(hx), dP = make_fdiv(P);
  if (sizeof(T) == 4 && tr) {
    // Z_k = A + iB for k <= nx/2 and Z_{nx-k} = conj(A) + i conj(B), with (A, B) the half-
    // spectrum entries of the row pair at k.  Threads walk the positions p of each line
    // (k = rev(p)); a position with k <= nx/2 loads its entry once and writes both p and the
    // partner position of nx - k.  All loads of a batch of U positions per thread are issued
    // before the first shared-memory write.
    const int totp = c * P * nx;
    const FDiv dnx = make_fdiv(nx);
    constexpr int U = 8;
    for (int base = 0; base < totp; base += U * (int)blockDim.x) {
      cpx<T> qa[U], qb[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = base + u * (int)blockDim.x + (int)threadIdx.x;
        qa[u] = {0, 0};
        qb[u] = {0, 0};
        if (i >= totp) continue;
        const int l = NL > 0 ? i / NL : (int)fdiv(i, dnx);
        const int p = i - l * nx;
        int k;
        if constexpr (NL > 0) k = digit_rev_ct<NL>(p);
        else k = pl.rev[p];
        if (2 * k > nx) continue;
        const int ch = (int)fdiv(l, dP), pr = l - ch * P;
        const int r0 = row0 + 2 * pr;
        const cpx<T> *src = spec + ch * cs + k * g.rows + r0;
        if (r0 + 1 < g.rows) {
          if constexpr (sizeof(T) == 4) {
            const float4 q = *reinterpret_cast<const float4 *>(src);
            qa[u] = {q.x, q.y};
            qb[u] = {q.z, q.w};
          } else {
            qa[u] = src[0];
            qb[u] = src[1];
          }
        } else if (r0 < g.rows) {
          qa[u] = src[0];
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = base + u * (int)blockDim.x + (int)threadIdx.x;
        if (i >= totp) continue;
        const int l = NL > 0 ? i / NL : (int)fdiv(i, dnx);
        const int p = i - l * nx;
        int k;
        if constexpr (NL > 0) k = digit_rev_ct<NL>(p);
        else k = pl.rev[p];
        if (2 * k > nx) continue;
        cpx<T> A = qa[u], B = qb[u];
        if (k == 0 || 2 * k == nx) {
          A.y = 0;
          B.y = 0;
        }
        sm[l * Np + smap<NL>(p)] = cpx<T>{A.x - B.y, A.y + B.x};
        if (k > 0 && 2 * k < nx) {
          int pn;
          if constexpr (NL > 0) pn = digit_unrev_ct<NL>(nx - k);
          else pn = pl.unrev[nx - k];
          sm[l * Np + smap<NL>(pn)] = cpx<T>{A.x + B.y, B.x - A.y};
        }
      }
    }
  }
  // as above, U entries' loads before the first shared-memory write
  constexpr int U = MERGE || NL == 0 ? 4 : 2;
  for (int base = 0; base < (sizeof(T) == 4 && tr ? 0 : tot); base += U * (int)blockDim.x) {
    cpx<T> qa[U], qb[U];
    int pk[U], pn[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = base + u * (int)blockDim.x + (int)threadIdx.x;
      qa[u] = {0, 0};
      qb[u] = {0, 0};
      pk[u] = pn[u] = -1;
      if (i >= tot) continue;
      const int l = NL > 0 ? i / (NL / 2 + 1) : (int)fdiv(i, dhx);
      const int k = i - l * hx;
      const int ch = (int)fdiv(l, dP), pr = l - ch * P;
      const int r0 = row0 + 2 * pr, r1 = r0 + 1;
      if (r0 < g.rows) qa[u] = spec[ch * cs + r0 * hx + k];
      if (r1 < g.rows) qb[u] = spec[ch * cs + r1 * hx + k];
      pk[u] = l * Np + smap<NL>(__ldg(pl.unrev + k));
      if (k > 0 && 2 * k < nx) {
        pn[u] = l * Np + smap<NL>(__ldg(pl.unrev + nx - k));
      } else {
        qa[u].y = 0;
        qb[u].y = 0;
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (pk[u] < 0) continue;
      const cpx<T> A = qa[u], B = qb[u];
      sm[pk[u]] = {A.x - B.y, A.y + B.x};
      if (pn[u] >= 0) sm[pn[u]] = {A.x + B.y, B.x - A.y};
    }
  }
  fft_lines<T, NL, true, 0, MERGE>(sm, c * P, 0, pl);
}

}  // namespace

// =========================== operator apply ==================================================
// Prologue (per voxel): input dq = (d_eps, d_phi, dE) (optionally formed by a fused
// BiCGStab update), d_eps' = d_eps + f dE, d_phi masked on the notch;
//   t      = C' d_eps' + sF d_phi        (channels 0..m-1 of the FFT, row-scaled F1 input)
//   d_phi                                  (channel m of the FFT)
//   pw     = kappa (sF . d_eps') + a' d_phi + notch * dq_phi   (pointwise part of row F2)
//   sum w d_phi                            (constraint row, block partial 0)
// A thread takes the two voxels (x, r0) and (x, r0 + 1) of a row pair: all loads of both are
// issued before either is used, and the pair fills one complex shared-memory slot.
template <typename T, int M>
struct ProIn {
  T q[M + 1];                 // input vector (after the fused update)
  T cc[M * (M + 1) / 2];      // C' upper triangle
  T sF[M];
  T kappa, av, w, notch;
};

template <typename T, int M>
__device__ __forceinline__ void pro_load(const ApplyArgs<T> &a, int n, int v, T beta, T omega, T alpha,
                                         ProIn<T, M> &in, int pm, bool pending) {
  using TI = TanIdx<M>;
#pragma unroll
  for (int k = 0; k <= M; ++k) {
    const int o = k * n + v;
    T val;
    if (pm == 1) {
      val = a.r[o] + beta * (a.x[o] - omega * a.v[o]);
      a.x[o] = val;
    } else if (pm == 5) {
      // the previous iteration's x += alpha p + omega s, r = s - omega t (when pending), then
      // p := r + beta (p - omega v); omega and alpha are still the previous iteration's
      const T p = a.x[o];
      T r;
      if (pending) {
        const T sv = a.s[o];
        r = sv - omega * a.t[o];
        a.xs[o] += alpha * p + omega * sv;
        a.r[o] = r;
      } else {
        r = a.r[o];
      }
      val = r + beta * (p - omega * a.v[o]);
      a.x[o] = val;
    } else if (pm == 2) {
      val = a.r[o] - alpha * a.v[o];
      a.x[o] = val;
    } else {
      val = a.x[o];
    }
    in.q[k] = val;
  }
#pragma unroll
  for (int k = 0; k < TI::NC; ++k) in.cc[k] = a.tan[k * n + v];
#pragma unroll
  for (int k = 0; k < M; ++k) in.sF[k] = a.tan[(TI::SF + k) * n + v];
  in.kappa = a.tan[TI::KAPPA * n + v];
  in.av = a.tan[TI::A * n + v];
  in.w = a.tan[TI::W * n + v];
  in.notch = a.tan[TI::NOTCH * n + v];
}

template <typename T, int M>
__device__ __forceinline__ void pro_compute(const ApplyArgs<T> &a, int n, int v, const T (&fx)[M],
                                            const ProIn<T, M> &in, T (&out)[M + 1], T &wdp) {
  T de[M];
#pragma unroll
  for (int k = 0; k < M; ++k) de[k] = in.q[k] + fx[k];
  const T dpm = in.q[M] * ((T)1 - in.notch);
  T sde = 0;
#pragma unroll
  for (int k = 0; k < M; ++k) sde += in.sF[k] * de[k];
#pragma unroll
  for (int k = 0; k <= M; ++k) out[k] = 0;
  int idx = 0;
#pragma unroll
  for (int i2 = 0; i2 < M; ++i2) {
#pragma unroll
    for (int j2 = i2; j2 < M; ++j2) {
      const T cij = in.cc[idx];
      out[i2] += cij * de[j2];
      if (j2 != i2) out[j2] += cij * de[i2];
      ++idx;
    }
  }
#pragma unroll
  for (int k = 0; k < M; ++k) out[k] += in.sF[k] * dpm;
  out[M] = dpm;
  a.y[M * n + v] = in.kappa * sde + in.av * dpm + in.notch * in.q[M];
  wdp += in.w * dpm;
}

// float32: 64 registers per thread, 1024 resident threads an SM; 2D blocks have 256 or 512 threads
// (row_threads)
template <typename T, int M>
constexpr int kRowThreads = sizeof(T) == 4 && M == 3 ? 512 : 256;
// PC > 0 / MODE >= 0: row pairs per block and prologue mode fixed at compile time (the
// float32 2D passes of the Krylov chunks), so every loop bound and branch folds; PC = 0 /
// MODE = -1 read them from the launch.
template <typename T, int M, int NL, int PC, int MODE>
__global__ void __launch_bounds__(kRowThreads<T, M>, sizeof(T) == 4 ? 1024 / kRowThreads<T, M> : 1) k_xfwd_apply(const __grid_constant__ ApplyGroup<T> grp, FftPlan pl, int P_rt) {
  pdl_begin();
  const ApplyArgs<T> &a = grp.m[blockIdx.y];
  const int P = PC > 0 ? PC : P_rt;
  const int pm = MODE >= 0 ? MODE : a.pro_mode;
  extern __shared__ unsigned char smraw[];
  cpx<T> *sm = reinterpret_cast<cpx<T> *>(smraw);
  if (a.ks && a.ks->done) return;
  const Geo &g = a.g;
  const int c = M + 1, nx = NL > 0 ? NL : g.nx, Np = line_slots<NL>(pl.Np);
  const int n = (int)g.n;
  const int row0 = blockIdx.x * 2 * P;
  const FDiv dnx = make_fdiv(nx);
  T xE;
  if (sizeof(T) == 4 && a.xEf_ptr) xE = (T)*a.xEf_ptr;
  else xE = (T)(*a.xE_ptr * (a.ks ? a.ks->escale : a.e_scale));
  T fx[M];
#pragma unroll
  for (int k = 0; k < M; ++k) fx[k] = a.fM[k] * xE;
  T beta = 0, omega = 0, alpha = 0;
  bool pending = false;
  if (pm == 1) {
    beta = ks_scalar<T>(a.ks->beta, a.ks->beta_f);
    omega = ks_scalar<T>(a.ks->omega, a.ks->omega_f);
  } else if (pm == 5) {
    beta = ks_scalar<T>(a.ks->beta, a.ks->beta_f);
    omega = ks_scalar<T>(a.ks->omega, a.ks->omega_f);
    alpha = ks_scalar<T>(a.ks->alpha, a.ks->alpha_f);
    pending = a.ks->pending != 0;
  } else if (pm == 2) {
    alpha = ks_scalar<T>(a.ks->alpha, a.ks->alpha_f);
  }
  // per-thread and warp sums stay in T (a few dozen terms); the block and grid sums are float64
  T wdp = 0;
  const int tot = P * nx;
  for (int i = threadIdx.x; i < tot; i += blockDim.x) {
    const int l0 = NL > 0 ? i / NL : (int)fdiv(i, dnx), x = i - l0 * nx;
    const int r0 = row0 + 2 * l0;
    const bool ok0 = r0 < g.rows, ok1 = r0 + 1 < g.rows;
    const int v0 = r0 * nx + x, v1 = v0 + nx;
    T out0[M + 1], out1[M + 1];
#pragma unroll
    for (int k = 0; k <= M; ++k) out0[k] = out1[k] = 0;
    if (pm == 4) {
      // projection of the strain channels of x alone (Newton update direction)
#pragma unroll
      for (int k = 0; k < M; ++k) {
        if (ok0) out0[k] = a.x[k * n + v0];
        if (ok1) out1[k] = a.x[k * n + v1];
      }
    } else {
      if constexpr (M == 6) {
        // 3D: 38 operands per voxel; holding both voxels' operands at once spills at the 64
        // registers of four resident blocks, so the two voxels are loaded and used in turn
        ProIn<T, M> in;
        if (ok0) {
          pro_load<T, M>(a, n, v0, beta, omega, alpha, in, pm, pending);
          pro_compute<T, M>(a, n, v0, fx, in, out0, wdp);
        }
        if (ok1) {
          pro_load<T, M>(a, n, v1, beta, omega, alpha, in, pm, pending);
          pro_compute<T, M>(a, n, v1, fx, in, out1, wdp);
        }
      } else {
        ProIn<T, M> in0, in1;
        if (ok0) pro_load<T, M>(a, n, v0, beta, omega, alpha, in0, pm, pending);
        if (ok1) pro_load<T, M>(a, n, v1, beta, omega, alpha, in1, pm, pending);
        if (ok0) pro_compute<T, M>(a, n, v0, fx, in0, out0, wdp);
        if (ok1) pro_compute<T, M>(a, n, v1, fx, in1, out1, wdp);
      }
    }
    const int px = smap<NL>(x);
#pragma unroll
    for (int k = 0; k <= M; ++k) sm[(k * P + l0) * Np + px] = {out0[k], out1[k]};
  }
  const T pv[1] = {wdp};
  block_partials_k<T, 1>(pv, a.part, gridDim.x, blockIdx.x);
  xfwd_tail<T, NL>(sm, c, P, row0, g, pl, a.spec, a.tr);
}

// Epilogue (per voxel): y_eps = projected t (row scaling and 1/n folded in earlier),
// y_phi = pw + b' L d_phi; optional fused BiCGStab dots (block partials 1.. ).  A thread
// takes the two voxels of a row pair (one complex shared-memory slot per channel).
template <typename T, int M>
struct EpiIn {
  T pw, bb;
  T o[M + 1];   // rhat (mode 1) or s (modes 2, 6)
  T o2[M + 1];  // rhat (mode 6)
};

template <typename T, int M>
__device__ __forceinline__ void epi_load(const ApplyArgs<T> &a, int n, int v, EpiIn<T, M> &in, int em) {
  using TI = TanIdx<M>;
  if (em == 3) return;  // projection: strain channels only
  in.pw = a.y[M * n + v];
  in.bb = a.tan[TI::B * n + v];
  if (em == 1) {
#pragma unroll
    for (int k = 0; k <= M; ++k) in.o[k] = a.rhat[k * n + v];
  } else if (em == 2) {
#pragma unroll
    for (int k = 0; k <= M; ++k) in.o[k] = a.s[k * n + v];
  } else if (em == 6) {
#pragma unroll
    for (int k = 0; k <= M; ++k) {
      in.o[k] = a.s[k * n + v];
      in.o2[k] = a.rhat[k * n + v];
    }
  }
}

template <typename T, int M>
__device__ __forceinline__ void epi_compute(const ApplyArgs<T> &a, int n, int v, T (&yv)[M + 1],
                                            const EpiIn<T, M> &in, T (&d)[5], int em) {
  if (em == 3) {
#pragma unroll
    for (int k = 0; k < M; ++k) a.y[k * n + v] = yv[k];
    return;
  }
  yv[M] = in.pw + in.bb * yv[M];
#pragma unroll
  for (int k = 0; k <= M; ++k) a.y[k * n + v] = yv[k];
  if (em == 1) {
#pragma unroll
    for (int k = 0; k <= M; ++k) d[0] += in.o[k] * yv[k];
  } else if (em == 2) {
#pragma unroll
    for (int k = 0; k <= M; ++k) {
      d[0] += yv[k] * in.o[k];
      d[1] += yv[k] * yv[k];
    }
  } else if (em == 6) {
#pragma unroll
    for (int k = 0; k <= M; ++k) {
      d[0] += yv[k] * in.o[k];      // (t, s)
      d[1] += yv[k] * yv[k];        // (t, t)
      d[2] += in.o2[k] * in.o[k];   // (rhat, s)
      d[3] += in.o2[k] * yv[k];     // (rhat, t)
      d[4] += in.o[k] * in.o[k];    // (s, s)
    }
  }
}

template <typename T, int M, int NL, int PC, int MODE>
__global__ void __launch_bounds__(kRowThreads<T, M>, sizeof(T) == 4 ? 1024 / kRowThreads<T, M> : 1) k_xinv_apply(const __grid_constant__ ApplyGroup<T> grp, FftPlan pl, int P_rt) {
  pdl_begin();
  const ApplyArgs<T> &a = grp.m[blockIdx.y];
  const int P = PC > 0 ? PC : P_rt;
  const int em = MODE >= 0 ? MODE : a.epi_mode;
  extern __shared__ unsigned char smraw[];
  cpx<T> *sm = reinterpret_cast<cpx<T> *>(smraw);
  if (a.ks && a.ks->done) return;
  // fin 3, 4: block 0 only forms the E slot of y, from the constraint-row partials of the x-forward
  // pass (an earlier launch), while the others run the pass: the chain of the 128-bit sum takes
  // 4 us, a quarter of the pass at 512^2
  const bool yE_block = a.fin == 3 || a.fin == 4;
  const int G = (int)gridDim.x - (yE_block ? 1 : 0);
  const int blk = (int)blockIdx.x - (yE_block ? 1 : 0);
  if (blk < 0) {
    if (a.fin == 4) {
      if (threadIdx.x == 0) *a.yE = *a.xE_ptr;
    } else if (threadIdx.x < 32) {
      const double sE = warp_sum<false>(a.part, G);
      if (threadIdx.x == 0) *a.yE = sE;
    }
    return;
  }
  const Geo &g = a.g;
  const int c = M + 1, nx = NL > 0 ? NL : g.nx, Np = line_slots<NL>(pl.Np);
  const int n = (int)g.n;
  const int row0 = blk * 2 * P;
  const FDiv dnx = make_fdiv(nx);
  xinv_head<T, NL, sizeof(T) == 4 && M == 6>(sm, c, P, row0, g, pl, a.spec, a.tr);
  [[maybe_unused]] const unsigned long long *meta = nullptr;
  if constexpr (sizeof(T) == 8) meta = fx_meta(sm, c * P, 0, Np);
  T d[5] = {0, 0, 0, 0, 0};  // per-thread and warp sums in T, block and grid sums in float64
  const int tot = P * nx;
  for (int i = threadIdx.x; i < tot; i += blockDim.x) {
    const int l0 = NL > 0 ? i / NL : (int)fdiv(i, dnx), x = i - l0 * nx;
    const int r0 = row0 + 2 * l0;
    const bool ok0 = r0 < g.rows, ok1 = r0 + 1 < g.rows;
    const int v0 = r0 * nx + x, v1 = v0 + nx;
    EpiIn<T, M> in0, in1;
    if (M == 3 || sizeof(T) == 8) {
      if (ok0) epi_load<T, M>(a, n, v0, in0, em);
      if (ok1) epi_load<T, M>(a, n, v1, in1, em);
    }
    const int px = smap<NL>(x);
    T y0[M + 1], y1[M + 1];
#pragma unroll
    for (int k = 0; k <= M; ++k) {
      const cpx<T> z = line_value<T>(sm[(k * P + l0) * Np + px], meta, k * P + l0);
      y0[k] = z.x;
      y1[k] = z.y;
    }
    if (M == 3 || sizeof(T) == 8) {
      if (ok0) epi_compute<T, M>(a, n, v0, y0, in0, d, em);
      if (ok1) epi_compute<T, M>(a, n, v1, y1, in1, d, em);
    } else {
      // 3D float32: one voxel after the other, within the 64 registers of four resident blocks
      if (ok0) {
        epi_load<T, M>(a, n, v0, in0, em);
        epi_compute<T, M>(a, n, v0, y0, in0, d, em);
      }
      if (ok1) {
        epi_load<T, M>(a, n, v1, in0, em);
        epi_compute<T, M>(a, n, v1, y1, in0, d, em);
      }
    }
  }
  if (em == 6) {
    block_partials_k<T, 5>(d, a.part + G, G, blk);
  } else if (em != 0) {
    const T pv[2] = {d[0], d[1]};
    block_partials_k<T, 2>(pv, a.part + G, G, blk);
  }
  if (a.fin == 1 || a.fin == 2 || a.fin == 5 || a.fin == 6) {
    // the member's last block finalises the iteration's scalars (no separate launch)
    if (last_block_arrives(a.arrive, G)) {
      finalise(a.fin, a.ksw, a.part, G);
    }
  }
}

// =========================== column passes (y, z) ============================================

// The spectral multiply on transformed lines in shared memory, in place: projection of the strain
// channels, |xi|^2 on the phase field (float64 lines: fixed point in, float64 out).
template <typename T, int M, int NL>
__device__ __forceinline__ void project_columns(const ColArgs<T> &a, cpx<T> *sm, const unsigned long long *meta, int N,
                                                int Np, int kx0, int other) {
  const int lw = a.lw, W = a.W;
  constexpr int D = (M == 3) ? 2 : 3;
  const int ky_other = (D == 3) ? a.yplan.rev[other] : 0;
  for (int i = threadIdx.x; i < (N << lw); i += blockDim.x) {
    const int p = i >> lw;
    const int w = i & (W - 1);
    if (kx0 + w > a.g.hx - 1) continue;
    int k[3];
    k[0] = kx0 + w;
    if (D == 2) {
      k[1] = a.plan.rev[p];
    } else {
      k[1] = ky_other;
      k[2] = a.plan.rev[p];
    }
    ProjDir<T, D> pd;
    T xi2;
    willot_dir<T, D>(a.tab, k, a.inv_n, pd, xi2);
    const int pp = smap<NL>(p);
    T re[M], im[M];
#pragma unroll
    for (int ch = 0; ch < M; ++ch) {
      const cpx<T> z = line_value<T>(sm[((ch * Np + pp) << lw) + w], meta, (ch << lw) + w);
      re[ch] = z.x;
      im[ch] = z.y;
    }
    project_mandel<T, M>(re, pd);
    project_mandel<T, M>(im, pd);
#pragma unroll
    for (int ch = 0; ch < M; ++ch) sm[((ch * Np + pp) << lw) + w] = {re[ch], im[ch]};
    const cpx<T> zp = line_value<T>(sm[((M * Np + pp) << lw) + w], meta, (M << lw) + w);
    const T sc = xi2 * a.inv_n;
    sm[((M * Np + pp) << lw) + w] = {zp.x * sc, zp.y * sc};
  }
}

// MODE 0: forward only (DIF, result stays digit-reversed along the axis)
// MODE 1: forward, spectral multiply, inverse (the last axis)
// MODE 2: inverse only (input digit-reversed along the axis, DIT)
template <typename T, int M, int MODE, int NL>
__global__ void __launch_bounds__(256) k_col(const __grid_constant__ ColGroup<T> grp) {
  pdl_begin();
  const ColArgs<T> &a = grp.base;
  cpx<T> *const spec = grp.spec[blockIdx.z];
  const KrylovScalars *const ks = grp.ks[blockIdx.z];
  extern __shared__ unsigned char smraw[];
  cpx<T> *sm = reinterpret_cast<cpx<T> *>(smraw);
  if (ks && ks->done) return;
  const Geo &g = a.g;
  const int c = M + 1;
  const int W = a.W, lw = a.lw;
  const int N = NL > 0 ? NL : a.plan.N, Np = line_slots<NL>(a.plan.Np);
  const int kx0 = blockIdx.x * W;
  const int other = blockIdx.y;
  int es_g, base_o;
  if (a.axis == 1) {
    es_g = g.hx;
    base_o = other * g.ny * g.hx;
  } else {
    es_g = g.hx * g.ny;
    base_o = other * g.hx;
  }
  const int cs = g.rows * g.hx;
  const int tot = (c * N) << lw;
  // float32 lines of a compiled length: the first step of the transform reads the scratch into
  // registers and the last one writes it from them (ct_dif_io, ct_dit_io); a 128-point pass
  // goes once through shared memory (four times in mode 1) instead of four (eight) times.
  // 128^3: forward 43 -> 27 us, fused z pass 69 -> 50 us
  if constexpr (sizeof(T) == 4 && NL > 0) {
    constexpr int S = stage_plan(NL).S;
    const cpx<T> *tw = (const cpx<T> *)a.plan.tw;
    cpx<T> *const col = spec + base_o + kx0;
    const int wmax = g.hx - kx0;  // columns of the block within the half spectrum
    auto gld = [&](int lc, int e, int w) -> cpx<T> {
      return w < wmax ? col[lc * cs + e * es_g + w] : cpx<T>{0, 0};
    };
    auto gst = [&](int lc, int e, int w, cpx<T> v) {
      if (w < wmax) col[lc * cs + e * es_g + w] = v;
    };
    auto smr = [&](int lc, int e, int w) -> cpx<T> & { return sm[((lc * NL + smap<NL>(e)) << lw) + w]; };
    auto sget = [&](int lc, int e, int w) { return smr(lc, e, w); };
    auto sput = [&](int lc, int e, int w, cpx<T> v) { smr(lc, e, w) = v; };
    if constexpr (MODE == 0) {
      ct_dif_io<T, NL, S - 1>(c, lw, tw, gld, smr, gst);
    } else if constexpr (MODE == 2) {
      ct_dit_io<T, NL, S - 1, S>(c, lw, tw, gld, smr, gst);
    } else {
      ct_dif_io<T, NL, S - 1>(c, lw, tw, gld, smr, sput);
      __syncthreads();
      project_columns<T, M, NL>(a, sm, nullptr, N, Np, kx0, other);
      __syncthreads();
      ct_dit_io<T, NL, S - 1, S>(c, lw, tw, sget, smr, gst);
    }
    return;
  }
  const FDiv dN = make_fdiv(N);
  // the block's lines are strided in the scratch (one L2 round trip per element): each thread
  // issues KU loads before its first shared-memory store, so they are in flight together
  constexpr int KU = 4;
  for (int base = 0; base < tot; base += KU * (int)blockDim.x) {
    cpx<T> val[KU];
    int slot[KU];
#pragma unroll
    for (int u = 0; u < KU; ++u) {
      const int i = base + u * (int)blockDim.x + (int)threadIdx.x;
      val[u] = {0, 0};
      slot[u] = -1;
      if (i < tot) {
        const int iw = i >> lw;
        const int w = i & (W - 1);
        const int ch = NL > 0 ? iw / NL : (int)fdiv(iw, dN);
        const int e = iw - ch * N;
        if (kx0 + w < g.hx) val[u] = spec[ch * cs + base_o + e * es_g + kx0 + w];
        slot[u] = ((ch * Np + smap<NL>(e)) << lw) + w;
      }
    }
#pragma unroll
    for (int u = 0; u < KU; ++u)
      if (slot[u] >= 0) sm[slot[u]] = val[u];
  }
  // (fft_lines starts with a barrier)
  [[maybe_unused]] const unsigned long long *meta = nullptr;
  if constexpr (sizeof(T) == 8) meta = fx_meta(sm, c, lw, Np);
  if (MODE == 0 || MODE == 1) fft_lines<T, NL, false, -1>(sm, c, lw, a.plan);
  if (MODE == 1) project_columns<T, M, NL>(a, sm, meta, N, Np, kx0, other);
  if (MODE == 1 || MODE == 2) fft_lines<T, NL, true, -1>(sm, c, lw, a.plan);
  for (int i = threadIdx.x; i < tot; i += blockDim.x) {
    const int iw = i >> lw;
    const int w = i & (W - 1);
    const int ch = NL > 0 ? iw / NL : (int)fdiv(iw, dN);
    const int e = iw - ch * N;
    if (kx0 + w < g.hx)
      spec[ch * cs + base_o + e * es_g + kx0 + w] =
          line_value<T>(sm[((ch * Np + smap<NL>(e)) << lw) + w], meta, (ch << lw) + w);
  }
}


// =========================== fused 2D column pass (float32, transposed scratch) =============
// The column (y) pass of the 2D apply on the transposed half spectrum spec[ch][kx][y]:
// every line (ch, kx) is contiguous.  A block takes KC columns (all 4 channels) with
// KC * N / 2 threads; KC is picked by the tile tuner (fewer columns per block give a
// single RVE more blocks, more give each block more work).
//   first DIF stage   global -> registers -> shared        (coalesced line loads)
//   middle DIF stages in shared memory
//   last DIF stage, projection (Eq. GFourier, Willot directions) and |xi|^2 multiply,
//   first DIT stage   three shared-memory phases (butterflies per line, then the projection
//                     per frequency position across the four channels, then butterflies)
//   middle DIT stages in shared memory
//   last DIT stage    shared -> registers -> global        (coalesced line stores)
// The radix of the last DIF / first DIT stage (span 1) is 8 for every compiled N.  Same
// arithmetic as k_col mode 1.
template <int N, int KC>
__global__ void __launch_bounds__(1024) k_col_fused2d(const __grid_constant__ ColGroup<float> grp) {
  pdl_begin();
  const ColArgs<float> &a = grp.base;
  cpx<float> *const spec = grp.spec[blockIdx.y];
  const KrylovScalars *const ks = grp.ks[blockIdx.y];
  extern __shared__ unsigned char smraw[];
  cpx<float> *sm = reinterpret_cast<cpx<float> *>(smraw);
  if (ks && ks->done) return;
  constexpr StagePlan SP = stage_plan(N);
  constexpr int S = SP.S;
  static_assert(S >= 2 && SP.R[0] == 8 && SP.Ns[0] == 1, "fused column pass needs a radix-8 span-1 stage");
  static_assert(KC * N / 2 <= 1024, "at most 1024 threads (N / 2 per column)");
  constexpr int Np = N;  // smap slots
  constexpr int C = 4;             // channels: 3 strain (Mandel) + phase field
  constexpr int RT = SP.R[S - 1], NST = SP.Ns[S - 1];  // outermost stage: span N / RT
  constexpr int NBT = N / RT;
  const Geo &g = a.g;
  const int kx0 = blockIdx.x * KC;
  const int cs = g.hx * N;
  const cpx<float> *tw = (const cpx<float> *)a.plan.tw;
  // line (col, ch) of the block sits at (col * C + ch) * Np in shared memory

  // ---- first DIF stage: global -> registers -> shared --------------------------------------
  for (int b = threadIdx.x; b < KC * C * NBT; b += blockDim.x) {
    const int line = b / NBT, j = b - line * NBT;
    const int col = line / C, ch = line - col * C;
    const bool ok = kx0 + col < g.hx;
    const cpx<float> *src = spec + ch * cs + (kx0 + col) * N + j;
    cpx<float> v[RT];
#pragma unroll
    for (int r = 0; r < RT; ++r) v[r] = ok ? src[r * NST] : cpx<float>{0.f, 0.f};
    if constexpr (RT == 8) dft8(v, -1.f);
    else if constexpr (RT == 4) dft4(v, -1.f);
    else if constexpr (RT == 2) dft2(v);
    if (j != 0) {  // twiddle step N / (NST RT) = 1
      cpx<float> wt[RT];
      load_twiddles<float, RT>(tw, j, wt);
#pragma unroll
      for (int r = 1; r < RT; ++r) v[r] = cmul(v[r], wt[r]);
    }
    cpx<float> *dst = sm + line * Np;
#pragma unroll
    for (int r = 0; r < RT; ++r) dst[smap<N>(j + r * NST)] = v[r];
  }
  __syncthreads();
  ct_dif_range<float, N, S - 2, 1>(sm, KC * C, tw);

  // ---- middle: last DIF stage, projection, first DIT stage -------------------------------
  // Three shared-memory phases over N / 2 threads per column: (1) the span-1 radix-8 DIF
  // butterflies of every (column, channel) line; (2) at each frequency position, the projection
  // of the three strain channels (Willot directions) and the |xi|^2 multiply of the phase-field
  // channel; (3) the span-1 radix-8 DIT butterflies.  The same operations in the same order as
  // a thread holding all four channels of a butterfly, with a quarter of the registers.
  {
    const int t = threadIdx.x;
    for (int b = t; b < KC * C * (N / 8); b += blockDim.x) {
      const int line = b / (N / 8), q = b - line * (N / 8);
      cpx<float> *ln = sm + line * Np;
      cpx<float> v[8];
#pragma unroll
      for (int r = 0; r < 8; ++r) v[r] = ln[smap<N>(8 * q + r)];
      dft8(v, -1.f);
#pragma unroll
      for (int r = 0; r < 8; ++r) ln[smap<N>(8 * q + r)] = v[r];
    }
    __syncthreads();
    for (int b = t; b < KC * N; b += blockDim.x) {
      const int col = b / N, pos = b - col * N;
      const int kx = kx0 + col;
      if (kx >= g.hx) continue;
      cpx<float> *base = sm + col * C * Np;
      const int sp = smap<N>(pos);
      {
        const float sc = (a.tab.xi2[0][kx] + a.tab.xi2[1][digit_rev_ct<N>(pos)]) * a.inv_n;
        const cpx<float> z = base[3 * Np + sp];
        base[3 * Np + sp] = {z.x * sc, z.y * sc};
      }
      int k[2] = {kx, digit_rev_ct<N>(pos)};
      ProjDir<float, 2> pd;
      float xi2;
      willot_dir<float, 2>(a.tab, k, a.inv_n, pd, xi2);
      float re[3], im[3];
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) {
        const cpx<float> z = base[ch * Np + sp];
        re[ch] = z.x;
        im[ch] = z.y;
      }
      project_mandel<float, 3>(re, pd);
      project_mandel<float, 3>(im, pd);
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) base[ch * Np + sp] = {re[ch], im[ch]};
    }
    __syncthreads();
    for (int b = t; b < KC * C * (N / 8); b += blockDim.x) {
      const int line = b / (N / 8), q = b - line * (N / 8);
      cpx<float> *ln = sm + line * Np;
      cpx<float> v[8];
#pragma unroll
      for (int r = 0; r < 8; ++r) v[r] = ln[smap<N>(8 * q + r)];
      dft8(v, 1.f);
#pragma unroll
      for (int r = 0; r < 8; ++r) ln[smap<N>(8 * q + r)] = v[r];
    }
  }
  __syncthreads();
  ct_dit_range<float, N, 1, S - 2>(sm, KC * C, tw);

  // ---- last DIT stage: shared -> registers -> global ---------------------------------------
  for (int b = threadIdx.x; b < KC * C * NBT; b += blockDim.x) {
    const int line = b / NBT, j = b - line * NBT;
    const int col = line / C, ch = line - col * C;
    const cpx<float> *src = sm + line * Np;
    cpx<float> v[RT];
#pragma unroll
    for (int r = 0; r < RT; ++r) v[r] = src[smap<N>(j + r * NST)];
    if (j != 0) {
      cpx<float> wt[RT];
      load_twiddles<float, RT>(tw, j, wt);
#pragma unroll
      for (int r = 1; r < RT; ++r) v[r] = cmul_conj(v[r], wt[r]);
    }
    if constexpr (RT == 8) dft8(v, 1.f);
    else if constexpr (RT == 4) dft4(v, 1.f);
    else if constexpr (RT == 2) dft2(v);
    if (kx0 + col < g.hx) {
      cpx<float> *dst = spec + ch * cs + (kx0 + col) * N + j;
#pragma unroll
      for (int r = 0; r < RT; ++r) dst[r * NST] = v[r];
    }
  }
}
