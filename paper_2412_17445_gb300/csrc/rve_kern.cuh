// Kernel interface of librve: argument structs shared by the kernel files and the host
// driver, block reductions, and the per-voxel material byte encoding.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "fft.cuh"

#define RVE_NOTCH_BIT 0x80  // material byte: bit 7 = notch (phi held at 1), bits 0..6 = phase

// Phase property table (device constant memory, one table per RVE is passed by value).
struct PhaseTab {
  double lam[16], mu[16], Gc[16];
};

// Constants of each phase that the float64 kernels would otherwise divide or multiply for in
// every voxel (a float64 division is a dozen instructions of 16 cycles each).
struct PhaseDer {
  double gl[16];    // Gc / l
  double r2gl[16];  // 2 / (Gc / l)
  double b[16];     // Gc l
  double bl[16];    // Gc l Lbar
};

// Grid description.
struct Geo {
  int d, m, c;          // dimension, Mandel components, channels (m + 1)
  int nx, ny, nz;
  int hx;               // nx / 2 + 1 half-spectrum row length
  int rows;             // ny * nz real rows of length nx
  long long n;          // voxels
};

// Per-axis frequency tables (natural index k in [0, N)):
//   sn = sin(pi ks / N), cs = cos(pi ks / N) (exactly 0 at the Nyquist index), xi2 = (2 pi ks / N)^2
// with ks the signed wave number.
template <typename T>
struct AxisTab {
  const T *sn[3], *cs[3], *xi2[3];
};

// Tangent channels of the scaled Newton operator, per voxel (structure of arrays, stride n):
//   [0, NC)            C' = s1 * C_t in Mandel form, upper triangle row by row (NC = m(m+1)/2)
//   [NC, NC+m)         sF1 = s1 * g'(phi) sigma_drive
//   NC+m               kappa = chi * s2 / s1 (free voxels), 0 on the notch
//   NC+m+1             a' = s2 * (Gc/l + 2H) (free), 0 on the notch
//   NC+m+2             w = (phi/l + l L phi) (free), 0 on the notch
//   NC+m+3             b' = s2 * Gc * l (free), 0 on the notch
//   NC+m+4             notch indicator (1 on the notch, else 0)
template <int M>
struct TanIdx {
  static constexpr int NC = M * (M + 1) / 2;
  static constexpr int SF = NC;
  static constexpr int KAPPA = NC + M;
  static constexpr int A = NC + M + 1;
  static constexpr int W = NC + M + 2;
  static constexpr int B = NC + M + 3;
  static constexpr int NOTCH = NC + M + 4;
  static constexpr int K = NC + M + 5;
};

// Several fixed-order reductions of per-block partials in one single-block launch
// (k_reduce_list): segment i reduces NQ quantities of G partials each (sum, or max when
// is_max) into out[off + q].
struct ReduceSeg {
  const double *part;
  int G, NQ, is_max, off;
};
struct ReduceList {
  ReduceSeg s[4];
  int n;
};

// Device scalars of one BiCGStab solve (read by every Krylov kernel).
struct KrylovScalars {
  double rho, alpha, omega, beta;
  double bn2, atol2, tol2;
  double rn2;
  double s3;            // row scaling of the constraint row
  // E-slots (scalar component) of the Krylov vectors
  double xE, rE, rhE, pE, vE, sE, tE;
  double bE;            // E slot of the right-hand side (kept for restarts)
  double escale;        // column scaling of the E unknown in this solve
  int strain;           // 1: constraint row is d_E (strain control), else s3 sum w d_phi
  int done;             // 1 once converged / stopped
  int status;           // 0 converged, 1 iteration limit, 2 breakdown
  int iters;
  int maxit;
  int fault_rho0;       // fault injection: the finalisers see rho = 0 (a breakdown)
  int pending;          // float32 chunks: x += alpha p + omega s, r = s - omega t of the last
                        // iteration not applied yet (the next x-forward pass, or the chunk's
                        // closing k_kx_finish, applies it)
  // float32 copies for the kernels of a float32 solve, whose threads would otherwise each convert
  // on the float64 pipe; pE_f, sE_f carry the column scaling (pE escale, sE escale)
  float alpha_f, omega_f, beta_f, pE_f, sE_f;
};
template <typename T>
__device__ __forceinline__ T ks_scalar(double d, float f) {
  if constexpr (sizeof(T) == 4) return f;
  else return d;
}

// ---- float64 roots and reciprocals ------------------------------------------------------
// By a float32 seed r, good to 2^-21, and the series of the exact value in its residual h to second
// order: 1 / x = r / (1 - h) = r (1 + h + h^2 + ...) with h = 1 - x r, and 1 / sqrt(x) = r (1 - h)^-1/2 =
// r (1 + h / 2 + 3 h^2 / 8 + ...) with h = 1 - x r^2.  What is cut, h^3, is 2^-63, so the reciprocal is
// within one step of the rounded quotient and the root within one unit in the last place: 3 and 5
// float64 operations.  The seed's bits are moved by integer instructions, not converted through the
// float64 pipe.  Arguments whose seed leaves the normal range take the library function.
__device__ __forceinline__ double f64_of_seed(float r, int shift) {  // r 2^shift, r in [2^-2, 2)
  const unsigned b = __float_as_uint(r);
  return __hiloint2double((int)((b >> 3) + ((896u + (unsigned)shift) << 20)), (int)(b << 29));
}
__device__ __forceinline__ double recip_nr(double x) {
  const int hi = __double2hiint(x);
  const int e = hi >> 20 & 2047;
  if ((unsigned)(e - 2) > 2041u) return 1.0 / x;
  const float m = __uint_as_float(0x3F800000u | (((unsigned)hi & 0xFFFFFu) << 3) | ((unsigned)__double2loint(x) >> 29));
  double r = f64_of_seed(__fdividef(1.f, m), 1023 - e);
  if (hi < 0) r = -r;
  const double h = 1.0 - x * r;
  return r + r * (h + h * h);
}
// 1 / sqrt(x) for x > 0; ok: false where x is not a positive normal number (0 is returned)
__device__ __forceinline__ double rsqrt_nr(double x, bool &ok) {
  const int hi = __double2hiint(x);
  const int e = hi >> 20;
  ok = (unsigned)(e - 2) <= 2041u;
  if (!ok) return 0.0;
  const int k = (e - 1023) >> 1, odd = (e - 1023) & 1;
  const float m = __uint_as_float((unsigned)(127 + odd) << 23 | (((unsigned)hi & 0xFFFFFu) << 3) |
                                  ((unsigned)__double2loint(x) >> 29));
  const double r = f64_of_seed(rsqrtf(m), -k);
  const double h = 1.0 - (x * r) * r;
  return r + (r * h) * (0.5 + 0.375 * h);
}
// x in type T, rounded to nearest; float32 by integer instructions in its normal range
template <typename T>
__device__ __forceinline__ T round_to(double x) {
  if constexpr (sizeof(T) == 4) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    if (((unsigned)(b >> 52 & 2047) - 897u) >= 253u) return (T)x;
    const unsigned long long t = b + 0x0FFFFFFFull + (b >> 29 & 1);
    return __uint_as_float((unsigned)(b >> 32) & 0x80000000u |
                           (((unsigned)(t >> 29) - (896u << 23)) & 0x7FFFFFFFu));
  } else {
    return x;
  }
}
// max(x, 0) and min(x, 0) by the sign bit; 0 for NaN, as fmax and fmin give
__device__ __forceinline__ double pos_part(double x) {
  return (unsigned)__double2hiint(x) <= 0x7FF00000u ? x : 0.0;
}
__device__ __forceinline__ double neg_part(double x) {
  return (unsigned)__double2hiint(x) - 0x80000000u <= 0x7FF00000u ? x : 0.0;
}

// ---- block reductions into per-block partials ------------------------------------------
// Sum NQ doubles over the block; thread 0 writes part[q * G + blk].
template <int NQ>
__device__ __forceinline__ void block_partials(double (&v)[NQ], double *part, int G, int blk) {
  __shared__ double red[32][NQ > 0 ? NQ : 1];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    double x = v[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if (lane == 0) red[wid][q] = x;
  }
  __syncthreads();
  if (wid == 0) {
    const int nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      double x = lane < nw ? red[lane][q] : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
      if (lane == 0) part[q * G + blk] = x;
    }
  }
  __syncthreads();
}

// As block_partials for per-thread sums held in the Krylov precision TK: with TK = float the
// warp-level shuffle tree stays in float32 (32 terms) and only the per-warp sums are added in
// float64, which keeps the float64 pipe (1/64 of the float32 rate) out of the float32 passes.
template <typename TK, int NQ>
__device__ __forceinline__ void block_partials_k(const TK (&v)[NQ], double *part, int G, int blk) {
  if constexpr (sizeof(TK) == 8) {
    double w[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) w[q] = (double)v[q];
    block_partials<NQ>(w, part, G, blk);
  } else {
    __shared__ double red[32][NQ > 0 ? NQ : 1];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      float x = v[q];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
      if (lane == 0) red[wid][q] = (double)x;
    }
    __syncthreads();
    const int nw = (blockDim.x + 31) >> 5;
    constexpr int LQ = NQ <= 2 ? 16 : 8;  // lanes a quantity
    if (NQ <= 4 && nw <= LQ) {
      // one warp: three or four dependent float64 adds
      if (threadIdx.x < 32) {
        const int q = threadIdx.x / LQ, w = threadIdx.x % LQ;
        double sum = q < NQ && w < nw ? red[w][q] : 0.0;
#pragma unroll
        for (int o = LQ / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (w == 0 && q < NQ) part[q * G + blk] = sum;
      }
    } else if (threadIdx.x < NQ) {
      double sum = 0.0;
      for (int w = 0; w < nw; ++w) sum += red[w][threadIdx.x];
      part[threadIdx.x * G + blk] = sum;
    }
    __syncthreads();
  }
}

template <int NQ>
__device__ __forceinline__ void block_max_partials(double (&v)[NQ], double *part, int G, int blk) {
  __shared__ double red[32][NQ > 0 ? NQ : 1];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    double x = v[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = fmax(x, __shfl_down_sync(0xffffffffu, x, o));
    if (lane == 0) red[wid][q] = x;
  }
  __syncthreads();
  if (wid == 0) {
    const int nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      double x = lane < nw ? red[lane][q] : -1.0e308;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x = fmax(x, __shfl_down_sync(0xffffffffu, x, o));
      if (lane == 0) part[q * G + blk] = x;
    }
  }
  __syncthreads();
}

// Programmatic dependent launch, at the top of the passes of an apply: wait for the kernels before
// (at once where the launch has no such dependency).  No pass triggers its successor early: the
// successor's launch is prepared while the pass runs and takes place when its last block ends, on
// an empty GPU.  Triggered at the top of the pass instead, the next blocks settle wherever an SM has
// room while the pass still runs, several to one SM and none to others (float32 2048 x 256:
// 62 us an apply, 123 us with the early trigger, 68 us with ordinary launches; 512^2: 24.5, 30.7, 29).
__device__ __forceinline__ void pdl_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ---- kernel argument structs ------------------------------------------------------------
// Operator apply: y = S J x (scaled Jacobian of the linearisation).
template <typename T>
struct ApplyArgs {
  Geo g;
  T *x;                 // c channels (written back when a fused update forms it)
  T *y;                 // c channels (phi channel also holds the pointwise part between passes)
  const T *tan;         // tangent channels (TanIdx)
  const double *xE_ptr; // E slot of x (device scalar)
  double e_scale;       // column scaling of the E unknown: d_E = e_scale * xE (ks == nullptr)
  T fM[6];              // load direction (Mandel)
  const float *xEf_ptr; // float32 solves: the scaled E slot e_scale * xE, when the scalars hold it
  cpx<T> *spec;         // spectral scratch c * rows * hx
  double *part;         // per-block partials
  // fused BiCGStab vector updates (prologue) and dots (epilogue)
  int pro_mode;         // 0: x as given; 1: x := r + beta (x - omega v); 2: x := r - alpha v;
                        // 4: projection only (strain channels of x through G, nothing else);
                        // 5: as 1, after the pending update of the previous iteration
                        //    (xs += alpha x + omega s, r := s - omega t) when ks->pending
  T *r;                 // (written in mode 5)
  const T *v, *rhat, *s;  // operands of the fused updates / dots
  T *xs;                // mode 5: the Krylov solution vector
  const T *t;           // mode 5: A s of the previous iteration
  int epi_mode;         // 0: none; 1: dot(rhat, y); 2: dots (y, s), (y, y); 3: projection
                        // (writes the m strain channels of y only); 6: dots (y, s), (y, y),
                        // (rhat, s), (rhat, y), (s, s) for the merged omega / convergence update
  const KrylovScalars *ks;
  int tr;               // 1: spectral scratch transposed [ch][kx][row] (fused 2D column pass)
  // finalisation by the x-inverse pass itself (krylov_fin.cuh): 0 none; 1 / 2 the member's
  // last block runs the alpha / omega update on ksw (epilogue modes 1 / 2); 3 one more block, the
  // first, writes yE = sum of the constraint-row partials; 4 it copies *xE_ptr to yE (strain control);
  // 5 the last block runs the alpha update and clears ks->pending; 6 the last block runs the
  // merged omega / convergence update (epilogue mode 6) and sets ks->pending
  int fin;
  KrylovScalars *ksw;
  unsigned int *arrive; // arrival counter of the member (fin 1, 2)
  double *yE;           // fin 3, 4
};

// Residual: spectral data of (sigma, phi) in float64, epilogue forms F, rhs and w.
struct ResidArgs {
  Geo g;
  const double *sigma;  // m channels
  const double *phi;    // 1 channel
  const double *H;      // current history max(psi+, H^n)
  const uint8_t *mat;
  PhaseDer pd;
  double ell, rell, s1;
  cpx<double> *spec;
  double *F;            // unscaled residual F1 (m ch), F2 (1 ch)
  double *Lphi;         // L phi
  void *rhs;            // Krylov rhs b = -S F (krylov precision), c channels
  int rhs_double;       // 1 if rhs is double
  void *tan;            // tangent channels (w written here)
  int tan_double;
  int tanK;             // number of tangent channels
  double *part;
};

// Column (y / z) pass of the spectral data.
template <typename T>
struct ColArgs {
  Geo g;
  cpx<T> *spec;
  int axis;          // 1 = y, 2 = z
  int W;             // kx columns per block (a power of two)
  int lw;            // log2 W
  FftPlan plan;      // along the axis
  FftPlan yplan;     // y plan (3D z-pass: ky of a stored row is digit_reverse(yplan, y))
  AxisTab<T> tab;
  T inv_n;
  const KrylovScalars *ks;
};

// Constitutive update at one Newton iterate (float64).
struct ConstArgs {
  Geo g;
  const double *eps_t;  // m channels
  const double *phi;
  const double *Hn;
  const uint8_t *mat;
  PhaseTab ph;
  double fM[6];
  double E;
  PhaseDer pd;
  double ell, k_res, s1;
  int isotropic;
  double *sigma;        // m channels out
  double *H;            // max(psi+, H^n) out
  double *part;         // partials: m stress sums, |s1 sigma|^2
  double *part_max;     // partial max of 2 psi+ / (Gc / l) over free voxels
};

// Krylov vectors: c channels of n values (type TK); E slots live in KrylovScalars.
template <typename TK>
struct KvArgs {
  long long len;        // c * n
  int c;
  long long n;
  TK *x, *r, *rhat, *p, *v, *s, *t;
  KrylovScalars *ks;
  double *part;
  int G;
  unsigned int *arrive; // non-null: the last block of k_kxr runs the convergence test
};

// ---- groups: one launch over several RVEs of the same shape ----------------------------
// Passed by value as __grid_constant__ kernel parameters; member i is handled by the blocks
// with blockIdx.y == i (blockIdx.z for the 3D column passes, blockIdx.x for the
// single-block finalisers).  A solo launch is a group of one.
constexpr int kGroupMax = 8;

template <typename T>
struct ApplyGroup {
  ApplyArgs<T> m[kGroupMax];
};

template <typename T>
struct ColGroup {
  ColArgs<T> base;                       // geometry, plans, tables (shared by the members)
  cpx<T> *spec[kGroupMax];               // per member: spectral scratch
  const KrylovScalars *ks[kGroupMax];    // per member: Krylov scalars (or null)
};

template <typename TK>
struct KvGroup {
  KvArgs<TK> m[kGroupMax];
};

