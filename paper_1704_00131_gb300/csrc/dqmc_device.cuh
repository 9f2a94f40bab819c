// GB300 (sm_103a) kernels of the BSS/DQMC sweep.
//
// Work decomposition: one thread-block cluster per Markov chain, one CTA per
// flavor (spin up / spin down of the spin-z decoupling).  The flavors are
// independent except in the acceptance ratio R = gamma * prod_s R_s, which the
// CTAs exchange through distributed shared memory; every other step (wraps,
// delayed updates, the FP64 QR/UDV stabilisation, the stable recompute of G)
// runs in the flavor's own CTA.
//
// Precision: the working Green function, the wraps and the delayed updates are
// templated on `Real` (double, float, or float pairs); the stabilisation chain
// (B-products, pivoted QR, T update, the stable (1 + UDV)^-1 and log|det|) is FP64
// or, in the float-pair modes, float pairs with FP64 scales.
//
// Method (ALF 1.0 documentation, arXiv:1704.00131):
//   B_tau = exp(-dtau K) exp(V_tau)                       Sec. 2.1, Eq. of B_tau
//   G(tau) = (1 + B(tau,0) B(beta,tau))^-1               Eq. Green_eq
//   sequential single-field updates, Metropolis         Sec. 2.2.1
//   QR-stabilised chain every n_wrap slices             Sec. 2.3, Eq. green_stable
//   sweep: tau = 1..L up, L..1 down                     Algorithm 1, Sec. 2.4
#pragma once
//
// This header holds the device code shared by the kernel translation units:
// the per-precision sweep units (dqmc_sweep_fp64.cu, dqmc_sweep_fp32.cu,
// dqmc_sweep_mixed.cu) instantiate the sweep and fresh-G kernels for one
// working precision each, so that nvcc compiles them in parallel;
// dqmc_kernels.cu holds the precision-independent kernels and the dispatch.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <type_traits>

#include "../../include/dqmc.h"
#include "dqmc_internal.h"

// DQMC_QR_CALL: how the panelled QR is called.  The sweep kernels' units say __noinline__:
// held to 128 registers they spilled in it, with its renewed norms and scaled panels the
// more (float pairs 480 bytes of spill loads, out of line 104; with split products 3220 and
// 2144).  Sweeps of 9 x 7, 40 chains in float pairs: 23.3 ms inlined, 22.9 out of line
// (22.4 before those corrections); 8 x 8, 64 chains in FP64: 35.5 and 34.7.  The
// adjoints, at 255 registers, lose by the call (log|det| of 64 8 x 8: 8.75 and 8.89 ms).
//
// DQMC_WITH_UMMA: 1 compiles the float pairs' tensor-core products into the
// float-pair kernels (the unit of DQMC_PREC_MIXED_TC), 0 leaves them out (the unit of
// DQMC_PREC_MIXED, whose kernels then keep their registers for the SIMT tiles).  The
// FP64 products' are in every unit.
#ifndef DQMC_QR_CALL
#define DQMC_QR_CALL
#endif
#ifndef DQMC_WITH_UMMA
#define DQMC_WITH_UMMA 1
#endif

namespace cg = cooperative_groups;

namespace dqmc {
// Internal linkage: every translation unit that includes this header gets its
// own copy of the device code it instantiates.
namespace {

// --------------------------------------------------------------------------
// Philox4x32-10 (Salmon et al., SC'11): the counter-based generator that
// draws the proposal (u1) and acceptance (u2) uniforms of every proposal.
// --------------------------------------------------------------------------
__device__ __forceinline__ void philox4x32_10(uint32_t c[4], uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t lo0 = 0xD2511F53u * c[0], hi0 = __umulhi(0xD2511F53u, c[0]);
    const uint32_t lo1 = 0xCD9E8D57u * c[2], hi1 = __umulhi(0xCD9E8D57u, c[2]);
    const uint32_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
    c[0] = n0; c[1] = lo1; c[2] = n2; c[3] = lo0;
    k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
  }
}

__device__ __forceinline__ double uniform53(uint32_t hi, uint32_t lo) {
  const uint64_t w = ((uint64_t)hi << 32) | lo;
  return (double)(w >> 11) * 0x1.0p-53;
}

// Sub-phase cycle counter: thread 0 adds the cycles since *t0 to acc[q].
__device__ __forceinline__ void tick(long long* acc, int q, long long& t0) {
  const long long t1 = clock64();
  if (acc && threadIdx.x == 0) acc[q] += t1 - t0;
  t0 = t1;
}

// --------------------------------------------------------------------------
// Field couplings: Ising (type 1) c(s) = lambda s; four-valued HS (type 2)
// c(l) = g eta(l) with weight gamma(l) (Sec. 2.1, the discrete HS transform).
// --------------------------------------------------------------------------
__device__ __forceinline__ double hs_eta(int l) {
  const double a = sqrt(2.0 * (3.0 - sqrt(6.0))), b = sqrt(2.0 * (3.0 + sqrt(6.0)));
  return l == 1 ? a : l == -1 ? -a : l == 2 ? b : -b;
}
__device__ __forceinline__ double hs_gamma(int l) {
  return (l == 1 || l == -1) ? 1.0 + sqrt(6.0) / 3.0 : 1.0 - sqrt(6.0) / 3.0;
}
__device__ __forceinline__ double coupling(int ft, double cscale, int f) {
  return ft == 1 ? cscale * (double)f : cscale * hs_eta(f);
}
__device__ __forceinline__ double field_weight(int ft, int f) { return ft == 1 ? 1.0 : hs_gamma(f); }
// Proposal: Ising flips; HS picks one of the three other values of
// (-2,-1,1,2), in ascending order, with index floor(3 u1).
__device__ __forceinline__ int propose_field(int ft, int f, double u1) {
  if (ft == 1) return -f;
  int idx = (int)floor(3.0 * u1);
  idx = idx > 2 ? 2 : idx;
  const int vals[4] = {-2, -1, 1, 2};
  int n = 0, out = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (vals[q] != f) {
      if (n == idx) out = vals[q];
      ++n;
    }
  return out;
}
__device__ __forceinline__ double coupling_dU(int ft, double dtau, double U, double cscale, int f) {
  if (ft == 1) return 0.5 * dtau * exp(0.5 * dtau * U) / sinh(cscale) * (double)f;
  return dtau / (4.0 * cscale) * hs_eta(f);
}

// --------------------------------------------------------------------------
// Block-wide reductions (deterministic order).
// --------------------------------------------------------------------------
__device__ __forceinline__ double block_sum(double v, double* red) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double r = 0.0;
#pragma unroll
  for (int w = 0; w < kThreads / 32; ++w) r += red[w];
  return r;
}
__device__ __forceinline__ double block_max(double v, double* red) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double r = red[0];
#pragma unroll
  for (int w = 1; w < kThreads / 32; ++w) r = fmax(r, red[w]);
  return r;
}

// --------------------------------------------------------------------------
// Float-float ("double-word") numbers: x = hi + lo with |lo| <= ulp(hi)/2,
// about 48 significant bits on the FP32 pipes, which run 64x faster than FP64
// on this GPU.  Error-free transformations: TwoSum (Knuth), FastTwoSum
// (Dekker), TwoProd with an FMA (Joldes, Muller, Popescu, ACM TOMS 2017).
// The working Green function of the mixed path is stored in this format.
// --------------------------------------------------------------------------
struct dd {
  float hi, lo;
};

__device__ __forceinline__ dd two_sum(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  return {s, (a - (s - bb)) + (b - bb)};
}
__device__ __forceinline__ dd fast_two_sum(float a, float b) {
  const float s = a + b;
  return {s, b - (s - a)};
}
__device__ __forceinline__ dd dd_add(dd a, dd b) {
  const dd s = two_sum(a.hi, b.hi);
  return fast_two_sum(s.hi, s.lo + (a.lo + b.lo));
}
__device__ __forceinline__ dd dd_mul(dd a, dd b) {
  const float p = a.hi * b.hi;
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, e));
  return fast_two_sum(p, e);
}
// c + a * b
__device__ __forceinline__ dd dd_fma(dd a, dd b, dd c) {
  const float p = a.hi * b.hi;
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, e));
  const dd s = two_sum(c.hi, p);
  return fast_two_sum(s.hi, s.lo + (c.lo + e));
}

// Arithmetic adapters of the working precision (double, float, dd).
__device__ __forceinline__ double to_d(double x) { return x; }
__device__ __forceinline__ double to_d(float x) { return (double)x; }
__device__ __forceinline__ double to_d(dd x) { return (double)x.hi + (double)x.lo; }
template <typename R>
__device__ __forceinline__ R from_d(double x);
template <>
__device__ __forceinline__ double from_d<double>(double x) { return x; }
template <>
__device__ __forceinline__ float from_d<float>(double x) { return (float)x; }
template <>
__device__ __forceinline__ dd from_d<dd>(double x) {
  const float h = (float)x;
  return {h, (float)(x - (double)h)};
}
template <typename R>
__device__ __forceinline__ R from_zero() { return R{}; }
// 1 or 0 without a conversion (conversions from FP64 run on the slow FP64 pipe)
template <typename R>
__device__ __forceinline__ R unit(bool one) { return one ? R(1) : R(0); }
template <>
__device__ __forceinline__ dd unit<dd>(bool one) { return {one ? 1.f : 0.f, 0.f}; }
__device__ __forceinline__ double rfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float rfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ dd rfma(dd a, dd b, dd c) { return dd_fma(a, b, c); }
__device__ __forceinline__ double rmul(double a, double b) { return a * b; }
__device__ __forceinline__ float rmul(float a, float b) { return a * b; }
__device__ __forceinline__ dd rmul(dd a, dd b) { return dd_mul(a, b); }
__device__ __forceinline__ double radd(double a, double b) { return a + b; }
__device__ __forceinline__ float radd(float a, float b) { return a + b; }
__device__ __forceinline__ dd radd(dd a, dd b) { return dd_add(a, b); }
__device__ __forceinline__ double rneg(double a) { return -a; }
__device__ __forceinline__ float rneg(float a) { return -a; }
__device__ __forceinline__ dd rneg(dd a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ double rsub(double a, double b) { return a - b; }
__device__ __forceinline__ float rsub(float a, float b) { return a - b; }
__device__ __forceinline__ dd rsub(dd a, dd b) { return dd_add(a, {-b.hi, -b.lo}); }

// Type of the acceptance ratios and of the diagonal they come from: float pairs
// where G is held in float pairs (an FP64 instruction of a warp holds its
// scheduler's FP64 unit for 65 cycles, a dependent float-pair operation takes
// about 30), FP64 otherwise.  The ratios are then as exact as the diagonal they are
// formed from: a pair rounds at 2^-47, the wrapped G between two stabilisations is
// off by 1e-8 on average.  For a given diagonal in float pairs the product of both flavors'
// ratios is off by 1.5e-15 to 3.2e-15 on average (at most 5.1e-14) at U = 1 to 20, where
// FP64 from the same diagonal would be off by 1e-16 (1.5e-15).
template <typename Real>
struct RatioOf { using type = double; };
template <>
struct RatioOf<dd> { using type = dd; };
__device__ __forceinline__ double to_ratio(double x, double) { return x; }
__device__ __forceinline__ double to_ratio(float x, double) { return (double)x; }
__device__ __forceinline__ dd to_ratio(dd x, dd) { return x; }
template <typename Real>
__device__ __forceinline__ Real ratio_to(double x) { return (Real)x; }
template <typename Real>
__device__ __forceinline__ Real ratio_to(dd x) { return x; }
__device__ __forceinline__ bool is_neg(double x) { return x < 0.0; }
__device__ __forceinline__ bool is_neg(dd x) { return x.hi < 0.f; }
// Metropolis: u < min(1, |R|); a NaN ratio counts as 1
__device__ __forceinline__ bool accepts(double u, double R) {
  const double a = fabs(R);
  // |R| >= 1 or NaN from the exponent bits, without an FP64 comparison
  if ((__double2hiint(a) & 0x7fffffff) >= 0x3ff00000) return true;
  return u < a;
}
__device__ __forceinline__ bool accepts(dd u, dd R) {
  const float h = fabsf(R.hi), l = R.hi < 0.f ? -R.lo : R.lo;
  if (!(h < 1.f || (h == 1.f && l < 0.f))) return true;
  return u.hi < h || (u.hi == h && u.lo < l);
}
// a / b by one reciprocal estimate and Newton corrections of the quotient
// (Markstein, IBM J. Res. Dev. 34, 1990) in a quarter of the plain division's dependent
// FP64 instructions.  The reciprocal is good to about 2^-46, the exact remainder times it
// to 2^-92 of the quotient, so the result is the correctly rounded one but for quotients
// within 2^-39 units of a rounding boundary (2e5 random quotients, emulated with exact
// multiply-adds: all equal to the plain division's); values outside the estimate's FP32
// range take the plain division.
__device__ __forceinline__ double quick_div(double a, double b) {
  const int e = (__double2hiint(b) >> 20) & 0x7ff;
  if (e < 1023 - 100 || e > 1023 + 100) return a / b;
  const double r0 = (double)(1.0f / (float)b);
  const double r = fma(r0, fma(-b, r0, 1.0), r0);
  const double q = a * r;
  return fma(fma(-b, q, a), r, q);
}
// float-pair quotient by long division with two correction steps
__device__ __forceinline__ dd quick_div(dd a, dd b) {
  const float r = 1.0f / b.hi;
  const float q0 = a.hi * r;
  dd t = dd_fma({-q0, 0.f}, b, a);
  const float q1 = t.hi * r;
  t = dd_fma({-q1, 0.f}, b, t);
  const dd q = fast_two_sum(q0, q1);
  return dd_add(q, {t.hi * r, 0.f});
}

// A pointer known to lie in shared memory, in a function that is not inlined and
// could not tell (generic loads of the panels cost the products a quarter).
template <typename T>
__device__ __forceinline__ T* as_shared(T* p) {
  return reinterpret_cast<T*>(__cvta_shared_to_generic(__cvta_generic_to_shared(p)));
}

// --------------------------------------------------------------------------
// CTA-level dense product C = op(A) op(B), row-major, generic pointers
// (global or shared).  Output tiles of 16R x 16R (R = 1..5 outputs per thread and
// dimension; R is picked per size so that N = 16, 144 or 400 need no padding),
// 16-deep K panels staged in shared memory.  C must not alias A or B.
// --------------------------------------------------------------------------
__host__ __device__ inline int gemm_pick_r(int n) {
  int best_r = 4, best = 1 << 30;
  for (int r = 5; r >= 1; --r) {
    const int t = 16 * r;
    const int padded = ((n + t - 1) / t) * t;
    if (padded < best) { best = padded; best_r = r; }
  }
  return best_r;
}

template <typename T, bool TA, bool TB, int R, bool ACC = false>
__device__ void cta_gemm_r(int M, int Nc, int Kd, const T* __restrict__ A, int lda, const T* __restrict__ B,
                           int ldb, T* __restrict__ C, int ldc, T* sm) {
  constexpr int TT = 16 * R;
  T* As = as_shared(sm);  // [16][TT]
  T* Bs = As + 16 * TT;   // [16][TT]
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  for (int m0 = 0; m0 < M; m0 += TT)
    for (int n0 = 0; n0 < Nc; n0 += TT) {
      T acc[R][R];
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j) acc[i][j] = T(0);
      for (int k0 = 0; k0 < Kd; k0 += 16) {
#pragma unroll
        for (int e = tid; e < 16 * TT; e += kThreads) {
          int r, kk;
          if (!TA) { r = e >> 4; kk = e & 15; } else { kk = e / TT; r = e - kk * TT; }
          const int gm = m0 + r, gk = k0 + kk;
          T val = T(0);
          if (gm < M && gk < Kd) val = TA ? A[(size_t)gk * lda + gm] : A[(size_t)gm * lda + gk];
          As[kk * TT + r] = val;
        }
#pragma unroll
        for (int e = tid; e < 16 * TT; e += kThreads) {
          int kk, c;
          if (!TB) { kk = e / TT; c = e - kk * TT; } else { c = e >> 4; kk = e & 15; }
          const int gk = k0 + kk, gn = n0 + c;
          T val = T(0);
          if (gk < Kd && gn < Nc) val = TB ? B[(size_t)gn * ldb + gk] : B[(size_t)gk * ldb + gn];
          Bs[kk * TT + c] = val;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
          T a[R], b[R];
#pragma unroll
          for (int i = 0; i < R; ++i) a[i] = As[kk * TT + ty * R + i];
#pragma unroll
          for (int j = 0; j < R; ++j) b[j] = Bs[kk * TT + tx * R + j];
#pragma unroll
          for (int i = 0; i < R; ++i)
#pragma unroll
            for (int j = 0; j < R; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
      }
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j) {
          const int gm = m0 + ty * R + i, gn = n0 + tx * R + j;
          if (gm < M && gn < Nc) {
            if (ACC) C[(size_t)gm * ldc + gn] += acc[i][j];
            else C[(size_t)gm * ldc + gn] = acc[i][j];
          }
        }
    }
  __syncthreads();
}

// One copy per kernel and operand form (a call costs nothing beside the product;
// inlined copies at every call site took minutes to compile and spilled).
template <typename T, bool TA, bool TB>
__device__ __noinline__ void cta_gemm(int M, int Nc, int Kd, const T* __restrict__ A, int lda, const T* __restrict__ B,
                         int ldb, T* __restrict__ C, int ldc, T* sm) {
  const int r = gemm_pick_r(M > Nc ? M : Nc);
  if (r == 1) cta_gemm_r<T, TA, TB, 1>(M, Nc, Kd, A, lda, B, ldb, C, ldc, sm);
  else if (r == 2) cta_gemm_r<T, TA, TB, 2>(M, Nc, Kd, A, lda, B, ldb, C, ldc, sm);
  else if (r == 3) cta_gemm_r<T, TA, TB, 3>(M, Nc, Kd, A, lda, B, ldb, C, ldc, sm);
  else if (r == 5) cta_gemm_r<T, TA, TB, 5>(M, Nc, Kd, A, lda, B, ldb, C, ldc, sm);
  else cta_gemm_r<T, TA, TB, 4>(M, Nc, Kd, A, lda, B, ldb, C, ldc, sm);
}

// The same tiling for float-float operands: every product hi*hi is split
// exactly (TwoProd), its high part summed with TwoSum into the accumulator's
// high word, the rounding errors and the hi*lo, lo*hi cross terms gathered in
// the low word and renormalised once per output.
template <bool TA, bool TB, int R, bool ACC = false>
__device__ void cta_gemm_dd_r(int M, int Nc, int Kd, const dd* __restrict__ A, int lda, const dd* __restrict__ B,
                              int ldb, dd* __restrict__ C, int ldc, dd* sm) {
  constexpr int TT = 16 * R;
  dd* As = as_shared(sm);  // [16][TT]
  dd* Bs = As + 16 * TT;   // [16][TT]
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  for (int m0 = 0; m0 < M; m0 += TT)
    for (int n0 = 0; n0 < Nc; n0 += TT) {
      float ah[R][R], al[R][R];
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j) { ah[i][j] = 0.f; al[i][j] = 0.f; }
      for (int k0 = 0; k0 < Kd; k0 += 16) {
#pragma unroll
        for (int e = tid; e < 16 * TT; e += kThreads) {
          int r, kk;
          if (!TA) { r = e >> 4; kk = e & 15; } else { kk = e / TT; r = e - kk * TT; }
          const int gm = m0 + r, gk = k0 + kk;
          dd val = {0.f, 0.f};
          if (gm < M && gk < Kd) val = TA ? A[(size_t)gk * lda + gm] : A[(size_t)gm * lda + gk];
          As[kk * TT + r] = val;
        }
#pragma unroll
        for (int e = tid; e < 16 * TT; e += kThreads) {
          int kk, c;
          if (!TB) { kk = e / TT; c = e - kk * TT; } else { c = e >> 4; kk = e & 15; }
          const int gk = k0 + kk, gn = n0 + c;
          dd val = {0.f, 0.f};
          if (gk < Kd && gn < Nc) val = TB ? B[(size_t)gn * ldb + gk] : B[(size_t)gk * ldb + gn];
          Bs[kk * TT + c] = val;
        }
        __syncthreads();
#pragma unroll 4
        for (int kk = 0; kk < 16; ++kk) {
          dd a[R], b[R];
#pragma unroll
          for (int i = 0; i < R; ++i) a[i] = As[kk * TT + ty * R + i];
#pragma unroll
          for (int j = 0; j < R; ++j) b[j] = Bs[kk * TT + tx * R + j];
#pragma unroll
          for (int i = 0; i < R; ++i)
#pragma unroll
            for (int j = 0; j < R; ++j) {
              const float p = a[i].hi * b[j].hi;
              const float pe = fmaf(a[i].hi, b[j].hi, -p);
              const float s = ah[i][j] + p;
              const float bb = s - ah[i][j];
              const float se = (ah[i][j] - (s - bb)) + (p - bb);
              ah[i][j] = s;
              float lo = al[i][j] + (se + pe);
              lo = fmaf(a[i].hi, b[j].lo, lo);
              al[i][j] = fmaf(a[i].lo, b[j].hi, lo);
            }
        }
        __syncthreads();
      }
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j) {
          const int gm = m0 + ty * R + i, gn = n0 + tx * R + j;
          if (gm < M && gn < Nc) {
            const dd r = fast_two_sum(ah[i][j], al[i][j]);
            C[(size_t)gm * ldc + gn] = ACC ? dd_add(C[(size_t)gm * ldc + gn], r) : r;
          }
        }
    }
  __syncthreads();
}


#include "dqmc_umma.cuh"

// tile: 3 (48 x 48 output tiles) or 4 (64 x 64); 0 picks the one with less
// padding of max(M, Nc) (the autotuner may override it per context)
template <bool TA, bool TB, bool ACC>
__device__ void gemm_dd_tiles(int M, int Nc, int Kd, const dd* A, int lda, const dd* B, int ldb, dd* C, int ldc,
                              dd* sm, int tile = 0) {
  if (tile != 3 && tile != 4) {
    const int n = M > Nc ? M : Nc;
    const int p3 = (n + 47) / 48 * 48, p4 = (n + 63) / 64 * 64;
    tile = (p3 < p4) ? 3 : 4;
  }
  if (tile == 3) cta_gemm_dd_r<TA, TB, 3, ACC>(M, Nc, Kd, A, lda, B, ldb, C, ldc, sm);
  else cta_gemm_dd_r<TA, TB, 4, ACC>(M, Nc, Kd, A, lda, B, ldb, C, ldc, sm);
}

// store(x, y, load(x, y)) for every element of an N x N matrix, four per thread in
// flight (the matrices come from L2: a loop of one load and one store at a time waits
// out its latency N^2 / 256 times, a tenth of a slice at N = 64).  In place is fine:
// every element is loaded and stored by one thread.  Ends with a barrier.
template <typename L, typename F>
__device__ __forceinline__ void each_element(int N, L load, F store) {
  constexpr int U = 4;
  const int n = N * N, dq = kThreads / N, dr = kThreads - dq * N;
  int e = threadIdx.x, x = e / N, y = e - x * N;
  if (n <= kThreads) {
    if (e < n) store(x, y, load(x, y));
    e = n;
  }
  while (e < n) {
    decltype(load(0, 0)) v[U];
    int xs[U], ys[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const bool ok = e < n;
      xs[u] = ok ? x : -1;
      ys[u] = y;
      v[u] = load(ok ? x : 0, ok ? y : 0);
      e += kThreads;
      x += dq;
      y += dr;
      if (y >= N) { y -= N; ++x; }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (xs[u] >= 0) store(xs[u], ys[u], v[u]);
  }
  __syncthreads();
}

template <typename T>
__device__ __forceinline__ void cta_copy(int N, int ld, const T* src, T* dst) {
  each_element(
      N, [&](int x, int y) { return src[(size_t)x * ld + y]; },
      [&](int x, int y, T v) { dst[(size_t)x * ld + y] = v; });
}

// --------------------------------------------------------------------------
// Shared-memory layout of the sweep kernel.
// --------------------------------------------------------------------------
struct Smem {
  double* gemm;     // kGemmRegionBytes: 2*16*kGemmMaxTile doubles of the SIMT GEMM panels (also
                    // float / float-pair)
  double* v;        // [ld] slice potential / exp factors
  double* ev;       // [ld]
  double* d;        // [ld] current diagonal of the effective G
  double* hv;       // [ld] Householder vector
  double* u2;       // [MV]
  double* delta;    // [MV]
  double* gam;      // [MV]
  double* xdiag;    // [ld] exchange: diagonal of G for the potential energy
  double* spare;    // [ld] scratch (the float-pair QR's list of norms to recompute)
  double* xs;       // [8]  exchange: scalars
  double* red;      // [32]
  int* ired;        // [32]
  int* qsite;       // [MV]
  int* qinv;        // [ld] position in the slice's visiting order of the vertex on site x (-1: none)
  int8_t* fnew;     // [MV]
  int8_t* fslice;   // [MV] fields of the current slice
  int* expA;        // [kExpLen(ld)] row exponents of the split tensor-core products
  int* expB;        // [kExpLen(ld)] column exponents
  double* ab;       // delayed vectors A, B [2][k][ld] when they fit in shared memory
  int flavor;       // the CTA's flavor
  double* qred;     // [8][128] partial sums of the QR trailing update
  Umma um;          // tensor-core products: barriers and TMEM slot, staging over gemm and ab
  const PlaneSet* ps;    // split products of float pairs (null: SIMT tiles)
  const PlaneSet* ps64;  // split products of FP64 operands (null: the FP64 pipe)
  int dd_tile;      // register tile of the float-pair SIMT products (0: by padding, 3, 4)
};

__device__ inline Smem carve_smem(unsigned char* base, int ld, int MV) {
  Smem s;
  unsigned char* const start = base;
  base += kSmemCounterBytes;
  double* p = reinterpret_cast<double*>(base);
  s.v = p; p += ld;
  s.ev = p; p += ld;
  s.d = p; p += ld;
  s.hv = p; p += ld;
  s.xdiag = p; p += ld;
  s.spare = p; p += ld;
  s.u2 = p; p += MV;
  s.delta = p; p += MV;
  s.gam = p; p += MV;
  s.xs = p; p += 8;
  s.red = p; p += 32;
  int* ip = reinterpret_cast<int*>(p);
  s.ired = ip; ip += 32;
  s.qsite = ip; ip += MV;
  s.qinv = ip; ip += ld;
  int8_t* bp = reinterpret_cast<int8_t*>(ip);
  s.fnew = bp; bp += MV;
  s.fslice = bp; bp += MV + 16;
  const size_t off = ((size_t)(bp - reinterpret_cast<int8_t*>(base)) + 15) / 16 * 16;
  s.qred = reinterpret_cast<double*>(base + off);
  const int le = exp_len(ld);
  s.expA = reinterpret_cast<int*>(s.qred + 8 * 128);
  s.expB = s.expA + le;
  unsigned char* q = reinterpret_cast<unsigned char*>(s.expB + le);
  q = base + (((size_t)(q - base) + 15) / 16 * 16);
  s.um.bar = reinterpret_cast<uint64_t*>(q);                 // 2 kUmmaStages mbarriers, counters
  s.um.tmem_slot = reinterpret_cast<uint32_t*>(q + 96);
  s.um.err = nullptr;
  s.um.where = nullptr;
  s.dd_tile = 0;
  s.ps = nullptr;
  s.ps64 = nullptr;
  s.um.limit = kUmmaWaitCycles;
  s.um.stall = 0;
  q += 128;
  // (offsets from the 128-byte aligned start, no pointer-to-integer casts: the compiler
  // then knows that the panels are shared memory)
  q = start + ((size_t)(q - start) + 127) / 128 * 128;
  s.gemm = reinterpret_cast<double*>(q);
  s.ab = reinterpret_cast<double*>(q + gemm_region_bytes(ld));
  uint32_t dyn;
  asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn));
  s.um.stage = q;
  s.um.stage_bytes = dyn - (uint32_t)(q - start);
  return s;
}

// The split products of this CTA: float pairs (want_dd) and / or FP64 operands,
// where the chain has plane buffers.  Returns whether tensor memory was allocated
// (every path out of the kernel then calls umma_free).
__device__ __forceinline__ bool umma_begin(ChainDev& C, int s, Smem& S, bool want_dd, bool want_64) {
  S.dd_tile = C.dd_tile;
  S.um.err = &C.error;
  // the caller's wait limit and the test hook concern the float-pair products; FP64
  // ones keep the default limit
  S.um.limit = (want_dd && C.wait_cycles > 0) ? C.wait_cycles : kUmmaWaitCycles;
  S.um.stall = want_dd ? C.test_stall : 0;
  S.um.where = C.wait_where[s];
  S.ps = want_dd ? C.ps[s] : nullptr;
  S.ps64 = want_64 ? C.ps64[s] : nullptr;
  const bool on = S.ps != nullptr || S.ps64 != nullptr;
  umma_acquire_maps(S.ps);
  umma_acquire_maps(S.ps64);
  if (on) umma_alloc(S.um);
  return on;
}

// Float-pair product of the mixed path: exact-split tensor-core products when
// the chain has plane buffers, the float-pair SIMT tiles otherwise.  constA /
// constB: index of a prepared constant operand (kCpEA ...), -1: split here.
template <bool TA, bool TB, bool ACC>
__device__ void gemm_dd(const ChainDev& C, int s, Smem& S, int M, int Nc, int Kd, const dd* A, int lda, const dd* B,
                        int ldb, dd* Cm, int ldc, int constA = -1, int constB = -1) {
#if DQMC_WITH_UMMA
  if (S.ps) {
    gemm_umma<dd>(TA, TB, ACC, M, Nc, Kd, A, lda, B, ldb, Cm, ldc, S.ps, S.expA, S.expB, S.um, constA, constB);
    return;
  }
#endif
  gemm_dd_tiles<TA, TB, ACC>(M, Nc, Kd, A, lda, B, ldb, Cm, ldc, reinterpret_cast<dd*>(S.gemm), S.dd_tile);
}

// FP64 product: exact-split tensor-core products when the chain has plane buffers
// (its N from kTc64MinSites), the FP64 pipe's tiles otherwise.
template <bool TA, bool TB>
__device__ void gemm_64(Smem& S, int M, int Nc, int Kd, const double* A, int lda, const double* B, int ldb, double* Cm,
                        int ldc, int constA = -1, int constB = -1) {
  if (S.ps64)
    gemm_umma<double>(TA, TB, false, M, Nc, Kd, A, lda, B, ldb, Cm, ldc, S.ps64, S.expA, S.expB, S.um, constA, constB);
  else
    cta_gemm<double, TA, TB>(M, Nc, Kd, A, lda, B, ldb, Cm, ldc, S.gemm);
}

// Bit 0 of the chain's error word.  (Beside bit 1 of a wait that gave up, which must stay:
// the products after it are skipped, their barriers' phases are no longer known.  The
// word is shared with the peer flavor's CTA.)
__device__ __forceinline__ void numerical_failure(ChainDev& C) {
  if (threadIdx.x == 0) atomicOr(&C.error, 1);
}

// Slice potential v^s_i of slice tau (1-based) from global fields.
__device__ void slice_potential_global(const ChainDev& C, int s, int tau, double* v) {
  for (int x = threadIdx.x; x < C.N; x += kThreads) v[x] = 0.0;
  __syncthreads();
  for (int k = threadIdx.x; k < C.MV; k += kThreads)
    v[C.site[k]] = C.vsign[s * C.MV + k] * coupling(C.ft, C.cscale, C.fields[(size_t)(tau - 1) * C.MV + k]);
  __syncthreads();
}

// Slice potential from the shared-memory copy of the slice's fields.
__device__ void slice_potential_smem(const ChainDev& C, int s, const int8_t* fsl, double* v) {
  for (int x = threadIdx.x; x < C.N; x += kThreads) v[x] = 0.0;
  __syncthreads();
  for (int k = threadIdx.x; k < C.MV; k += kThreads)
    v[C.site[k]] = C.vsign[s * C.MV + k] * coupling(C.ft, C.cscale, fsl[k]);
  __syncthreads();
}

// --------------------------------------------------------------------------
// FP64 stabilisation building blocks (Sec. 2.3).
// --------------------------------------------------------------------------
struct UDV {
  const double* Q;
  const double* D;
  const double* T;
  int detq;
};

__device__ inline double* wmat(const ChainDev& C, int s, int m) {
  return C.work[s] + (size_t)m * C.N * C.ld;
}
__device__ inline double* wvec(const ChainDev& C, int s, int v) {
  return C.work[s] + (size_t)kWorkMats * C.N * C.ld + (size_t)v * C.ld;
}
__device__ inline UDV ident_udv(const ChainDev& C) {
  UDV u;
  u.Q = C.ident;
  u.T = C.ident + (size_t)C.N * C.ld;
  u.D = C.ident + (size_t)2 * C.N * C.ld;
  u.detq = 1;
  return u;
}
__device__ inline double* slot_base(const ChainDev& C, int s, int j) {
  return C.slots[s] + (size_t)j * slot_stride(C.N, C.ld);
}
__device__ inline UDV slot_udv(const ChainDev& C, int s, int j) {
  UDV u;
  double* b = slot_base(C, s, j);
  u.Q = b;
  u.T = b + (size_t)C.N * C.ld;
  u.D = b + (size_t)2 * C.N * C.ld;
  u.detq = C.slot_detq[s][j];
  return u;
}

__device__ inline void to_dd_mat(int N, int ld, const double* src, dd* dst) {
  each_element(
      N, [&](int x, int y) { return src[(size_t)x * ld + y]; },
      [&](int x, int y, double v) { dst[(size_t)x * ld + y] = from_d<dd>(v); });
}

// dd -> double in place (same 8-byte slot)
__device__ inline void dd_to_d_inplace(int N, int ld, void* buf) {
  dd* a = reinterpret_cast<dd*>(buf);
  double* b = reinterpret_cast<double*>(buf);
  each_element(
      N, [&](int x, int y) { return a[(size_t)x * ld + y]; },
      [&](int x, int y, dd v) { b[(size_t)x * ld + y] = to_d(v); });
}

// ---- pivoted QR in panels, LU and solves, on FP64 or float-pair matrices --------
// Scalars of the reflectors and the LU in the matrix's own type.
__device__ __forceinline__ double rsqrt_of_sum(double x) { return sqrt(x); }
// sqrt of a float pair: FP32 root and one Newton step (Heron) on the pair
__device__ __forceinline__ dd rsqrt_of_sum(dd x) {
  if (!(x.hi > 0.f)) return {0.f, 0.f};
  const float r = sqrtf(x.hi);
  const dd e = dd_fma({-r, 0.f}, {r, 0.f}, x);
  return fast_two_sum(r, e.hi / (2.f * r));
}
__device__ __forceinline__ bool is_pos(double x) { return x > 0.0; }
__device__ __forceinline__ bool is_pos(dd x) { return x.hi > 0.f; }
__device__ __forceinline__ double rabs(double x) { return fabs(x); }
__device__ __forceinline__ dd rabs(dd x) { return x.hi < 0.f ? dd{-x.hi, -x.lo} : x; }
__device__ __forceinline__ double shfl_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ dd shfl_xor(dd v, int o) {
  return {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}
__device__ __forceinline__ double shfl(double v, int l) { return __shfl_sync(0xffffffffu, v, l); }
__device__ __forceinline__ dd shfl(dd v, int l) {
  return {__shfl_sync(0xffffffffu, v.hi, l), __shfl_sync(0xffffffffu, v.lo, l)};
}

// Panels in shared memory, column-major with an odd column stride (neighbouring
// threads' rows and columns fall into different banks).
__device__ __forceinline__ int panel_ld(int N) { return N | 1; }
// Columns per panel of the QR.  Wider panels save passes over the matrix, but the
// products of more reflectors lose the small rows of Q: with 16 columns the wrapped
// G's drift on 4 x 4 lattices is four times the unblocked factorisation's, with 4
// the same (FP64, U = 4: mean 1.4e-11, 3.7e-12 and 3.5e-12).
// (kPanel; a matrix so large that the shared memory holds only narrower panels takes
// qr_panel_cols of them.)
// Columns per panel of the LU and the solves: the largest power of two <= 16 of which
// two panels fit the product area.
__device__ inline int panel_width(int N, const Smem& S) {
  const int cap = (int)(S.um.stage_bytes / 16);
  int w = 16;
  while (w > 1 && w * panel_ld(N) > cap) w >>= 1;
  return w;
}

// log2 of a positive FP64 number in FP32 (an order for the columns, not a value)
__device__ __forceinline__ float log2_rough(double x) {
  const int hi = __double2hiint(x), ex = (hi >> 20) & 0x7ff;
  const float m = __int_as_float(((hi & 0xfffff) << 3) | 0x3f800000);
  return ex == 0 ? -3.0e38f : (float)(ex - 1023) + __log2f(m);
}
// order of a column: log2 of its norm (from the square) and scale; zero and NaN columns
// last, but finite: above the -Inf of a column that is no candidate
constexpr float kLeastKey = -3.4e38f;
__device__ __forceinline__ float column_key(float norm2, float lsc) {
  return fmaxf(0.5f * log2f(norm2) + lsc, kLeastKey);  // (fmaxf drops a NaN)
}
__device__ __forceinline__ float column_key(double norm2, float lsc) {
  return norm2 > 0.0 ? fmaxf(0.5f * log2_rough(norm2) + lsc, kLeastKey) : kLeastKey;
}
__device__ __forceinline__ float column_key(dd norm2, float lsc) { return column_key(fmaxf(norm2.hi, 0.f), lsc); }
__device__ __forceinline__ float as_float(double x) { return (float)x; }
__device__ __forceinline__ float as_float(dd x) { return x.hi; }
// a downdated squared norm below 2^-26 of its last full value (or not positive)
__device__ __forceinline__ bool norm_spent(double n, double full) {
  const int a = __double2hiint(n), b = __double2hiint(full);
  return a <= 0 || b - a > (26 << 20);
}
__device__ __forceinline__ bool norm_spent(dd n, dd full) { return !(n.hi > 1.4901161e-8f * full.hi); }

// Squared norm of rows r0.. of column j, in FP64 (one thread).
template <typename T>
__device__ __noinline__ double column_norm2(int N, int ld, const T* X, int j, int r0) {
  double a = 0.0;
#pragma unroll 4
  for (int i = r0; i < N; ++i) {
    const double x = to_d(X[(size_t)i * ld + j]);
    a = fma(x, x, a);
  }
  return a;
}
// Whether an FP32 sum of squares is good for a key: neither overflown nor (squares of
// entries below 1e-19) underflown.
__device__ __forceinline__ bool norm2_in_range(float a) { return a > 0x1.0p-100f && a < INFINITY; }

// Keys (log2 of the scaled column norms, by list position) of the columns of M = X
// diag(dsc), and log2 dsc (by column).  The keys only order the columns, so the sums of
// squares are formed in FP32; a column whose sum leaves its range is summed in FP64 (X is
// a product of n_wrap slices with an orthogonal matrix, usually far inside).
template <typename T>
__device__ void column_keys(int N, int ld, const T* X, const double* dsc, float* key, float* lsc, Smem& S) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int nw = kThreads / 32;
  float* part = reinterpret_cast<float*>(S.qred);   // [nw][32] partial sums of squares
  for (int j0 = 0; j0 < N; j0 += 32) {
    const int j = j0 + lane;
    float a0 = 0.f, a1 = 0.f;
    if (j < N) {
      int i = warp;
      for (; i + nw < N; i += 2 * nw) {
        const float x = as_float(X[(size_t)i * ld + j]), y = as_float(X[(size_t)(i + nw) * ld + j]);
        a0 = fmaf(x, x, a0);
        a1 = fmaf(y, y, a1);
      }
      if (i < N) {
        const float x = as_float(X[(size_t)i * ld + j]);
        a0 = fmaf(x, x, a0);
      }
    }
    part[warp * 32 + lane] = a0 + a1;
    __syncthreads();
    if (warp == 0 && j < N) {
      float a = 0.f;
#pragma unroll
      for (int w = 0; w < nw; ++w) a += part[w * 32 + lane];
      lsc[j] = log2_rough(dsc[j]);
      key[j] = norm2_in_range(a) ? column_key(a, lsc[j]) : column_key(column_norm2<T>(N, ld, X, j, 0), lsc[j]);
    }
    __syncthreads();
  }
}

// A[r0:, j0:] -= V (W^T A[r0:, j0:]) with the N - r0 rows of V and W in shared
// panels of `nb` <= kPanel columns: one column of A per thread (and G threads, one row
// class each, where the columns leave threads over), the nb sums in registers.
// FLIP: the roles of V and W exchanged.  LIST: position j stands for column list[j],
// and the keys of the rows below the panel are renewed.
template <typename T, bool FLIP, bool LIST>
__device__ void panel_apply(int N, int ld, T* A, int r0, int j0, int nb, const T* Vp, const T* Wp, Smem& S,
                            const int* list, float* key, const float* lsc) {
  constexpr int PW = kPanel;
  const int tid = threadIdx.x, ldp = panel_ld(N);
  const T* Lp = FLIP ? Wp : Vp;  // left factor of the update
  const T* Rp = FLIP ? Vp : Wp;  // the sums' factor
  T* red = reinterpret_cast<T*>(S.qred);  // [G][4][cw] <= 1024
  for (int c0 = j0; c0 < N; c0 += kThreads) {
    const int nc = (N - c0 < kThreads) ? N - c0 : kThreads;
    const int cw = (nc + 31) / 32 * 32, G = kThreads / cw;
    const int g = tid / cw, jj = tid - g * cw;
    const bool act = g < G && jj < nc;
    const int j = act ? (LIST ? list[c0 + jj] : c0 + jj) : 0;
    float n2 = 0.f;
    T y[PW];
#pragma unroll
    for (int q = 0; q < PW; ++q) y[q] = from_zero<T>();
    if (act) {
      // four rows at a time, their loads issued together (eight were slower)
      int i = r0 + g;
      for (; i + 3 * G < N; i += 4 * G) {
        T x[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) x[b] = A[(size_t)(i + b * G) * ld + j];
        const T* r = Rp + (i - r0);
#pragma unroll
        for (int q = 0; q < PW; ++q)
          if (q < nb) {
#pragma unroll
            for (int b = 0; b < 4; ++b) y[q] = rfma(r[q * ldp + b * G], x[b], y[q]);
          }
      }
      for (; i < N; i += G) {
        const T x = A[(size_t)i * ld + j];
        const T* r = Rp + (i - r0);
#pragma unroll
        for (int q = 0; q < PW; ++q)
          if (q < nb) y[q] = rfma(r[q * ldp], x, y[q]);
      }
    }
    if (G > 1) {
      // the row classes' sums in rounds of four, each summed by one class
#pragma unroll
      for (int b = 0; b < PW; b += 4) {
        if (b >= nb) continue;
        if (act) {
#pragma unroll
          for (int q = 0; q < 4; ++q) red[(g * 4 + q) * cw + jj] = y[b + q];
        }
        __syncthreads();
        if (act) {
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (q % G == g) {
              T t = red[q * cw + jj];
              for (int h = 1; h < G; ++h) t = radd(t, red[(h * 4 + q) * cw + jj]);
              red[q * cw + jj] = t;
            }
        }
        __syncthreads();
        if (act) {
#pragma unroll
          for (int q = 0; q < 4; ++q) y[b + q] = red[q * cw + jj];
        }
        __syncthreads();
      }
    }
    if (act) {
#pragma unroll
      for (int q = 0; q < PW; ++q) y[q] = rneg(y[q]);
      int i = r0 + g;
      for (; i + 3 * G < N; i += 4 * G) {
        T x[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) x[b] = A[(size_t)(i + b * G) * ld + j];
        const T* l = Lp + (i - r0);
#pragma unroll
        for (int q = 0; q < PW; ++q)
          if (q < nb) {
#pragma unroll
            for (int b = 0; b < 4; ++b) x[b] = rfma(l[q * ldp + b * G], y[q], x[b]);
          }
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          A[(size_t)(i + b * G) * ld + j] = x[b];
          if (LIST && i + b * G >= r0 + nb) {
            const float f = as_float(x[b]);
            n2 = fmaf(f, f, n2);
          }
        }
      }
      for (; i < N; i += G) {
        T x = A[(size_t)i * ld + j];
        const T* l = Lp + (i - r0);
#pragma unroll
        for (int q = 0; q < PW; ++q)
          if (q < nb) x = rfma(l[q * ldp], y[q], x);
        A[(size_t)i * ld + j] = x;
        if (LIST && i >= r0 + nb) {
          const float f = as_float(x);
          n2 = fmaf(f, f, n2);
        }
      }
    }
    if (LIST) {
      float* part = reinterpret_cast<float*>(S.qred);
      if (act) part[g * cw + jj] = n2;
      __syncthreads();
      if (act && g == 0) {
        for (int h = 1; h < G; ++h) n2 += part[h * cw + jj];
        key[c0 + jj] = norm2_in_range(n2) ? column_key(n2, lsc[j])
                                          : column_key(column_norm2<T>(N, ld, A, j, r0 + nb), lsc[j]);
      }
      __syncthreads();
    }
  }
  __syncthreads();
}

// Wp = Vp Tm (nb x nb, row stride kPanel)
template <typename T>
__device__ void panel_times_t(int rows, int ldp, int nb, const T* Vp, const T* Tm, T* Wp) {
  const int q = threadIdx.x % kPanel;
  if (q < nb)
    for (int i = threadIdx.x / kPanel; i < rows; i += kThreads / kPanel) {
      T a = from_zero<T>();
      for (int j = 0; j < nb; ++j) a = rfma(Vp[j * ldp + i], Tm[j * kPanel + q], a);
      Wp[q * ldp + i] = a;
    }
  __syncthreads();
}

// alpha = -sign(x_0) |x|, v_0 = x_0 - alpha and beta = 2 / v^T v from x_0 and |x|^2.
template <typename T>
__device__ __forceinline__ void reflector_scalars(T x0, T xn2, T& alpha, T& v0, T& beta) {
  const T xn = rsqrt_of_sum(xn2);
  alpha = is_neg(x0) ? xn : rneg(xn);
  v0 = rsub(x0, alpha);
  beta = quick_div(unit<T>(true), rfma(rabs(x0), xn, xn2));  // v^T v = 2 (|x|^2 + |x_0| |x|)
}

// Power of two that brings a panel's column to a norm of about one, from the log2 of its
// norm, so that squares of float pairs neither underflow (entries below 1e-19 would lose
// their reflector, from 1e-16 bits of it) nor overflow.  Exact both ways; FP64 needs none.
__device__ __forceinline__ int panel_shift(float log2_norm, double) { return 0; }
__device__ __forceinline__ int panel_shift(float log2_norm, dd) {
  return fabsf(log2_norm) < 150.f ? max(-120, min(120, __float2int_rn(log2_norm))) : 0;
}
__device__ __forceinline__ double times_pow2(double x, int) { return x; }
__device__ __forceinline__ dd times_pow2(dd x, int e) {
  const float f = __int_as_float((127 + e) << 23);
  return {x.hi * f, x.lo * f};
}

// T of the panel at hand, behind qr_blocked's other entries of S.qred.
template <typename T>
__device__ __forceinline__ T* panel_tri(const Smem& S) { return reinterpret_cast<T*>(S.qred) + 256; }

// Pivoted Householder QR of M = X diag(dsc), X N x N, in panels: reflections act on rows
// and commute with the column scales, so the factors are X's, R_M = R_X diag(dsc[perm]).
// Columns do not move: perm[k] is the column at position k, R_kj sits at X[k][perm[j]],
// reflector k's vector below row k of column perm[k] (its leading entry in vk0[k]); in
// float pairs each vector is that of its column scaled to norm one (panel_shift).
// tri[panel][kPanel][kPanel]: the triangular factors T of the panels' products H_0 .. H_{nb-1} =
// 1 - V T V^T (compact WY, Schreiber & Van Loan 1989).  Returns det(Q) = (-1)^#reflectors.
//
// Pivoting: a panel takes the columns of largest remaining scaled norm, renewed from the
// updated matrix, and orders them by their downdated norms while it is factorised: the
// order of Businger and Golub's pivoting but for a column that overtakes a panel's
// last ones within the panel.  Norms that cancel below 2^-26 of the square they were
// downdated from are formed again from the panel (LAPACK's xGEQPF rule): in float pairs
// the rest is rounding error, of either sign.  (Sorting the columns once before an unpivoted
// factorisation is cheaper still, but made the wrapped G's drift up to 3.5 times
// larger: the first block of a chain has no graded scales to sort by.)
//
// A panel is factorised in shared memory, one reduction per column: the products of
// the column with every column of the panel give its norm, the update's coefficients
// and T's next column at once.  One warp forms the scalars and the next pivot (a warp's
// FP64 instruction holds its scheduler's unit for 65 cycles; eight warps computing the
// same square root and quotients cost most of a column before).  The rest of the matrix
// is updated once per panel, from registers.
template <typename T>
__device__ DQMC_QR_CALL int qr_blocked(int N, int ld, T* X, const double* dsc, int* perm, T* vk0, T* tri, Smem& S) {
  // (pw: the arrays' strides; wide: the columns a panel takes)
  constexpr int pw = kPanel, RG = kThreads / pw, nwarp = kThreads / 32;
  static_assert(32 / pw == nwarp, "one lane group of the scalar warp per warp's partial products");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, q = tid % pw, rg = tid / pw;
  const int ldp = panel_ld(N), wide = qr_panel_cols(N, S.um.stage_bytes);
  T* Vp = reinterpret_cast<T*>(S.gemm);
  T* Wp = Vp + wide * ldp;
  T* red = reinterpret_cast<T*>(S.qred);        // [nwarp][pw] partial products
  T* wq = red + nwarp * pw;                     // [pw] update coefficients of the columns to come
  T* zq = wq + pw;                              // [2][pw] products with the earlier vectors
  T* sc = zq + 2 * pw;                          // [2][2] leading entry of v, beta
  T* Tm = panel_tri<T>(S);                      // [pw][pw], by panel column
  float* key = reinterpret_cast<float*>(S.hv);  // [N] by position
  float* lsc = key + N;                         // [N] by column
  int* list = S.qinv;                           // [N] columns by position
  int* rank = reinterpret_cast<int*>(S.spare);  // [N]
  int* pos_of = S.ired + 16;                    // [pw] position in the panel of its columns (-1: to come)
  int* next_p = S.ired;                         // [2] pivot of the next step
  int* renew = S.ired + 2;                      // [1] the columns' norms are to be formed again
  int detq = 1;
  column_keys<T>(N, ld, X, dsc, key, lsc, S);
  for (int j = tid; j < N; j += kThreads) list[j] = j;
  __syncthreads();
  for (int k0 = 0; k0 < N; k0 += wide) {
    const int nb = (N - k0 < wide) ? N - k0 : wide, rows = N - k0;
    // the panel's columns: the nb largest keys, in order; the others keep theirs
    for (int t = tid; t < rows; t += kThreads) {
      const float kt = key[k0 + t];
      int r = 0;
      for (int u = 0; u < rows; ++u) {
        const float ku = key[k0 + u];
        r += (ku > kt || (ku == kt && u < t)) ? 1 : 0;
      }
      rank[t] = r;
    }
    __syncthreads();
    {
      int at[9], cj[9];  // N <= 9 kThreads positions (the shared vectors allow fewer)
      float kk[9];
#pragma unroll
      for (int b = 0; b < 9; ++b) {
        const int t = tid + b * kThreads;
        at[b] = -1;
        if (t < rows) {
          const int r = rank[t];
          int idx = r;
          if (r >= nb) {
            idx = nb + t;
            for (int u = 0; u < t; ++u) idx -= rank[u] < nb ? 1 : 0;
          }
          at[b] = k0 + idx;
          cj[b] = list[k0 + t];
          kk[b] = key[k0 + t];
        }
      }
      __syncthreads();
#pragma unroll
      for (int b = 0; b < 9; ++b)
        if (at[b] >= 0) {
          list[at[b]] = cj[b];
          key[at[b]] = kk[b];
        }
      __syncthreads();
    }
    // (a thread's panel column is q, here and below)
    const int shift = (q < nb) ? panel_shift(key[k0 + q] - lsc[list[k0 + q]], T{}) : 0;
    for (int e = tid; e < rows * pw; e += kThreads) {
      const int r = e / pw, c = e - r * pw;
      if (c < nb) Vp[c * ldp + r] = times_pow2(X[(size_t)(k0 + r) * ld + list[k0 + c]], -shift);
    }
    if (tid < pw * pw) Tm[tid] = from_zero<T>();
    if (tid < 2 * pw) zq[tid] = from_zero<T>();
    if (tid < pw) pos_of[tid] = -1;
    if (tid == 0) next_p[0] = 0;  // the selection is in order
    __syncthreads();
    // squared norms of the panel's columns (warp 0, lane q), downdated step by step, and
    // their last full values
    T nrm2 = from_zero<T>(), full2 = from_zero<T>();
    const float lscq = (q < nb) ? lsc[list[k0 + q]] + (float)shift : 0.f;
    auto over_groups = [](T v) {  // the sum over a warp's lanes of the same q
#pragma unroll
      for (int o = 16; o >= pw; o >>= 1) v = radd(v, shfl_xor(v, o));
      return v;
    };
    {
      T a = from_zero<T>();
      if (q < nb)
        for (int r = rg; r < rows; r += RG) a = rfma(Vp[q * ldp + r], Vp[q * ldp + r], a);
      a = over_groups(a);
      if (lane < pw) red[warp * pw + lane] = a;
      __syncthreads();
      if (warp == 0) full2 = nrm2 = over_groups(red[lane]);
      __syncthreads();
    }
    // the column to come of largest norm (ties: the lowest), for warp 0
    auto next_pivot = [&](bool done) {
      float k = done ? -INFINITY : column_key(nrm2, lscq);
      int kp = q;
#pragma unroll
      for (int o = pw / 2; o; o >>= 1) {
        const float ok = __shfl_xor_sync(0xffffffffu, k, o);
        const int op = __shfl_xor_sync(0xffffffffu, kp, o);
        if (ok > k || (ok == k && op < kp)) { k = ok; kp = op; }
      }
      return kp;
    };
    for (int c = 0; c < nb; ++c) {
      const int p = next_p[c & 1];
      const T* x = Vp + p * ldp;
      T a = from_zero<T>();
      if (q < nb) {
        const T* y = Vp + q * ldp;
        for (int r = c + rg; r < rows; r += RG) a = rfma(x[r], y[r], a);
      }
      a = over_groups(a);
      if (lane < pw) red[warp * pw + lane] = a;
      __syncthreads();
      if (warp == 0) {
        const T t = over_groups(red[lane]);  // lane group w holds warp w's sums
        const T xn2 = shfl(t, p);
        const T x0 = x[c];
        T alpha = x0, v0 = x0, beta = from_zero<T>();
        if (is_pos(xn2)) reflector_scalars(x0, xn2, alpha, v0, beta);
        // v_q^T v (earlier columns), v^T y_q (columns to come)
        const int pq = pos_of[q];
        const bool done = q >= nb || pq >= 0 || q == p;
        const T yc = (q < nb) ? Vp[q * ldp + c] : from_zero<T>();
        const T z = rfma(rneg(alpha), yc, t);
        const T w = rneg(rmul(beta, z));
        if (lane < pw) {
          if (pq >= 0) zq[(c & 1) * pw + q] = z;
          wq[q] = done ? from_zero<T>() : w;
        }
        // the next pivot: largest downdated norm among the columns to come
        const T rc = rfma(w, v0, yc);
        nrm2 = rfma(rneg(rc), rc, nrm2);
        const int kp = next_pivot(done);
        const int shift_p = __shfl_sync(0xffffffffu, shift, p);
        const bool spent = __any_sync(0xffffffffu, !done && norm_spent(nrm2, full2));
        __syncwarp();
        if (lane == 0) {
          *renew = spent;
          sc[(c & 1) * 2] = v0;
          sc[(c & 1) * 2 + 1] = beta;
          pos_of[p] = c;
          next_p[(c & 1) ^ 1] = kp;
          X[(size_t)(k0 + c) * ld + list[k0 + p]] = times_pow2(alpha, shift_p);  // R's diagonal
          vk0[k0 + c] = v0;
        }
      }
      __syncthreads();
      const T v0 = sc[(c & 1) * 2], beta = sc[(c & 1) * 2 + 1];
      if (is_pos(beta)) detq = -detq;
      if (q < nb && pos_of[q] < 0) {
        const T w = wq[q];
        T* y = Vp + q * ldp;
        for (int r = c + rg; r < rows; r += RG) y[r] = rfma(w, (r == c) ? v0 : x[r], y[r]);
      }
      // T's next column (last warp): -beta T (V^T v) over the earlier ones, beta itself
      if (warp == nwarp - 1 && lane < pw) {
        T t = from_zero<T>();
        for (int j = 0; j < nb; ++j) t = rfma(Tm[lane * pw + j], zq[(c & 1) * pw + j], t);
        t = rneg(rmul(beta, t));
        __syncwarp((1u << pw) - 1u);
        Tm[lane * pw + p] = lane == p ? beta : t;
      }
      __syncthreads();
      if (tid == 0) Vp[p * ldp + c] = v0;
      if (*renew) {
        const bool done = q >= nb || pos_of[q] >= 0;
        T a2 = from_zero<T>();
        if (!done) {
          const T* y = Vp + q * ldp;
          for (int r = c + 1 + rg; r < rows; r += RG) a2 = rfma(y[r], y[r], a2);
        }
        a2 = over_groups(a2);
        if (lane < pw) red[warp * pw + lane] = a2;
        __syncthreads();
        if (warp == 0) {
          full2 = nrm2 = over_groups(red[lane]);
          const int kp = next_pivot(done);
          if (lane == 0) next_p[(c & 1) ^ 1] = kp;
        }
        __syncthreads();
      }
    }
    __syncthreads();
    // R's strict upper part and the vectors back to X; V gets its zeros above the diagonal
    for (int e = tid; e < rows * pw; e += kThreads) {
      const int r = e / pw, c = e - r * pw;
      if (c < nb && r != pos_of[c])
        X[(size_t)(k0 + r) * ld + list[k0 + c]] = times_pow2(Vp[c * ldp + r], r < pos_of[c] ? shift : 0);
    }
    int col = 0, pc = 0;
    if (q < nb) { col = list[k0 + q]; pc = pos_of[q]; }
    const int tr = rg;  // row of T (threads below pw * pw)
    const T tv = (tid < pw * pw) ? Tm[tid] : from_zero<T>();
    __syncthreads();
    // (a position is below kPanel, so one row per thread covers the zeros)
    if (q < nb && rg < pc) Vp[q * ldp + rg] = from_zero<T>();
    if (tid < nb) list[k0 + pc] = col;  // the panel's columns by position
    // T by position: in global memory, or in place for a single panel
    T* tg = N > pw ? tri + (size_t)(k0 / wide) * pw * pw : Tm;
    if (tid < pw * pw && tr < nb && q < nb) tg[pos_of[tr] * pw + pc] = tv;
    __syncthreads();
    if (k0 + nb < N) {
      panel_times_t<T>(rows, ldp, nb, Vp, Tm, Wp);
      // Q^T A = A - V T^T V^T A = A - V (V T)^T A
      panel_apply<T, false, true>(N, ld, X, k0, k0 + nb, nb, Vp, Wp, S, list, key, lsc);
    }
  }
  for (int j = tid; j < N; j += kThreads) perm[j] = list[j];
  __syncthreads();
  return detq;
}

// Q = H_0 H_1 ... H_{N-1} from qr_blocked's vectors, panel by panel from the last:
// Q A = A - (V T) (V^T A).
template <typename T>
__device__ void form_q_blk(int N, int ld, const T* X, const int* perm, const T* vk0, const T* tri, T* Q, Smem& S) {
  const int tid = threadIdx.x;
  constexpr int pw = kPanel;
  const int ldp = panel_ld(N), wide = qr_panel_cols(N, S.um.stage_bytes);
  T* Vp = reinterpret_cast<T*>(S.gemm);
  T* Wp = Vp + wide * ldp;
  for (int e = tid; e < N * N; e += kThreads) {
    const int x = e / N, y = e - x * N;
    Q[(size_t)x * ld + y] = unit<T>(x == y);
  }
  __syncthreads();
  for (int k0 = (N - 1) / wide * wide; k0 >= 0; k0 -= wide) {
    const int nb = (N - k0 < wide) ? N - k0 : wide, rows = N - k0;
    for (int e = tid; e < rows * pw; e += kThreads) {
      const int r = e / pw, c = e - r * pw;
      if (c < nb)
        Vp[c * ldp + r] = r < c ? from_zero<T>() : r == c ? vk0[k0 + c] : X[(size_t)(k0 + r) * ld + perm[k0 + c]];
    }
    __syncthreads();
    panel_times_t<T>(rows, ldp, nb, Vp, N > pw ? tri + (size_t)(k0 / wide) * pw * pw : panel_tri<T>(S), Wp);
    panel_apply<T, true, false>(N, ld, Q, k0, k0, nb, Vp, Wp, S, nullptr, nullptr, nullptr);
  }
}

// LU and solves of the middle matrix, blocked, templated on double and float
// pairs.  On the mixed path they run in float pairs on the FP32 pipes: every
// row of Mid has an entry of order one (for each i either Db_R,i = 1 or
// Ds_R,i = 1, and likewise for the columns), so Mid, its LU factors and the
// solution X = Mid^-1 Db_R^-1 Q_R^T stay inside the float range; entries that
// underflow are below 1e-38 of their row and change G by less than that in
// absolute value.
//
// Blocking: a panel of columns (or a block of rows of the right-hand sides) is
// staged in shared memory and finished there; everything beyond it is updated by
// one accumulate-GEMM.  Pivots are chosen on the top 32 bits of |a| (a pivot within
// 2^-20 of the largest); one warp forms each pivot's reciprocal, log|det| is summed
// once at the end.

// C += A B (row-major, no transposes) on the register-tiled CTA products.
__device__ __noinline__ void gemm_acc(int M, int Nc, int Kd, const double* A, int lda, const double* B, int ldb, double* C, int ldc,
                                Smem& S) {
  const int r = gemm_pick_r(M > Nc ? M : Nc);
  if (r == 1) cta_gemm_r<double, false, false, 1, true>(M, Nc, Kd, A, lda, B, ldb, C, ldc, S.gemm);
  else if (r == 2) cta_gemm_r<double, false, false, 2, true>(M, Nc, Kd, A, lda, B, ldb, C, ldc, S.gemm);
  else if (r == 3) cta_gemm_r<double, false, false, 3, true>(M, Nc, Kd, A, lda, B, ldb, C, ldc, S.gemm);
  else if (r == 5) cta_gemm_r<double, false, false, 5, true>(M, Nc, Kd, A, lda, B, ldb, C, ldc, S.gemm);
  else cta_gemm_r<double, false, false, 4, true>(M, Nc, Kd, A, lda, B, ldb, C, ldc, S.gemm);
}
__device__ inline void gemm_acc(int M, int Nc, int Kd, const dd* A, int lda, const dd* B, int ldb, dd* C, int ldc,
                                Smem& S) {
  gemm_dd_tiles<false, false, true>(M, Nc, Kd, A, lda, B, ldb, C, ldc, reinterpret_cast<dd*>(S.gemm), S.dd_tile);
}

// order of |a| for the pivot search: its top 32 bits; -1 for NaN, 1 for what they miss
__device__ __forceinline__ int pivot_key(double a) {
  const int k = umma_mag(a);
  return a != a ? -1 : (k == 0 && a != 0.0) ? 1 : k;
}
__device__ __forceinline__ int pivot_key(dd a) { return a.hi != a.hi ? -1 : umma_mag(a); }

// P A = L U in place (unit L below the diagonal, rows interchanged whole); rowof[i] =
// the row of A now at row i, diag[k] = 1 / U_kk.  tmp: 16 x N scratch (ld).  Returns 1
// if a pivot column has no finite nonzero entry.
template <typename T>
__device__ int lu_factor_blk(int N, int ld, T* A, int* rowof, T* diag, T* tmp, double& logdet, int& sign, Smem& S) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int PB = panel_width(N, S), ldp = panel_ld(N);
  T* P = reinterpret_cast<T*>(S.gemm);  // [PB][ldp], column-major
  T* U = P + PB * ldp;                  // [PB][<= N] rows of U12
  T* ud = reinterpret_cast<T*>(S.spare);  // [N] diagonal of U
  int* piv = S.ired + 16;               // [16] the panel's interchanges
  T* dinv_s = reinterpret_cast<T*>(S.xs + 6);
  int sg = 1;
  for (int i = tid; i < N; i += kThreads) rowof[i] = i;
  for (int k0 = 0; k0 < N; k0 += PB) {
    const int nb = (N - k0 < PB) ? N - k0 : PB, rows = N - k0, n2 = N - k0 - nb;
    for (int e = tid; e < rows * nb; e += kThreads) {
      const int r = e / nb, q = e - r * nb;
      P[q * ldp + r] = A[(size_t)(k0 + r) * ld + k0 + q];
    }
    __syncthreads();
    for (int c = 0; c < nb; ++c) {
      int bk = -1, bi = rows;
      for (int r = c + tid; r < rows; r += kThreads) {
        const int k = pivot_key(P[c * ldp + r]);
        if (k > bk) { bk = k; bi = r; }
      }
      const int wk = __reduce_max_sync(0xffffffffu, bk);
      const int wi = __reduce_min_sync(0xffffffffu, bk == wk ? bi : rows);
      if (lane == 0) { S.ired[warp] = wk; S.ired[8 + warp] = wi; }
      __syncthreads();
      int key = -1, p = rows;
#pragma unroll
      for (int w = 0; w < kThreads / 32; ++w) {
        const int k = S.ired[w], i = S.ired[8 + w];
        if (k > key || (k == key && i < p)) { key = k; p = i; }
      }
      if (key <= 0) return 1;
      const T d = P[c * ldp + p];
      if (p != c) sg = -sg;
      if (is_neg(d)) sg = -sg;
      __syncthreads();
      if (warp == 0) {
        if (lane == 0) {
          *dinv_s = quick_div(unit<T>(true), d);
          ud[k0 + c] = d;
        }
      } else if (warp == 1) {
        if (lane == 0) piv[c] = p;
        if (p != c) {
          for (int q = lane; q < nb; q += 32) {
            const T t = P[q * ldp + c];
            P[q * ldp + c] = P[q * ldp + p];
            P[q * ldp + p] = t;
          }
          if (lane == 0) {
            const int t = rowof[k0 + c];
            rowof[k0 + c] = rowof[k0 + p];
            rowof[k0 + p] = t;
          }
        }
      }
      __syncthreads();
      const T dinv = *dinv_s;
      if (tid == 0) diag[k0 + c] = dinv;
      for (int r = c + 1 + tid; r < rows; r += kThreads) {
        const T l = rmul(P[c * ldp + r], dinv);
        P[c * ldp + r] = l;
        const T ml = rneg(l);
        for (int q = c + 1; q < nb; ++q) P[q * ldp + r] = rfma(ml, P[q * ldp + c], P[q * ldp + r]);
      }
      __syncthreads();
    }
    for (int e = tid; e < rows * nb; e += kThreads) {
      const int r = e / nb, q = e - r * nb;
      A[(size_t)(k0 + r) * ld + k0 + q] = P[q * ldp + r];
    }
    // the panel's interchanges on the columns outside it (one thread per column)
    for (int j = tid; j < N; j += kThreads) {
      if (j >= k0 && j < k0 + nb) continue;
      for (int c = 0; c < nb; ++c) {
        const int p = k0 + piv[c];
        if (p != k0 + c) {
          const T t = A[(size_t)(k0 + c) * ld + j];
          A[(size_t)(k0 + c) * ld + j] = A[(size_t)p * ld + j];
          A[(size_t)p * ld + j] = t;
        }
      }
    }
    __syncthreads();
    if (n2 > 0) {
      // U12 = L11^-1 A12 column by column (L11 = P rows 0..nb-1)
      for (int jj = tid; jj < n2; jj += kThreads) {
        const int j = k0 + nb + jj;
        for (int q = 0; q < nb; ++q) {
          T u = A[(size_t)(k0 + q) * ld + j];
          for (int p2 = 0; p2 < q; ++p2) u = rfma(rneg(P[p2 * ldp + q]), U[p2 * n2 + jj], u);
          U[q * n2 + jj] = u;
          A[(size_t)(k0 + q) * ld + j] = u;
          tmp[(size_t)q * ld + jj] = rneg(u);
        }
      }
      __syncthreads();
      // A22 -= L21 U12
      gemm_acc(rows - nb, n2, nb, A + (size_t)(k0 + nb) * ld + k0, ld, tmp, ld, A + (size_t)(k0 + nb) * ld + k0 + nb,
               ld, S);
    }
  }
  double lg = 0.0;
  for (int k = tid; k < N; k += kThreads) lg += log(fabs(to_d(ud[k])));
  logdet = block_sum(lg, S.red);
  sign = sg;
  return 0;
}

// Solve (LU) X = B for all N columns of B, B already in interchanged row order
// (B <- X).  Blocks of PB rows are solved in shared memory, one thread per
// column; the rows beyond a block are updated by one accumulate-GEMM.  tmp: PB x N.
template <typename T>
__device__ void lu_solve_blk(int N, int ld, const T* LU, const T* diag, T* B, T* tmp, Smem& S) {
  const int tid = threadIdx.x;
  const int PB = panel_width(N, S);
  T* Y = reinterpret_cast<T*>(S.gemm);   // [PB][N] block of right-hand sides
  T* Lb = Y + PB * N;                    // [PB][PB] diagonal block
  for (int pass = 0; pass < 2; ++pass) {
    const int nblk = (N + PB - 1) / PB;
    for (int bi = 0; bi < nblk; ++bi) {
      // forward: blocks top to bottom; backward: bottom to top
      const int r0 = pass == 0 ? bi * PB : (nblk - 1 - bi) * PB;
      const int nb = (N - r0 < PB) ? N - r0 : PB;
      for (int e = tid; e < nb * nb; e += kThreads) {
        const int q = e / nb, p2 = e - q * nb;
        Lb[q * PB + p2] = rneg(LU[(size_t)(r0 + q) * ld + r0 + p2]);
      }
      for (int e = tid; e < nb * N; e += kThreads) {
        const int q = e / N, j = e - q * N;
        Y[q * N + j] = B[(size_t)(r0 + q) * ld + j];
      }
      __syncthreads();
      for (int j = tid; j < N; j += kThreads) {
        if (pass == 0) {
          for (int q = 1; q < nb; ++q) {
            T y = Y[q * N + j];
            for (int p2 = 0; p2 < q; ++p2) y = rfma(Lb[q * PB + p2], Y[p2 * N + j], y);
            Y[q * N + j] = y;
          }
        } else {
          for (int q = nb - 1; q >= 0; --q) {
            T y = Y[q * N + j];
            for (int p2 = q + 1; p2 < nb; ++p2) y = rfma(Lb[q * PB + p2], Y[p2 * N + j], y);
            Y[q * N + j] = rmul(y, diag[r0 + q]);
          }
        }
        for (int q = 0; q < nb; ++q) {
          const T y = Y[q * N + j];
          B[(size_t)(r0 + q) * ld + j] = y;
          tmp[(size_t)q * ld + j] = rneg(y);
        }
      }
      __syncthreads();
      if (pass == 0 && r0 + nb < N)
        gemm_acc(N - r0 - nb, N, nb, LU + (size_t)(r0 + nb) * ld + r0, ld, tmp, ld, B + (size_t)(r0 + nb) * ld, ld, S);
      if (pass == 1 && r0 > 0) gemm_acc(r0, N, nb, LU + r0, ld, tmp, ld, B, ld, S);
    }
  }
}

// The decomposition M = Q D T of M = X diag(src.D) src.T (X the product of a block of
// slices with src.Q, in W0 or W1): pivoted QR of X, D = |diag R_M|,
// T = D^-1 R_M P^T T_src with R_M,ij = R_X,ij dsc_j.  Result in (W2, wvec 0, W5), FP64;
// returns det(Q).
template <typename T>
__device__ int udv_of_product(const ChainDev& C, int s, T* X, UDV src, Smem& S, long long* det, long long t0) {
  const int N = C.N, ld = C.ld;
  double* Dn = wvec(C, s, 0);
  T* vk0 = reinterpret_cast<T*>(wvec(C, s, 2));
  double* dsc = wvec(C, s, 5);
  double* invr = wvec(C, s, 6);
  int* perm = C.iwork[s];
  T* tri = reinterpret_cast<T*>(wmat(C, s, 3));  // W3 and W4: about kPanel N entries
  const int detq = qr_blocked<T>(N, ld, X, src.D, perm, vk0, tri, S);
  T* Qn = reinterpret_cast<T*>(wmat(C, s, 2));
  form_q_blk<T>(N, ld, X, perm, vk0, tri, Qn, S);
  if constexpr (std::is_same<T, dd>::value) dd_to_d_inplace(N, ld, Qn);
  tick(det, 5, t0);
  T* PT = reinterpret_cast<T*>(wmat(C, s, 3));
  T* Rt = reinterpret_cast<T*>(wmat(C, s, 4));
  for (int x = threadIdx.x; x < N; x += kThreads) dsc[x] = src.D[perm[x]];
  __syncthreads();  // src.D may be the vector that takes the new D
  for (int x = threadIdx.x; x < N; x += kThreads) {
    const double rkk = fabs(to_d(X[(size_t)x * ld + perm[x]]));
    Dn[x] = rkk * dsc[x];
    invr[x] = (rkk > 0.0 && dsc[x] > 0.0) ? 1.0 / (rkk * dsc[x]) : 0.0;
  }
  __syncthreads();
  each_element(
      N, [&](int x, int y) { return src.T[(size_t)perm[x] * ld + y]; },
      [&](int x, int y, double v) { PT[(size_t)x * ld + y] = from_d<T>(v); });
  each_element(
      N, [&](int x, int y) { return X[(size_t)x * ld + perm[y]]; },
      [&](int x, int y, T v) {
        Rt[(size_t)x * ld + y] = y >= x ? rmul(v, from_d<T>(invr[x] * dsc[y])) : from_zero<T>();
      });
  T* Tn = reinterpret_cast<T*>(wmat(C, s, 5));
  if constexpr (std::is_same<T, dd>::value) {
    gemm_dd<false, false, false>(C, s, S, N, N, N, Rt, ld, PT, ld, Tn, ld);
    dd_to_d_inplace(N, ld, Tn);
  } else {
    gemm_64<false, false>(S, N, N, N, Rt, ld, PT, ld, Tn, ld);
  }
  tick(det, 6, t0);
  return detq;
}

// One-sided Jacobi SVD (Hestenes) of M = U S V^T, N x N in place: column
// pairs of M are rotated until mutually orthogonal (|m_p . m_q| <= 1e-15
// |m_p| |m_q| for every pair, at most 60 sweeps); then S_j = |m_j|, the
// columns of M are normalised to U (e_j for a zero column) and V holds the
// product of the rotations.  One-sided Jacobi keeps the relative accuracy of
// the small singular values of a column-scaled matrix, which is what the scale
// separation of the stable G needs.  The pairs of a sweep follow the
// round-robin (circle) schedule, N/2 disjoint pairs per round, one warp per
// pair; every warp sums its dot products in the same butterfly order, so the
// result does not depend on timing.
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ void svd_jacobi(int N, int ld, double* M, double* V, double* Sv) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int e = tid; e < N * N; e += kThreads) {
    const int x = e / N, y = e - x * N;
    V[(size_t)x * ld + y] = (x == y) ? 1.0 : 0.0;
  }
  __syncthreads();
  const int n = N + (N & 1);  // players of the schedule (a dummy when N is odd)
  for (int sweep = 0; sweep < 60; ++sweep) {
    int rotated = 0;
    for (int r = 0; r < n - 1; ++r) {
      for (int k = warp; k < n / 2; k += kThreads / 32) {
        int p = (k == 0) ? n - 1 : (r + k) % (n - 1);
        int q = (k == 0) ? r : (r - k + n - 1) % (n - 1);
        if (p > q) { const int t = p; p = q; q = t; }
        if (q >= N) continue;
        double a = 0.0, b = 0.0, c = 0.0;
        for (int i = lane; i < N; i += 32) {
          const double xp = M[(size_t)i * ld + p], xq = M[(size_t)i * ld + q];
          a = fma(xp, xp, a);
          b = fma(xq, xq, b);
          c = fma(xp, xq, c);
        }
        a = warp_sum(a);
        b = warp_sum(b);
        c = warp_sum(c);
        if (c == 0.0 || fabs(c) <= 1e-15 * sqrt(a * b)) continue;
        rotated = 1;
        const double zeta = (b - a) / (2.0 * c);
        const double t = (zeta >= 0.0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
        const double cs = 1.0 / sqrt(1.0 + t * t), sn = cs * t;
        for (int i = lane; i < N; i += 32) {
          double* mp = M + (size_t)i * ld + p;
          double* mq = M + (size_t)i * ld + q;
          const double xp = *mp, xq = *mq;
          *mp = cs * xp - sn * xq;
          *mq = sn * xp + cs * xq;
          double* vp = V + (size_t)i * ld + p;
          double* vq = V + (size_t)i * ld + q;
          const double yp = *vp, yq = *vq;
          *vp = cs * yp - sn * yq;
          *vq = sn * yp + cs * yq;
        }
      }
      __syncthreads();
    }
    if (!__syncthreads_or(rotated)) break;
  }
  for (int j = tid; j < N; j += kThreads) {
    double s2 = 0.0;
    for (int i = 0; i < N; ++i) s2 = fma(M[(size_t)i * ld + j], M[(size_t)i * ld + j], s2);
    Sv[j] = sqrt(s2);
  }
  __syncthreads();
  for (int e = tid; e < N * N; e += kThreads) {
    const int x = e / N, y = e - x * N;
    const double sj = Sv[y];
    M[(size_t)x * ld + y] = (sj > 0.0) ? M[(size_t)x * ld + y] / sj : (x == y ? 1.0 : 0.0);
  }
  __syncthreads();
}

// One step of a UDV chain (Sec. 2.3): X = Bcal Q_src, M = X D_src, M P = Q R,
// D = |diag R|, T = D^-1 R P^T T_src.  Right chain (left == false): Bcal =
// B_t2 ... B_t1+1.  Left chain: Bcal = B_t1+1^T ... B_t2^T.  Result in
// (W2, wvec 0, W5); returns det(Q).
__device__ int chain_step(const ChainDev& C, int s, int t1, int t2, bool left, UDV src, Smem& S,
                                       long long* det = nullptr) {
  long long t0 = clock64();
  const int N = C.N, ld = C.ld;
  double* X = wmat(C, s, 0);
  double* Y = wmat(C, s, 1);
  cta_copy(N, ld, src.Q, X);
  const double* E = C.E[s];
  if (!left) {
    for (int t = t1 + 1; t <= t2; ++t) {
      slice_potential_global(C, s, t, S.v);
      for (int x = threadIdx.x; x < N; x += kThreads) S.ev[x] = exp(S.v[x]);
      __syncthreads();
      each_element(
          N, [&](int x, int y) { return X[(size_t)x * ld + y]; },
          [&](int x, int y, double v) { X[(size_t)x * ld + y] = v * S.ev[x]; });
      gemm_64<false, false>(S, N, N, N, E, ld, X, ld, Y, ld, kCpEA, -1);
      double* t_ = X; X = Y; Y = t_;
    }
  } else {
    for (int t = t2; t >= t1 + 1; --t) {
      gemm_64<true, false>(S, N, N, N, E, ld, X, ld, Y, ld, kCpEtA, -1);
      slice_potential_global(C, s, t, S.v);
      for (int x = threadIdx.x; x < N; x += kThreads) S.ev[x] = exp(S.v[x]);
      __syncthreads();
      each_element(
          N, [&](int x, int y) { return Y[(size_t)x * ld + y]; },
          [&](int x, int y, double v) { Y[(size_t)x * ld + y] = v * S.ev[x]; });
      double* t_ = X; X = Y; Y = t_;
    }
  }
  tick(det, 4, t0);
  double* Dn = wvec(C, s, 0);
  if (C.stab_svd) {
    // M = X D_src
    for (int e = threadIdx.x; e < N * N; e += kThreads) {
      const int x = e / N, y = e - x * N;
      X[(size_t)x * ld + y] *= src.D[y];
    }
    __syncthreads();
    // M = U S V^T: Q = U, D = S, T = V^T T_src, det Q from an LU of U
    double* V = Y;
    svd_jacobi(N, ld, X, V, Dn);
    double* Qn = wmat(C, s, 2);
    double* Ucp = wmat(C, s, 3);
    for (int e = threadIdx.x; e < N * N; e += kThreads) {
      const int x = e / N, y = e - x * N;
      Qn[(size_t)x * ld + y] = X[(size_t)x * ld + y];
      Ucp[(size_t)x * ld + y] = X[(size_t)x * ld + y];
    }
    __syncthreads();
    double ldu;
    int detq = 1;
    if (lu_factor_blk(N, ld, Ucp, S.qinv, S.hv, wmat(C, s, 9), ldu, detq, S)) detq = 1;
    tick(det, 5, t0);
    gemm_64<true, false>(S, N, N, N, V, ld, src.T, ld, wmat(C, s, 5), ld);
    tick(det, 6, t0);
    return detq;
  }
  return udv_of_product<double>(C, s, X, src, S, det, t0);
}

// Stable G from a right chain R (B(tau,0) = Q_R D_R T_R) and a left chain Lf
// (B(beta,tau)^T = Q_L D_L T_L) by scale separation, D = Db Ds with
// Db = max(D,1), Ds = min(D,1):
//   Mid = Db_R^-1 Q_R^T Q_L Db_L^-1 + Ds_R (T_R T_L^T) Ds_L
//   G   = Q_L Db_L^-1 Mid^-1 Db_R^-1 Q_R^T
//   log|det G^-1| = sum log Db_R + sum log Db_L + log|det Mid|.
// Uses W0, W1; the result goes to Gout.  Returns nonzero if Mid is singular.
__device__ int green_from_udv(const ChainDev& C, int s, UDV R, UDV Lf, double* Gout, double& logdet,
                              int& sign, Smem& S) {
  const int N = C.N, ld = C.ld;
  double* W0 = wmat(C, s, 0);
  double* W1 = wmat(C, s, 1);
  gemm_64<true, false>(S, N, N, N, R.Q, ld, Lf.Q, ld, W0, ld);
  gemm_64<false, true>(S, N, N, N, R.T, ld, Lf.T, ld, W1, ld);
  // 1/Db and Ds of both chains (vectors 5..7 of the workspace)
  double* ibR = wvec(C, s, 5);
  double* ibL = wvec(C, s, 6);
  for (int i = threadIdx.x; i < N; i += kThreads) {
    ibR[i] = 1.0 / (R.D[i] > 1.0 ? R.D[i] : 1.0);
    ibL[i] = 1.0 / (Lf.D[i] > 1.0 ? Lf.D[i] : 1.0);
  }
  __syncthreads();
  each_element(
      N, [&](int i, int j) { return make_double2(W0[(size_t)i * ld + j], W1[(size_t)i * ld + j]); },
      [&](int i, int j, double2 v) {
        const double dR = R.D[i], dL = Lf.D[j];
        const double dsR = dR > 1.0 ? 1.0 : dR, dsL = dL > 1.0 ? 1.0 : dL;
        W0[(size_t)i * ld + j] = v.x * (ibR[i] * ibL[j]) + dsR * v.y * dsL;
      });
  double ldm;
  int sm;
  int* rowof = S.qinv;
  double* udiag = S.hv;
  double* tmp = wmat(C, s, 9);
  if (lu_factor_blk(N, ld, W0, rowof, udiag, tmp, ldm, sm, S)) return 1;
  each_element(
      N, [&](int i, int j) { return R.Q[(size_t)j * ld + rowof[i]]; },
      [&](int i, int j, double v) { W1[(size_t)i * ld + j] = v * ibR[rowof[i]]; });
  lu_solve_blk(N, ld, W0, udiag, W1, tmp, S);
  each_element(
      N, [&](int i, int j) { return W1[(size_t)i * ld + j]; },
      [&](int i, int j, double v) { W1[(size_t)i * ld + j] = v * ibL[i]; });
  gemm_64<false, false>(S, N, N, N, Lf.Q, ld, W1, ld, Gout, ld);
  double part = 0.0;
  for (int i = threadIdx.x; i < N; i += kThreads) {
    const double dR = R.D[i], dL = Lf.D[i];
    part += log(dR > 1.0 ? dR : 1.0) + log(dL > 1.0 ? dL : 1.0);
  }
  logdet = ldm + block_sum(part, S.red);
  sign = sm * R.detq * Lf.detq;
  return 0;
}

__device__ void copy_udv_to_slot(const ChainDev& C, int s, int j, int detq) {
  const int N = C.N, ld = C.ld;
  double* b = slot_base(C, s, j);
  cta_copy(N, ld, (const double*)wmat(C, s, 2), b);
  cta_copy(N, ld, (const double*)wmat(C, s, 5), b + (size_t)N * ld);
  const double* Dn = wvec(C, s, 0);
  for (int x = threadIdx.x; x < N; x += kThreads) b[(size_t)2 * N * ld + x] = Dn[x];
  if (threadIdx.x == 0) C.slot_detq[s][j] = detq;
  __syncthreads();
}

__device__ inline UDV work_udv(const ChainDev& C, int s, int detq) {
  UDV u;
  u.Q = wmat(C, s, 2);
  u.T = wmat(C, s, 5);
  u.D = wvec(C, s, 0);
  u.detq = detq;
  return u;
}

// Fill the storage with the left chain (Algorithm 1, the loop before the bins)
// and compute G(0) into W6.
__device__ int fill_left_chain(const ChainDev& C, int s, Smem& S, double& logdet, int& sign) {
  const int nst = C.L / C.nw;
  for (int j = nst - 1; j >= 0; --j) {
    const UDV src = (j + 1 == nst) ? ident_udv(C) : slot_udv(C, s, j + 1);
    const int dq = chain_step(C, s, j * C.nw, (j + 1) * C.nw, true, src, S);
    copy_udv_to_slot(C, s, j, dq);
  }
  return green_from_udv(C, s, ident_udv(C), slot_udv(C, s, 0), wmat(C, s, 6), logdet, sign, S);
}

// The float-pair stabilisation (defined with the mixed path below).
__device__ int chain_step_mixed(const ChainDev& C, int s, int t1, int t2, bool left, UDV src, Smem& S,
                                long long* det);
__device__ int green_from_udv_mixed(const ChainDev& C, int s, UDV R, UDV Lf, double* Gout, double& logdet,
                                    int& sign, Smem& S);

// Left chain and G(0) with the stabilisation arithmetic of the working
// precision: float pairs (FP64 scales) for the mixed paths, FP64 otherwise.
// Used when a chain starts or restarts from fields, so that the stored chain is
// the one the sweep itself would have left.
template <typename Real>
__device__ int fill_left_chain_working(const ChainDev& C, int s, Smem& S, double& logdet, int& sign) {
  if constexpr (std::is_same<Real, dd>::value) {
    const int nst = C.L / C.nw;
    for (int j = nst - 1; j >= 0; --j) {
      const UDV src = (j + 1 == nst) ? ident_udv(C) : slot_udv(C, s, j + 1);
      const int dq = chain_step_mixed(C, s, j * C.nw, (j + 1) * C.nw, true, src, S, nullptr);
      copy_udv_to_slot(C, s, j, dq);
    }
    return green_from_udv_mixed(C, s, ident_udv(C), slot_udv(C, s, 0), wmat(C, s, 6), logdet, sign, S);
  } else {
    return fill_left_chain(C, s, S, logdet, sign);
  }
}

// --------------------------------------------------------------------------
// Kernels templated on the working precision.
// --------------------------------------------------------------------------
// Fresh G(0) for every (chain, flavor): the left chain is (re)computed into the
// storage slots, G(0) lands in W6.  mode 0 (start from fields, in the working
// precision's stabilisation arithmetic): also write the working G, the
// fresh log|det| and the sign (initialisation); mode 1: copy G(0) of chain
// `out_chain` to `out` (FP64, [nfl][N][N]).
template <typename Real>
__global__ void __launch_bounds__(kThreads) fresh_green_kernel(ChainDev* chains, int n_chains, int mode,
                                                               double* out, int out_chain) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int nfl = chains[0].nfl;
  const int c = blockIdx.x / nfl, s = blockIdx.x % nfl;
  if (c >= n_chains) return;
  if (mode == 1 && c != out_chain) return;
  ChainDev& C = chains[c];
  Smem S = carve_smem(smem_raw, C.ld, C.MV);
  const bool pairs = std::is_same<Real, dd>::value && mode == 0;
  const bool umma = umma_begin(C, s, S, DQMC_WITH_UMMA && pairs, !pairs);
  double logdet;
  int sign;
  const int bad = (mode == 0) ? fill_left_chain_working<Real>(C, s, S, logdet, sign)
                              : fill_left_chain(C, s, S, logdet, sign);
  if (umma) umma_free(S.um);
  if (bad) {
    numerical_failure(C);
    return;
  }
  const double* Gf = wmat(C, s, 6);
  if (mode == 0) {
    Real* G = (Real*)C.G[s];
    for (int e = threadIdx.x; e < C.N * C.N; e += kThreads) {
      const int x = e / C.N, y = e - x * C.N;
      G[(size_t)x * C.ld + y] = from_d<Real>(Gf[(size_t)x * C.ld + y]);
    }
  } else {
    for (int e = threadIdx.x; e < C.N * C.N; e += kThreads) {
      const int x = e / C.N, y = e - x * C.N;
      out[(size_t)s * C.N * C.N + e] = Gf[(size_t)x * C.ld + y];
    }
  }
  if (threadIdx.x == 0) {
    C.logdet[s] = logdet;
    C.fresh_sign[s] = sign;
  }
}

// Hopping and potential wraps of one slice (defined with the sweep pieces below).
template <typename Real>
__device__ void v_wrap(const ChainDev& C, Real* G, const double* v, double a, Smem& S);
template <typename Real>
__device__ void t_wrap(const ChainDev& C, int s, Real* G, Real* Gt, bool up, Smem& S);

// G^s(tau) of one chain on its current fields as the upward pass of a sweep
// holds it when every proposal of the slices tau0+1..tau is rejected (Sec. 2.3,
// the wrapped Green function between stabilisations; Algorithm 1 wrapgrup):
// the stable G(tau0) at the last stabilisation point tau0 = n_wrap floor(tau /
// n_wrap), from the right chain B(tau0,0) built here and the stored left chain
// B(beta,tau0)^T, in the working precision's stabilisation arithmetic, then
// tau - tau0 wraps G <- E e^V G e^-V E^-1 in the working precision.  One CTA per
// flavor; the stored chain, the working G and the fields are only read.  Uses
// the work matrices W0..W8; out: [nfl][N][N] FP64.
template <typename Real>
__global__ void __launch_bounds__(kThreads) green_tau_kernel(ChainDev* chains, int chain, int tau, double* out) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  ChainDev& C = chains[chain];
  const int s = blockIdx.x;
  if (s >= C.nfl) return;
  Smem S = carve_smem(smem_raw, C.ld, C.MV);
  S.flavor = s;
  const int N = C.N, ld = C.ld, nw = C.nw, nst = C.L / nw;
  const int j0 = tau / nw;
  constexpr bool mixed = std::is_same<Real, dd>::value;
  const bool umma = umma_begin(C, s, S, DQMC_WITH_UMMA && mixed, !mixed);
  int dq = 1;
  for (int j = 1; j <= j0; ++j) {
    const UDV src = (j == 1) ? ident_udv(C) : work_udv(C, s, dq);
    dq = mixed ? chain_step_mixed(C, s, (j - 1) * nw, j * nw, false, src, S, nullptr)
               : chain_step(C, s, (j - 1) * nw, j * nw, false, src, S);
  }
  const UDV R = (j0 == 0) ? ident_udv(C) : work_udv(C, s, dq);
  const UDV Lf = (j0 >= nst) ? ident_udv(C) : slot_udv(C, s, j0);
  double* Gf = wmat(C, s, 6);
  double logdet;
  int sg;
  const int bad = mixed ? green_from_udv_mixed(C, s, R, Lf, Gf, logdet, sg, S)
                        : green_from_udv(C, s, R, Lf, Gf, logdet, sg, S);
  if (bad) {
    if (umma) umma_free(S.um);
    numerical_failure(C);
    return;
  }
  Real* G = reinterpret_cast<Real*>(wmat(C, s, 7));
  Real* Gt = reinterpret_cast<Real*>(wmat(C, s, 8));
  for (int e = threadIdx.x; e < N * N; e += kThreads) {
    const int x = e / N, y = e - x * N;
    G[(size_t)x * ld + y] = from_d<Real>(Gf[(size_t)x * ld + y]);
  }
  __syncthreads();
  for (int t = j0 * nw + 1; t <= tau; ++t) {
    slice_potential_global(C, s, t, S.v);
    v_wrap<Real>(C, G, S.v, +1.0, S);
    t_wrap<Real>(C, s, G, Gt, true, S);
  }
  if (umma) umma_free(S.um);
  for (int e = threadIdx.x; e < N * N; e += kThreads) {
    const int x = e / N, y = e - x * N;
    out[(size_t)s * N * N + e] = to_d(G[(size_t)x * ld + y]);
  }
}

template <typename Real>
__global__ void copy_green_kernel(ChainDev* chains, int chain, int flavor, double* out) {
  const ChainDev& C = chains[chain];
  const Real* G = (const Real*)C.G[flavor];
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < C.N * C.N; e += gridDim.x * blockDim.x) {
    const int x = e / C.N, y = e - x * C.N;
    out[e] = to_d(G[(size_t)x * C.ld + y]);
  }
}

// ---- pieces of the sweep --------------------------------------------------

// G <- diag(ev) G diag(1/ev)  with ev = exp(a v)
template <typename Real>
__device__ void v_wrap(const ChainDev& C, Real* G, const double* v, double a, Smem& S) {
  const int N = C.N, ld = C.ld;
  Real* evr = reinterpret_cast<Real*>(S.ev);
  Real* evi = reinterpret_cast<Real*>(S.hv);
  for (int x = threadIdx.x; x < N; x += kThreads) {
    evr[x] = from_d<Real>(exp(a * v[x]));
    evi[x] = from_d<Real>(exp(-a * v[x]));
  }
  __syncthreads();
  each_element(
      N, [&](int x, int y) { return G[(size_t)x * ld + y]; },
      [&](int x, int y, Real g) { G[(size_t)x * ld + y] = rmul(rmul(g, evr[x]), evi[y]); });
}

// Hopping wrap: up  G <- E G E^-1;  down  G <- E^-1 G E.
template <typename Real>
__device__ void t_wrap(const ChainDev& C, int s, Real* G, Real* Gt, bool up, Smem& S);

template <>
__device__ void t_wrap<double>(const ChainDev& C, int s, double* G, double* Gt, bool up, Smem& S) {
  const int N = C.N, ld = C.ld;
  const double* X = up ? C.E[s] : C.Einv[s];
  const double* Y = up ? C.Einv[s] : C.E[s];
  gemm_64<false, false>(S, N, N, N, X, ld, G, ld, Gt, ld, up ? kCpEA : kCpEiA, -1);
  gemm_64<false, false>(S, N, N, N, Gt, ld, Y, ld, G, ld, -1, up ? kCpEiB : kCpEB);
}
template <>
__device__ void t_wrap<float>(const ChainDev& C, int s, float* G, float* Gt, bool up, Smem& S) {
  const int N = C.N, ld = C.ld;
  const float* X = up ? C.E32[s] : C.Einv32[s];
  const float* Y = up ? C.Einv32[s] : C.E32[s];
  float* sm = reinterpret_cast<float*>(S.gemm);
  cta_gemm<float, false, false>(N, N, N, X, ld, G, ld, Gt, ld, sm);
  cta_gemm<float, false, false>(N, N, N, Gt, ld, Y, ld, G, ld, sm);
}

template <>
__device__ void t_wrap<dd>(const ChainDev& C, int s, dd* G, dd* Gt, bool up, Smem& S) {
  const int N = C.N, ld = C.ld;
  const dd* X = (const dd*)(up ? C.Edd[s] : C.Einvdd[s]);
  const dd* Y = (const dd*)(up ? C.Einvdd[s] : C.Edd[s]);
  gemm_dd<false, false, false>(C, s, S, N, N, N, X, ld, G, ld, Gt, ld, up ? kCpEA : kCpEiA, -1);
  gemm_dd<false, false, false>(C, s, S, N, N, N, Gt, ld, Y, ld, G, ld, -1, up ? kCpEiB : kCpEB);
}

// G += sum_m a_m b_m^T in float pairs: 16R x 16R tiles of G in registers, the vectors read
// where they are (shared memory, or the chain's arena).  The sums start from G, whose
// loads are the tile's only global reads, and keep its value and their error terms
// apart until the end (the products' scheme).  Instruction issue is the bound: 12 FP32
// operations per product and output, N^2 k 12 / 128 cycles per CTA.
template <int R>
__device__ void rank_update_dd(int N, int ld, dd* G, const dd* A, const dd* B, int nacc) {
  constexpr int TT = 16 * R;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  for (int m0 = 0; m0 < N; m0 += TT)
    for (int n0 = 0; n0 < N; n0 += TT) {
      int row[R], col[R];
      float h[R][R], l[R][R];
#pragma unroll
      for (int i = 0; i < R; ++i) {
        row[i] = min(m0 + ty * R + i, N - 1);
        col[i] = min(n0 + tx * R + i, N - 1);
      }
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j) {
          const dd g = G[(size_t)row[i] * ld + col[j]];
          h[i][j] = g.hi;
          l[i][j] = g.lo;
        }
#pragma unroll 2
      for (int m = 0; m < nacc; ++m) {
        dd a[R], b[R];
#pragma unroll
        for (int i = 0; i < R; ++i) a[i] = A[(size_t)m * ld + row[i]];
#pragma unroll
        for (int j = 0; j < R; ++j) b[j] = B[(size_t)m * ld + col[j]];
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
          for (int j = 0; j < R; ++j) {
            const float p = a[i].hi * b[j].hi;
            const float pe = fmaf(a[i].hi, b[j].hi, -p);
            const float t = h[i][j] + p;
            const float bb = t - h[i][j];
            const float te = (h[i][j] - (t - bb)) + (p - bb);
            h[i][j] = t;
            float lo = l[i][j] + (te + pe);
            lo = fmaf(a[i].hi, b[j].lo, lo);
            l[i][j] = fmaf(a[i].lo, b[j].hi, lo);
          }
      }
      // (clamped rows and columns repeat another thread's outputs and are not stored)
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j)
          if (m0 + ty * R + i < N && n0 + tx * R + j < N)
            G[(size_t)row[i] * ld + col[j]] = fast_two_sum(h[i][j], l[i][j]);
    }
  __syncthreads();
}

// G <- G + sum_m a_m b_m^T  (flush of the delayed rank-k update), a register-
// blocked product G += A^T B with A, B stored as rows a_m, b_m.
template <typename Real>
__device__ void flush_delayed(const ChainDev& C, Real* G, const Real* A, const Real* B, int nacc, Smem& S);

template <>
__device__ void flush_delayed<double>(const ChainDev& C, double* G, const double* A, const double* B, int nacc,
                                      Smem& S) {
  const int N = C.N, ld = C.ld;
  // depth nacc <= 64: the FP64 pipe's N^2 nacc / 1.65 cycles against the split
  // product's cost per output (N = 64, 16 vectors: 19 us on the pipe, 22 us split;
  // N = 144: 97 and 60 us)
  if (S.ps64 && N >= 96) {
    gemm_umma<double>(true, false, true, N, N, nacc, A, ld, B, ld, G, ld, S.ps64, S.expA, S.expB, S.um, -1, -1);
    return;
  }
  const int r = gemm_pick_r(N);
  if (r == 1) cta_gemm_r<double, true, false, 1, true>(N, N, nacc, A, ld, B, ld, G, ld, S.gemm);
  else if (r == 2) cta_gemm_r<double, true, false, 2, true>(N, N, nacc, A, ld, B, ld, G, ld, S.gemm);
  else if (r == 3) cta_gemm_r<double, true, false, 3, true>(N, N, nacc, A, ld, B, ld, G, ld, S.gemm);
  else if (r == 5) cta_gemm_r<double, true, false, 5, true>(N, N, nacc, A, ld, B, ld, G, ld, S.gemm);
  else cta_gemm_r<double, true, false, 4, true>(N, N, nacc, A, ld, B, ld, G, ld, S.gemm);
}
template <>
__device__ void flush_delayed<float>(const ChainDev& C, float* G, const float* A, const float* B, int nacc,
                                     Smem& S) {
  const int N = C.N, ld = C.ld;
  float* sm = reinterpret_cast<float*>(S.gemm);
  const int r = gemm_pick_r(N);
  if (r == 1) cta_gemm_r<float, true, false, 1, true>(N, N, nacc, A, ld, B, ld, G, ld, sm);
  else if (r == 2) cta_gemm_r<float, true, false, 2, true>(N, N, nacc, A, ld, B, ld, G, ld, sm);
  else if (r == 3) cta_gemm_r<float, true, false, 3, true>(N, N, nacc, A, ld, B, ld, G, ld, sm);
  else if (r == 5) cta_gemm_r<float, true, false, 5, true>(N, N, nacc, A, ld, B, ld, G, ld, sm);
  else cta_gemm_r<float, true, false, 4, true>(N, N, nacc, A, ld, B, ld, G, ld, sm);
}
// ... of vectors in the chain's arena, staged in shared memory panel by panel (out of line:
// its registers are not the sweep's).
__device__ __noinline__ void rank_update_staged_dd(int N, int ld, dd* G, const dd* A, const dd* B, int nacc, dd* sm,
                                                   int dd_tile) {
  gemm_dd_tiles<true, false, true>(N, N, nacc, A, ld, B, ld, G, ld, sm, dd_tile);
}
template <>
__device__ void flush_delayed<dd>(const ChainDev& C, dd* G, const dd* A, const dd* B, int nacc, Smem& S) {
  // Vectors that did not fit the shared memory (N = 400 from rank 32): read directly, every
  // thread waits for L2 vector by vector.  20 x 20, L = 20, 4 chains: 2033 ms a sweep
  // directly, 1578 staged; L = 200, 32 chains: flushes 9.6 and 3.3 s of 14.5 and 8.2 s.
  if (!__isShared(A)) {
    rank_update_staged_dd(C.N, C.ld, G, A, B, nacc, reinterpret_cast<dd*>(S.gemm), S.dd_tile);
    return;
  }
  // a rank-k update (k <= 64): the float-pair register tiles beat the split tensor-core
  // product, whose digit split and recombination cost O(N^2) whatever k
  int r = S.dd_tile;
  if (r != 3 && r != 4) {
    r = 4;
    for (int q = 3; q >= 1; --q)
      if (umma_pad(C.N, 16 * q) < umma_pad(C.N, 16 * r)) r = q;
  }
  if (r == 1) rank_update_dd<1>(C.N, C.ld, G, A, B, nacc);
  else if (r == 2) rank_update_dd<2>(C.N, C.ld, G, A, B, nacc);
  else if (r == 3) rank_update_dd<3>(C.N, C.ld, G, A, B, nacc);
  else rank_update_dd<4>(C.N, C.ld, G, A, B, nacc);
}

// Sequential single-field updates of one slice (Sec. 2.2.1) for this CTA's
// flavor, in windows of kWin consecutive positions of the visiting order.
//
// Decisions: the acceptances of a window depend on G only through its kWin x kWin
// block on the window's sites, for both flavors.  Each CTA publishes its flavor's
// block of the effective G once per window; then both CTAs run the same chain of
// decisions on both blocks in shared memory, updated by a rank-1 step per
// acceptance, so the flavors meet once per window instead of once per
// acceptance.  The first acceptance in visiting order is found by a ballot over
// the remaining positions' ratios, which is exactly the sequential Metropolis
// chain because rejected proposals leave G unchanged.  One warp per flavor follows
// the chain (the ratios of all lanes are renewed from the accepted flip's vectors
// alone, so it finds the next acceptance while the other warps renew the blocks).
// Vectors: afterwards the accepted flips' delayed vectors
//   a = -(delta/R_s) G_eff[:,i],  b = e_i - G_eff[i,:],  G_eff += a b^T
// are formed for all N sites at once, each thread carrying kVecChunk flips'
// sums of one column or row element through the earlier ones (no barrier between
// flips: the elements of earlier vectors at the window's sites come from the
// decisions).  They are flushed into G every delay_k acceptances.
//
// The bound is the serial chain per acceptance and the FP64 unit (a warp's FP64
// instruction holds its scheduler's unit for 65 cycles).  Per acceptance on GB300, one
// CTA per SM, N = 64: the decisions 1130 cycles in float pairs and 2460 in FP64, the
// vectors 580 and 920, the window's exchange 240; two cluster barriers, FP64 ratios,
// quotients and vectors of all N sites by every warp took 11000 and 5900.
constexpr int kWin = 32;       // positions per window: one warp lane each
constexpr int kWinAcc = 16;    // acceptances per window (the vectors' shared memory)
constexpr int kVecChunk = 8;   // flips whose vectors one thread forms together
static_assert(kMaxFlavors + 6 == kThreads / 32 && 6 * 6 >= kWin, "six warps renew a window's rows in six turns");
constexpr int kWinLd = kWin + 1;  // row stride of a block: rows and columns without bank conflicts

// Shared memory of a window: the idle product panels (S.gemm) and the QR's
// partial sums (S.qred).
template <typename Real>
struct Window {
  using Ratio = typename RatioOf<Real>::type;
  Real* E;        // [kMaxFlavors][kWin][kWinLd] the flavors' blocks of the effective G
  Ratio* d;       // [kWin] this flavor's diagonal
  Ratio* del;     // [kWin] exp(dv) - 1 of this flavor
  Ratio* Rs;      // [kMaxFlavors][kWin] ratios
  Real* a;        // [kMaxFlavors][kWin] the accepted site's delayed vectors on the window
  Real* b;
  Real* mfa;      // [kWinAcc] this flavor's -(delta/R_s) per acceptance
  int* ctl;       // [2] accepted position in the window (-1: none), R < 0
  int* at;        // [kWinAcc] window positions of the acceptances
  Real* sA;       // [kWinAcc][kWin] this flavor's a and b on the window, per acceptance
  Real* sB;
};
template <typename Real>
__device__ __forceinline__ Window<Real> window_of(const Smem& S) {
  Window<Real> w;
  double* p = S.gemm;
  constexpr int blk = kMaxFlavors * kWin * kWinLd;
  static_assert((blk + 2 * kWin + 3 * kMaxFlavors * kWin + 2 * kWinAcc + 1) * 8 <= kGemmRegionBytes,
                "the window's blocks fit the product panels");
  w.E = reinterpret_cast<Real*>(p); p += blk;
  using Ratio = typename RatioOf<Real>::type;
  w.d = reinterpret_cast<Ratio*>(p); p += kWin;
  w.del = reinterpret_cast<Ratio*>(p); p += kWin;
  w.Rs = reinterpret_cast<Ratio*>(p); p += kMaxFlavors * kWin;
  w.a = reinterpret_cast<Real*>(p); p += kMaxFlavors * kWin;
  w.b = reinterpret_cast<Real*>(p); p += kMaxFlavors * kWin;
  w.mfa = reinterpret_cast<Real*>(p); p += kWinAcc;
  w.ctl = reinterpret_cast<int*>(p); p += 1;
  w.at = reinterpret_cast<int*>(p);
  static_assert(2 * kWinAcc * kWin <= 8 * 128, "the window's vectors fit the QR's partial sums");
  w.sA = reinterpret_cast<Real*>(S.qred);
  w.sB = w.sA + kWinAcc * kWin;
  return w;
}

// One column (ROW = false: a) or row (ROW = true: b) element x of the vectors of
// the nb <= kVecChunk acceptances j0..j0+nb-1 of the window whose first position
// is pos; n0 vectors were pending before the window.  The sums run over the
// earlier vectors in order.
template <typename Real, bool ROW>
__device__ __forceinline__ void window_vectors(const Real* G, int ld, int x, int pos, int n0, int j0, int nb, Real* A,
                                               Real* B, const Window<Real>& w, const int* qsite) {
  Real e[kVecChunk];
  int f[kVecChunk], site[kVecChunk];
#pragma unroll
  for (int j = 0; j < kVecChunk; ++j) {
    f[j] = w.at[j0 + (j < nb ? j : 0)];
    site[j] = qsite[pos + f[j]];
    e[j] = ROW ? G[(size_t)site[j] * ld + x] : G[(size_t)x * ld + site[j]];
  }
  for (int m = 0; m < n0; ++m) {
    const Real v = ROW ? B[(size_t)m * ld + x] : A[(size_t)m * ld + x];
    const Real* other = (ROW ? A : B) + (size_t)m * ld;
#pragma unroll
    for (int j = 0; j < kVecChunk; ++j) e[j] = rfma(v, other[site[j]], e[j]);
  }
  for (int q = 0; q < j0; ++q) {
    const Real v = ROW ? B[(size_t)(n0 + q) * ld + x] : A[(size_t)(n0 + q) * ld + x];
    const Real* other = (ROW ? w.sA : w.sB) + q * kWin;
#pragma unroll
    for (int j = 0; j < kVecChunk; ++j) e[j] = rfma(v, other[f[j]], e[j]);
  }
#pragma unroll
  for (int j = 0; j < kVecChunk; ++j) {
    if (j >= nb) continue;
    const Real v = ROW ? rsub(unit<Real>(x == site[j]), e[j]) : rmul(w.mfa[j0 + j], e[j]);
    (ROW ? B : A)[(size_t)(n0 + j0 + j) * ld + x] = v;
    const Real* other = (ROW ? w.sA : w.sB) + (j0 + j) * kWin;
#pragma unroll
    for (int q = j + 1; q < kVecChunk; ++q) e[q] = rfma(v, other[f[q]], e[q]);
  }
}

template <typename Real>
__device__ void update_slice(ChainDev& C, int s, int tau, int dir, const SweepParams& P, Smem& S,
                             cg::cluster_group& cl, Real* G, Real* A, Real* B, int& sign, long long* det) {
  using Ratio = typename RatioOf<Real>::type;
  const int N = C.N, ld = C.ld, MV = C.MV, nfl = C.nfl, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  long long t0 = clock64();
  const uint32_t key0 = (uint32_t)P.seed, key1 = (uint32_t)(P.seed >> 32) ^ C.chain_id;
  Ratio* diag = reinterpret_cast<Ratio*>(S.d);
  Ratio* u2_q = reinterpret_cast<Ratio*>(S.u2);
  Ratio* delta_q = reinterpret_cast<Ratio*>(S.delta);
  Ratio* gam_q = reinterpret_cast<Ratio*>(S.gam);
  const Ratio one = unit<Ratio>(true);
  for (int x = tid; x < N; x += kThreads) {
    diag[x] = to_ratio(G[(size_t)x * ld + x], Ratio());
    S.qinv[x] = -1;
  }
  __syncthreads();
  for (int q = tid; q < MV; q += kThreads) {
    const int k = dir ? MV - 1 - q : q;
    uint32_t ctr[4] = {(uint32_t)P.sweep, (uint32_t)(2 * tau + dir), (uint32_t)k, (uint32_t)(P.sweep >> 32)};
    philox4x32_10(ctr, key0, key1);
    const double u1 = uniform53(ctr[0], ctr[1]);
    u2_q[q] = from_d<Ratio>(uniform53(ctr[2], ctr[3]));
    const int f = S.fslice[k];
    const int fn = propose_field(C.ft, f, u1);
    const double dc = coupling(C.ft, C.cscale, fn) - coupling(C.ft, C.cscale, f);
    delta_q[q] = from_d<Ratio>(exp(C.vsign[s * MV + k] * dc) - 1.0);
    gam_q[q] = from_d<Ratio>(field_weight(C.ft, fn) / field_weight(C.ft, f));
    S.fnew[q] = (int8_t)fn;
    S.qsite[q] = C.site[k];
    S.qinv[C.site[k]] = q;
  }
  __syncthreads();
  tick(det, 0, t0);
  const Window<Real> w = window_of<Real>(S);
  int pos = 0, nacc = 0;
  int64_t n_acc_slice = 0;
  const int kdel = P.delay_k;
  while (pos < MV) {
    const int W = (MV - pos < kWin) ? MV - pos : kWin;
    // ---- this flavor's block of the effective G, published to the peer
    {
      const int ic = S.qsite[pos + (lane < W ? lane : 0)];
      Real e[kWin / 8];
      int ir[kWin / 8];
#pragma unroll
      for (int j = 0; j < kWin / 8; ++j) {
        const int r = warp + 8 * j;
        ir[j] = S.qsite[pos + (r < W ? r : 0)];
        e[j] = G[(size_t)ir[j] * ld + ic];
      }
      for (int m = 0; m < nacc; ++m) {
        const Real bm = B[(size_t)m * ld + ic];
#pragma unroll
        for (int j = 0; j < kWin / 8; ++j)
          if (warp + 8 * j < W) e[j] = rfma(A[(size_t)m * ld + ir[j]], bm, e[j]);
      }
#pragma unroll
      for (int j = 0; j < kWin / 8; ++j) w.E[(s * kWin + warp + 8 * j) * kWinLd + lane] = e[j];
      if (warp == 0) {
        w.d[lane] = diag[ic];
        w.del[lane] = delta_q[pos + (lane < W ? lane : 0)];
      }
    }
    cl.sync();
    Ratio dw = one, delw = one;  // warp r: diagonal and delta of flavor r
    for (int r = 0; r < nfl; ++r) {
      if (r != s) {
        const Real* pe = cl.map_shared_rank(w.E, r) + r * kWin * kWinLd;
        Real* me = w.E + r * kWin * kWinLd;
#pragma unroll
        for (int j = 0; j < kWin / 8; ++j) me[(warp + 8 * j) * kWinLd + lane] = pe[(warp + 8 * j) * kWinLd + lane];
      }
      if (warp == r) {
        dw = ((r == s) ? w.d : cl.map_shared_rank(w.d, r))[lane];
        delw = ((r == s) ? w.del : cl.map_shared_rank(w.del, r))[lane];
        w.Rs[r * kWin + lane] = rfma(delw, rsub(one, dw), one);
      }
    }
    cl.sync();  // the peer has read this block; both flavors' blocks and ratios are in place
    const Ratio u2 = u2_q[pos + (lane < W ? lane : 0)], gam = gam_q[pos + (lane < W ? lane : 0)];
    const bool weighted = C.ft != 1;  // Ising fields: gamma = 1
    int last = -1, na = 0;
    // ---- decisions
    while (true) {
      // the flavors' warps: the next acceptance (both find the same) and its factor
      Real mf = unit<Real>(false);
      int f = -1;
      if (warp < nfl) {
        const Ratio Rw = w.Rs[warp * kWin + lane];
        Ratio R = (warp == 0) ? Rw : w.Rs[lane];
        if (weighted) R = rmul(gam, R);
        if (nfl == 2) R = rmul(R, (warp == 1) ? Rw : w.Rs[kWin + lane]);
        const bool ok = lane > last && lane < W && accepts(u2, R);
        const unsigned m = __ballot_sync(0xffffffffu, ok);
        f = m ? __ffs(m) - 1 : -1;
        const unsigned negs = __ballot_sync(0xffffffffu, is_neg(R));
        if (warp == 0 && lane == 0) {
          w.ctl[0] = f;
          w.ctl[1] = f >= 0 ? (int)((negs >> f) & 1u) : 0;
        }
        if (f >= 0) {
          // every lane the accepted position's quotient
          const Ratio df = shfl(delw, f), Rf = shfl(Rw, f);
          mf = rneg(ratio_to<Real>(quick_div(df, Rf)));
        }
      } else if (last >= 0 && warp >= kMaxFlavors) {
        // the other warps meanwhile: the rows after the last acceptance of the flavors'
        // blocks, each row by one of six warps (of a single flavor, warp 1 sits out)
        for (int r = 0; r < nfl; ++r) {
          const Real bc = w.b[r * kWin + lane];
          Real* blk = w.E + r * kWin * kWinLd + lane;
#pragma unroll
          for (int j = 0; j < 6; ++j) {
            const int row = last + 1 + (warp - kMaxFlavors) + 6 * j;
            if (row < W) blk[row * kWinLd] = rfma(w.a[r * kWin + row], bc, blk[row * kWinLd]);
          }
        }
      }
      __syncthreads();
      if (warp >= nfl) f = w.ctl[0];
      if (f < 0) break;
      if (w.ctl[1]) sign = -sign;
      if (warp < nfl) {
        const Real* blk = w.E + warp * kWin * kWinLd;
        const Real ax = rmul(mf, blk[lane * kWinLd + f]);
        const Real bx = rsub(unit<Real>(lane == f), blk[f * kWinLd + lane]);
        w.a[warp * kWin + lane] = ax;
        w.b[warp * kWin + lane] = bx;
        if (warp == s) {
          w.sA[na * kWin + lane] = ax;
          w.sB[na * kWin + lane] = bx;
          if (lane == 0) {
            w.mfa[na] = mf;
            w.at[na] = f;
          }
        }
        dw = rfma(to_ratio(ax, Ratio()), to_ratio(bx, Ratio()), dw);
        w.Rs[warp * kWin + lane] = rfma(delw, rsub(one, dw), one);
      } else if (tid == 64) {
        const int q = pos + f;
        S.fslice[dir ? MV - 1 - q : q] = S.fnew[q];
      }
      last = f;
      ++na;
      __syncthreads();
      if (na == kWinAcc || nacc + na == kdel) break;
    }
    // a window that stopped at its limit goes on behind its last acceptance
    const int next = (na == kWinAcc || nacc + na == kdel) ? pos + last + 1 : pos + W;
    tick(det, 1, t0);
    // ---- the accepted flips' vectors on all sites: columns, then rows
    if (na) {
      const int Np = (N + 31) / 32 * 32;
      for (int j0 = 0; j0 < na; j0 += kVecChunk) {
        const int nb = (na - j0 < kVecChunk) ? na - j0 : kVecChunk;
        for (int u = tid; u < 2 * Np; u += kThreads) {
          if (u < Np) {
            if (u < N) window_vectors<Real, false>(G, ld, u, pos, nacc, j0, nb, A, B, w, S.qsite);
          } else if (u - Np < N) {
            window_vectors<Real, true>(G, ld, u - Np, pos, nacc, j0, nb, A, B, w, S.qsite);
          }
        }
      }
      __syncthreads();
      // the diagonal on the sites still to be visited in this slice
      for (int x = tid; x < N; x += kThreads)
        if (S.qinv[x] >= next) {
          Ratio dx = diag[x];
          for (int m = nacc; m < nacc + na; ++m)
            dx = rfma(to_ratio(A[(size_t)m * ld + x], Ratio()), to_ratio(B[(size_t)m * ld + x], Ratio()), dx);
          diag[x] = dx;
        }
      nacc += na;
      n_acc_slice += na;
    }
    tick(det, 2, t0);
    if (nacc == kdel) {
      flush_delayed<Real>(C, G, A, B, nacc, S);
      nacc = 0;
      tick(det, 3, t0);
    }
    __syncthreads();
    pos = next;
  }
  if (nacc) flush_delayed<Real>(C, G, A, B, nacc, S);
  tick(det, 3, t0);
  if (s == 0 && tid == 0) {
    C.proposals += MV;
    C.accepted += n_acc_slice;
  }
}

// ---- stabilisation with float-float products (mixed path) ----------------
// Same steps as chain_step / green_from_udv in float pairs: the dense products (the B
// chain, T = D^-1 R P^T T, Q_R^T Q_L, T_R T_L^T, Q_L Y), the pivoted QR, Q, LU and
// triangular solves; the scales D and the pivots' norms are FP64, and the stored Q
// and T are widened to FP64.
__device__ int chain_step_mixed(const ChainDev& C, int s, int t1, int t2, bool left, UDV src, Smem& S,
                                             long long* det = nullptr) {
  long long t0 = clock64();
  const int N = C.N, ld = C.ld;
  dd* X = reinterpret_cast<dd*>(wmat(C, s, 0));
  dd* Y = reinterpret_cast<dd*>(wmat(C, s, 1));
  dd* evr = reinterpret_cast<dd*>(S.ev);
  to_dd_mat(N, ld, src.Q, X);
  const dd* E = (const dd*)C.Edd[s];
  if (!left) {
    for (int t = t1 + 1; t <= t2; ++t) {
      slice_potential_global(C, s, t, S.v);
      for (int x = threadIdx.x; x < N; x += kThreads) evr[x] = from_d<dd>(exp(S.v[x]));
      __syncthreads();
      each_element(
          N, [&](int x, int y) { return X[(size_t)x * ld + y]; },
          [&](int x, int y, dd v) { X[(size_t)x * ld + y] = dd_mul(v, evr[x]); });
      gemm_dd<false, false, false>(C, s, S, N, N, N, E, ld, X, ld, Y, ld, kCpEA, -1);
      dd* t_ = X; X = Y; Y = t_;
    }
  } else {
    for (int t = t2; t >= t1 + 1; --t) {
      gemm_dd<true, false, false>(C, s, S, N, N, N, E, ld, X, ld, Y, ld, kCpEtA, -1);
      slice_potential_global(C, s, t, S.v);
      for (int x = threadIdx.x; x < N; x += kThreads) evr[x] = from_d<dd>(exp(S.v[x]));
      __syncthreads();
      each_element(
          N, [&](int x, int y) { return Y[(size_t)x * ld + y]; },
          [&](int x, int y, dd v) { Y[(size_t)x * ld + y] = dd_mul(v, evr[x]); });
      dd* t_ = X; X = Y; Y = t_;
    }
  }
  tick(det, 4, t0);
  return udv_of_product<dd>(C, s, X, src, S, det, t0);
}

__device__ int green_from_udv_mixed(const ChainDev& C, int s, UDV R, UDV Lf, double* Gout, double& logdet,
                                    int& sign, Smem& S) {
  const int N = C.N, ld = C.ld;
  dd* W0d = reinterpret_cast<dd*>(wmat(C, s, 0));
  dd* W1d = reinterpret_cast<dd*>(wmat(C, s, 1));
  dd* QRd = reinterpret_cast<dd*>(wmat(C, s, 3));
  dd* QLd = reinterpret_cast<dd*>(wmat(C, s, 4));
  dd* TRd = reinterpret_cast<dd*>(wmat(C, s, 7));
  dd* TLd = reinterpret_cast<dd*>(wmat(C, s, 8));
  to_dd_mat(N, ld, R.Q, QRd);
  to_dd_mat(N, ld, Lf.Q, QLd);
  to_dd_mat(N, ld, R.T, TRd);
  to_dd_mat(N, ld, Lf.T, TLd);
  gemm_dd<true, false, false>(C, s, S, N, N, N, QRd, ld, QLd, ld, W0d, ld);
  gemm_dd<false, true, false>(C, s, S, N, N, N, TRd, ld, TLd, ld, W1d, ld);
  double* ibR = wvec(C, s, 5);
  double* ibL = wvec(C, s, 6);
  for (int i = threadIdx.x; i < N; i += kThreads) {
    ibR[i] = 1.0 / (R.D[i] > 1.0 ? R.D[i] : 1.0);
    ibL[i] = 1.0 / (Lf.D[i] > 1.0 ? Lf.D[i] : 1.0);
  }
  __syncthreads();
  // Mid (float pairs, scale factors applied in FP64) in W0; right-hand side in W1
  struct Pair { dd q, t; };
  each_element(
      N, [&](int i, int j) { return Pair{W0d[(size_t)i * ld + j], W1d[(size_t)i * ld + j]}; },
      [&](int i, int j, Pair v) {
        const double dR = R.D[i], dL = Lf.D[j];
        const double dsR = dR > 1.0 ? 1.0 : dR, dsL = dL > 1.0 ? 1.0 : dL;
        W0d[(size_t)i * ld + j] = from_d<dd>(to_d(v.q) * (ibR[i] * ibL[j]) + dsR * to_d(v.t) * dsL);
      });
  double ldm;
  int smi;
  int* rowof = S.qinv;
  dd* udiag = reinterpret_cast<dd*>(S.hv);
  dd* tmpd = reinterpret_cast<dd*>(wmat(C, s, 9));
  if (lu_factor_blk(N, ld, W0d, rowof, udiag, tmpd, ldm, smi, S)) return 1;
  // right-hand side Db_R^-1 Q_R^T with the LU row interchanges applied
  each_element(
      N, [&](int i, int j) { return R.Q[(size_t)j * ld + rowof[i]]; },
      [&](int i, int j, double v) { W1d[(size_t)i * ld + j] = from_d<dd>(v * ibR[rowof[i]]); });
  lu_solve_blk(N, ld, W0d, udiag, W1d, tmpd, S);
  dd* Yd = reinterpret_cast<dd*>(wmat(C, s, 9));
  each_element(
      N, [&](int i, int j) { return W1d[(size_t)i * ld + j]; },
      [&](int i, int j, dd v) { Yd[(size_t)i * ld + j] = from_d<dd>(to_d(v) * ibL[i]); });
  gemm_dd<false, false, false>(C, s, S, N, N, N, QLd, ld, Yd, ld, reinterpret_cast<dd*>(Gout), ld);
  dd_to_d_inplace(N, ld, Gout);
  double part = 0.0;
  for (int i = threadIdx.x; i < N; i += kThreads) {
    const double dR = R.D[i], dL = Lf.D[i];
    part += log(dR > 1.0 ? dR : 1.0) + log(dL > 1.0 ? dL : 1.0);
  }
  logdet = ldm + block_sum(part, S.red);
  sign = smi * R.detq * Lf.detq;
  return 0;
}

// Stabilisation event of this CTA's flavor at slice tau: new chain, fresh G,
// precision monitor, working G replaced, storage slot j written.
template <typename Real>
__device__ void stabilise(ChainDev& C, int s, int j, bool up, Real* G, Smem& S, double& ev_max,
                          double& ev_sum, int& fresh_sign, long long* det) {
  long long t0 = clock64();
  const int N = C.N, ld = C.ld, nst = C.L / C.nw, nw = C.nw;
  int dq;
  UDV R, Lf;
  constexpr bool mixed = std::is_same<Real, dd>::value;
  if (up) {
    const UDV src = (j == 1) ? ident_udv(C) : slot_udv(C, s, j - 1);
    dq = mixed ? chain_step_mixed(C, s, (j - 1) * nw, j * nw, false, src, S, det)
               : chain_step(C, s, (j - 1) * nw, j * nw, false, src, S, det);
    R = work_udv(C, s, dq);
    Lf = (j == nst) ? ident_udv(C) : slot_udv(C, s, j);
  } else {
    const UDV src = (j + 1 == nst) ? ident_udv(C) : slot_udv(C, s, j + 1);
    dq = mixed ? chain_step_mixed(C, s, j * nw, (j + 1) * nw, true, src, S, det)
               : chain_step(C, s, j * nw, (j + 1) * nw, true, src, S, det);
    Lf = work_udv(C, s, dq);
    R = (j == 0) ? ident_udv(C) : slot_udv(C, s, j);
  }
  t0 = clock64();
  double* Gf = wmat(C, s, 6);
  double logdet;
  int sg;
  const int bad = mixed ? green_from_udv_mixed(C, s, R, Lf, Gf, logdet, sg, S)
                        : green_from_udv(C, s, R, Lf, Gf, logdet, sg, S);
  if (bad) {
    numerical_failure(C);
    sg = 1;
  }
  tick(det, 7, t0);
  double mx = 0.0, sm = 0.0;
  struct Both { double fresh; Real wrapped; };
  each_element(
      N, [&](int x, int y) { return Both{Gf[(size_t)x * ld + y], G[(size_t)x * ld + y]}; },
      [&](int x, int y, Both v) {
        const double dg = fabs(v.fresh - to_d(v.wrapped));
        mx = fmax(mx, dg);
        sm += dg;
        G[(size_t)x * ld + y] = from_d<Real>(v.fresh);
      });
  ev_max = block_max(mx, S.red);
  ev_sum = block_sum(sm, S.red);
  fresh_sign = sg;
  if (threadIdx.x == 0) {
    C.logdet[s] = logdet;
    C.fresh_sign[s] = sg;
  }
  copy_udv_to_slot(C, s, j, dq);
}

// Energy estimator at the current G (Sec. 6 observables, U n_up n_dn form).
template <typename Real>
__device__ void measure(ChainDev& C, int s, const Real* G, Smem& S, cg::cluster_group& cl, int sign) {
  const int N = C.N, ld = C.ld;
  const double* K = C.K[s];
  double kin = 0.0, part = 0.0;
  for (int e = threadIdx.x; e < N * N; e += kThreads) {
    const int x = e / N, y = e - x * N;
    kin += K[(size_t)x * ld + y] * ((x == y ? 1.0 : 0.0) - to_d(G[(size_t)y * ld + x]));
  }
  for (int x = threadIdx.x; x < N; x += kThreads) {
    const double gxx = to_d(G[(size_t)x * ld + x]);
    part += 1.0 - gxx;
    S.xdiag[x] = gxx;
  }
  kin = block_sum(kin, S.red);
  part = block_sum(part, S.red);
  if (threadIdx.x == 0) { S.xs[0] = kin; S.xs[1] = part; }
  cl.sync();
  if (s == 0) {
    double pot = 0.0;
    if (C.nfl == 2) {
      const double* pd = cl.map_shared_rank(S.xdiag, 1);
      for (int x = threadIdx.x; x < N; x += kThreads) pot += C.U * (1.0 - S.xdiag[x]) * (1.0 - pd[x]);
    }
    pot = block_sum(pot, S.red);
    double kin_t = S.xs[0], part_t = S.xs[1];
    if (C.nfl == 2) {
      const double* px = cl.map_shared_rank(S.xs, 1);
      kin_t += px[0];
      part_t += px[1];
    }
    if (threadIdx.x == 0) {
      const double sg = (double)sign;
      C.meas[0] += sg * kin_t;
      C.meas[1] += sg * pot;
      C.meas[2] += sg * part_t;
      C.meas[3] += sg * (kin_t + pot);
      C.meas_sign += sg;
      C.n_meas += 1;
    }
  }
  cl.sync();
}

// Exchange this flavor's fresh sign and precision figures; returns the product
// of the fresh signs.  Rank 0 books the event.
__device__ int close_event(ChainDev& C, int s, Smem& S, cg::cluster_group& cl, double ev_max, double ev_sum,
                           int fresh_sign, int sign) {
  if (threadIdx.x == 0) S.xs[2] = (double)fresh_sign;
  cl.sync();
  int prod = 1;
  for (int r = 0; r < C.nfl; ++r) {
    const double* px = (r == s) ? S.xs : cl.map_shared_rank(S.xs, r);
    prod *= (px[2] < 0.0) ? -1 : 1;
  }
  if (threadIdx.x == 0) {
    C.prec_sum[s] += ev_sum / ((double)C.N * C.N * C.nfl);
    C.prec_max[s] = fmax(C.prec_max[s], ev_max);
    if (s == 0) {
      C.phase_max = fmax(C.phase_max, fabs((double)prod - (double)sign));
      C.prec_events += 1;
    }
  }
  cl.sync();
  return prod;
}

// One sweep of every chain (Algorithm 1, upward then downward).
template <typename Real>
__global__ void __launch_bounds__(kThreads, 2) sweep_kernel(ChainDev* chains, SweepParams P) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  cg::cluster_group cl = cg::this_cluster();
  const int nfl = (int)cl.num_blocks();
  const int s = (int)cl.block_rank();
  const int c = P.order[blockIdx.x / nfl];
  ChainDev& C = chains[c];
  Smem S = carve_smem(smem_raw, C.ld, C.MV);
  S.flavor = s;
  // the split tensor-core products need the CTA's tensor memory for the whole sweep
  const bool umma = umma_begin(C, s, S, DQMC_WITH_UMMA && std::is_same<Real, dd>::value,
                               !std::is_same<Real, dd>::value);
  Real* G = (Real*)C.G[s];
  Real* Gt = (Real*)C.Gtmp[s];
  Real* A = P.ab_smem ? reinterpret_cast<Real*>(S.ab) : (Real*)C.dA[s];
  Real* B = P.ab_smem ? A + (size_t)P.delay_k * C.ld : (Real*)C.dB[s];
  const int L = C.L, nw = C.nw, MV = C.MV;
  int sign = C.sign;
  // thread 0's phase counters: cyc[0..3] per phase, det[0..7] per sub-phase
  long long* cyc = reinterpret_cast<long long*>(smem_raw);
  long long* det = cyc + 4;
  if (threadIdx.x == 0)
    for (int q = 0; q < 12; ++q) cyc[q] = 0;
  long long t0 = clock64();
  auto lap = [&](int phase) {
    const long long t1 = clock64();
    if (threadIdx.x == 0) cyc[phase] += t1 - t0;
    t0 = t1;
  };
  for (int tau = 1; tau <= L; ++tau) {
    for (int k = threadIdx.x; k < MV; k += kThreads) S.fslice[k] = C.fields[(size_t)(tau - 1) * MV + k];
    __syncthreads();
    slice_potential_smem(C, s, S.fslice, S.v);
    v_wrap<Real>(C, G, S.v, +1.0, S);
    lap(1);
    update_slice<Real>(C, s, tau, 0, P, S, cl, G, A, B, sign, det);
    if (s == 0)
      for (int k = threadIdx.x; k < MV; k += kThreads) C.fields[(size_t)(tau - 1) * MV + k] = S.fslice[k];
    lap(0);
    t_wrap<Real>(C, s, G, Gt, true, S);
    lap(1);
    if (tau % nw == 0) {
      cl.sync();
      double mx, sm;
      int fs;
      stabilise<Real>(C, s, tau / nw, true, G, S, mx, sm, fs, det);
      sign = close_event(C, s, S, cl, mx, sm, fs, sign);
      lap(2);
    }
    if (P.measure && tau >= P.meas_first && tau <= P.meas_last) {
      measure<Real>(C, s, G, S, cl, sign);
      lap(3);
    }
  }
  for (int tau = L; tau >= 1; --tau) {
    for (int k = threadIdx.x; k < MV; k += kThreads) S.fslice[k] = C.fields[(size_t)(tau - 1) * MV + k];
    __syncthreads();
    t_wrap<Real>(C, s, G, Gt, false, S);
    lap(1);
    update_slice<Real>(C, s, tau, 1, P, S, cl, G, A, B, sign, det);
    if (s == 0)
      for (int k = threadIdx.x; k < MV; k += kThreads) C.fields[(size_t)(tau - 1) * MV + k] = S.fslice[k];
    lap(0);
    slice_potential_smem(C, s, S.fslice, S.v);
    v_wrap<Real>(C, G, S.v, -1.0, S);
    lap(1);
    const int t0s = tau - 1;
    if (t0s % nw == 0) {
      cl.sync();
      double mx, sm;
      int fs;
      stabilise<Real>(C, s, t0s / nw, false, G, S, mx, sm, fs, det);
      sign = close_event(C, s, S, cl, mx, sm, fs, sign);
      lap(2);
    }
    if (P.measure && t0s >= P.meas_first && t0s <= P.meas_last) {
      measure<Real>(C, s, G, S, cl, sign);
      lap(3);
    }
  }
  cl.sync();
  if (umma) umma_free(S.um);
  if (threadIdx.x == 0) {
    for (int q = 0; q < 4; ++q) C.cyc[s][q] += cyc[q];
    for (int q = 0; q < 8; ++q) C.cycd[s][q] += det[q];
    if (s == 0) {
      C.sign = sign;
      C.sweep_sign_sum += (double)sign;
    }
  }
}

// --------------------------------------------------------------------------
// Launch helpers (instantiated once per precision unit).
// --------------------------------------------------------------------------
// The kernel may be launched with up to the architecture's shared memory: the same value
// in every call, as the attribute is the kernel's, not the launch's, and another thread
// may be between its own call and its launch.
static inline cudaError_t set_smem(const void* fn, size_t bytes) {
  if (bytes > kMaxSmemBytes) return cudaErrorInvalidValue;
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmemBytes);
}

template <typename Real>
static cudaError_t launch_fresh_green_t(ChainDev* chains, int n_chains, int nfl, size_t smem, int mode,
                                        double* out, int out_chain, cudaStream_t st) {
  cudaError_t e = set_smem((const void*)fresh_green_kernel<Real>, smem);
  if (e != cudaSuccess) return e;
  fresh_green_kernel<Real><<<n_chains * nfl, kThreads, smem, st>>>(chains, n_chains, mode, out, out_chain);
  return cudaGetLastError();
}

template <typename Real>
static cudaError_t launch_green_tau_t(ChainDev* chains, int chain, int nfl, size_t smem, int tau, double* out,
                                      cudaStream_t st) {
  cudaError_t e = set_smem((const void*)green_tau_kernel<Real>, smem);
  if (e != cudaSuccess) return e;
  green_tau_kernel<Real><<<nfl, kThreads, smem, st>>>(chains, chain, tau, out);
  return cudaGetLastError();
}

template <typename Real>
static cudaError_t launch_sweep_t(ChainDev* chains, const SweepParams& p, int nfl, size_t smem,
                                  cudaStream_t st) {
  cudaError_t e = set_smem((const void*)sweep_kernel<Real>, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.n_chains * nfl, 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = nfl;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, sweep_kernel<Real>, chains, p);
}

// Time-displaced Green functions from the two chains, sharing the middle
// matrix of the stable G (Sec. 2.1 observables, two times):
//   G(tau,0) = Q_L Db_L^-1 Mid^-1 Ds_R T_R,
//   G(0,tau) = -T_L^T Ds_L Mid^-1 Db_R^-1 Q_R^T.
// Uses W0, W1, W7, W8.  Returns nonzero if Mid is singular.
__device__ int displaced_from_udv(const ChainDev& C, int s, UDV R, UDV Lf, double* Gt0, double* G0t, Smem& S) {
  const int N = C.N, ld = C.ld;
  double* W0 = wmat(C, s, 0);
  double* W1 = wmat(C, s, 1);
  double* W7 = wmat(C, s, 7);
  double* W8 = wmat(C, s, 8);
  gemm_64<true, false>(S, N, N, N, R.Q, ld, Lf.Q, ld, W0, ld);
  gemm_64<false, true>(S, N, N, N, R.T, ld, Lf.T, ld, W1, ld);
  for (int e = threadIdx.x; e < N * N; e += kThreads) {
    const int i = e / N, j = e - i * N;
    const double dR = R.D[i], dL = Lf.D[j];
    const double dbR = dR > 1.0 ? dR : 1.0, dsR = dR > 1.0 ? 1.0 : dR;
    const double dbL = dL > 1.0 ? dL : 1.0, dsL = dL > 1.0 ? 1.0 : dL;
    W0[(size_t)i * ld + j] = W0[(size_t)i * ld + j] / (dbR * dbL) + dsR * W1[(size_t)i * ld + j] * dsL;
  }
  __syncthreads();
  double ldm;
  int smi;
  int* rowof = S.qinv;
  double* udiag = S.hv;
  double* tmp = wmat(C, s, 9);
  if (lu_factor_blk(N, ld, W0, rowof, udiag, tmp, ldm, smi, S)) return 1;
  for (int e = threadIdx.x; e < N * N; e += kThreads) {
    const int i = e / N, j = e - i * N;
    W1[(size_t)i * ld + j] = (rowof[i] == j) ? 1.0 : 0.0;
  }
  __syncthreads();
  lu_solve_blk(N, ld, W0, udiag, W1, tmp, S);  // W1 = Mid^-1
  for (int e = threadIdx.x; e < N * N; e += kThreads) {
    const int i = e / N, j = e - i * N;
    const double m = W1[(size_t)i * ld + j];
    const double dLi = Lf.D[i], dRj = R.D[j];
    W7[(size_t)i * ld + j] = m / (dLi > 1.0 ? dLi : 1.0) * (dRj > 1.0 ? 1.0 : dRj);
    W8[(size_t)i * ld + j] = (dLi > 1.0 ? 1.0 : dLi) * m / (dRj > 1.0 ? dRj : 1.0);
  }
  __syncthreads();
  gemm_64<false, false>(S, N, N, N, Lf.Q, ld, W7, ld, W0, ld);
  gemm_64<false, false>(S, N, N, N, W0, ld, R.T, ld, Gt0, ld);
  gemm_64<true, false>(S, N, N, N, Lf.T, ld, W8, ld, W0, ld);
  gemm_64<false, true>(S, N, N, N, W0, ld, R.Q, ld, G0t, ld);
  for (int e = threadIdx.x; e < N * N; e += kThreads) {
    const int i = e / N, j = e - i * N;
    G0t[(size_t)i * ld + j] = -G0t[(size_t)i * ld + j];
  }
  __syncthreads();
  return 0;
}

}  // namespace

size_t get_smem_bytes();  // dynamic shared memory of the fresh-G / adjoint / measurement kernels

// One pair per precision unit: 0 = FP64, 1 = FP32, 2/3 = float-pair (mixed).
cudaError_t launch_sweep_fp64(ChainDev* chains, const SweepParams& p, int nfl, size_t smem, cudaStream_t st);
cudaError_t launch_sweep_fp32(ChainDev* chains, const SweepParams& p, int nfl, size_t smem, cudaStream_t st);
cudaError_t launch_sweep_mixed(ChainDev* chains, const SweepParams& p, int nfl, size_t smem, cudaStream_t st);
cudaError_t launch_fresh_green_fp64(ChainDev* chains, int n_chains, int nfl, size_t smem, int mode, double* out,
                                    int out_chain, cudaStream_t st);
cudaError_t launch_fresh_green_fp32(ChainDev* chains, int n_chains, int nfl, size_t smem, int mode, double* out,
                                    int out_chain, cudaStream_t st);
cudaError_t launch_fresh_green_mixed(ChainDev* chains, int n_chains, int nfl, size_t smem, int mode, double* out,
                                     int out_chain, cudaStream_t st);
cudaError_t launch_green_tau_fp64(ChainDev* chains, int chain, int nfl, size_t smem, int tau, double* out,
                                  cudaStream_t st);
cudaError_t launch_green_tau_fp32(ChainDev* chains, int chain, int nfl, size_t smem, int tau, double* out,
                                  cudaStream_t st);
cudaError_t launch_green_tau_mixed(ChainDev* chains, int chain, int nfl, size_t smem, int tau, double* out,
                                   cudaStream_t st);
cudaError_t launch_sweep_mixed_tc(ChainDev* chains, const SweepParams& p, int nfl, size_t smem, cudaStream_t st);
cudaError_t launch_fresh_green_mixed_tc(ChainDev* chains, int n_chains, int nfl, size_t smem, int mode, double* out,
                                        int out_chain, cudaStream_t st);
cudaError_t launch_green_tau_mixed_tc(ChainDev* chains, int chain, int nfl, size_t smem, int tau, double* out,
                                      cudaStream_t st);

}  // namespace dqmc
