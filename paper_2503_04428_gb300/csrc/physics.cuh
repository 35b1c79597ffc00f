// physics.cuh -- per-cell and per-face device arithmetic of the Godunov update.
//
// Ideal-gas EoS (HERACLES++ Sect. 2.3 Eq. 5), physical fluxes of the Euler
// system (Sect. 2.1 Eq. 1), slope limiters (Sect. 3.2 Eq. 17), HLL/HLLC
// Riemann solvers (Sect. 3.2, Toro 2009 ch. 10), the exact Riemann solver
// (App. C.1, Toro 2009 ch. 4) and the MLP star-pressure guess.
//
// Vectors are register arrays of compile-time length NV = 2 + D + NSX:
// (rho, u_1..u_D, P, f_1..f_NSX) for primitives and (rho, m_1..m_D, E,
// rho f_1..rho f_NSX) for conserved variables.  Scalars beyond the run's
// actual count are carried as zeros and never stored.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

namespace hydro {

enum { LIM_FIRST = 0, LIM_MINMOD = 1, LIM_VANLEER = 2, LIM_VANALBADA = 3 };
enum { RS_HLL = 0, RS_HLLC = 1, RS_EXACT = 2 };
enum { ST_OK = 0, ST_NEG = -3, ST_NONFINITE = -4, ST_NEWTON = -5, ST_VACUUM = -8 };

// Gas constants precomputed on the host (double) and passed by value.
// Gas<T> is the ideal gas of Eq. 5.
template <typename T>
struct Gas {
  static constexpr bool RAD = false;
  T g;        // gamma
  T gm1;      // gamma - 1
  T igm1;     // 1/(gamma - 1)
  T z;        // (gamma - 1)/(2 gamma)
  T iz;       // 1/z
  T zp;       // (gamma + 1)/(2 gamma)
  T A2;       // 2/(gamma + 1)
  T Bq;       // (gamma - 1)/(gamma + 1)
  T two_gm1;  // 2/(gamma - 1)
  T ig;       // 1/gamma
  int root;   // 1/z if that is one of 4, ..., 8 (gamma = 2, 5/3, 3/2, 7/5, 4/3), else 0
};

// FP64 on this part: one warp instruction occupies an SM's FP64 pipe for 19
// cycles (measured; DFMA, DADD, DMUL and the compares alike, whatever the
// active lanes), an integer instruction an ALU for about half a cycle.  So
// the FP64 forms below count FP64 operations: signs and orders are read from
// the bit patterns, and reciprocals, quotients and square roots take Newton
// steps (error e -> O(e^2)) from the documented PTX approximations, whose
// relative error is below 2^-18, the last one with the residual of the
// unrounded result (Markstein, Computation of elementary functions on the IBM
// RISC System/6000 processor, 1990): 4, 5 and 6 FP64 operations against 4.5,
// 7.5 and 7.5 of the operators, which they equal but for results within ~2^-20
// of an ulp of the middle between two numbers.  (One third-order step each took
// 3, 4 and 5, with errors of 0.501, 1.5 and 1 ulp: Sedov 128^3 9.06 ms per 3
// steps against 9.46, Sod 1000 8.5 us per step against 8.9.)

// FP32 takes the hardware approximations (1-2 ulp; the FP32 bulk's rounding
// error is ~1e-7 per operation either way) in their .ftz forms: the others
// guard subnormal arguments with four more instructions each, a fifth of the
// exact solver's stream (guarded reciprocals alone: exact 101 x 67 x 53 1.18 ->
// 1.41 ms, Sedov 256^3 9.3 -> 10.0, radiation wedge 4.5 -> 5.1).  What they gain
// is a factor of 4 at the bottom of the range: a reciprocal overflows below
// 2^-128 in any form, and here below 2^-126, where it is infinite and ends the
// step with an error.

__device__ __forceinline__ bool is_zero(double x) {
  return ((__double2hiint(x) & 0x7fffffff) | __double2loint(x)) == 0;
}
__device__ __forceinline__ double rcp_estimate(double x) {  // to ~2^-36
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  return fma(r, fma(-x, r, 1.0), r);
}

__device__ __forceinline__ float rcp_estimate(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// 1/x (x normal; FP32: |x| < 2^126, FP64: |x| < 2^1021).
template <typename T> __device__ __forceinline__ T rcp(T x);
template <> __device__ __forceinline__ float rcp<float>(float x) { return rcp_estimate(x); }
template <> __device__ __forceinline__ double rcp<double>(double x) {
  const double r = rcp_estimate(x);
  return fma(r, fma(-x, r, 1.0), r);
}

// Square roots of 0 and normal numbers (FP64: from 2^-1000).  The FP32 bulk takes x rsqrt(x) (about 3 ulp):
// the correctly rounded sqrtf sequence cost 2-3 % of the FP32 step's
// instructions.  rsqrt_fast: 1/sqrt(x), of the smallest normal number if x is
// less, so that every x >= 0 has a finite root x rsqrt_fast(x).
__device__ __forceinline__ float rsqrt_fast(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(fmaxf(x, 1.17549435e-38f)));
  return r;
}
template <typename T> __device__ __forceinline__ T dsqrt(T x);
template <> __device__ __forceinline__ float dsqrt<float>(float x) { return x * rsqrt_fast(x); }
template <> __device__ __forceinline__ double dsqrt<double>(double x) {
  double h;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(h) : "d"(x));
  double s = x * h;                                                      // sqrt(x)
  h = __hiloint2double(__double2hiint(h) - (1 << 20), __double2loint(h));  // 1/(2 sqrt(x))
  const double e = fma(-s, h, 0.5);
  s = fma(s, e, s);
  h = fma(h, e, h);
  s = fma(fma(-s, s, x), h, s);
  return is_zero(x) ? x : s;
}

// x > 0 (false for NaN).
__device__ __forceinline__ bool is_pos(float x) { return x > 0.0f; }
__device__ __forceinline__ bool is_pos(double x) {
  return (unsigned long long)__double_as_longlong(x) - 1ull < 0x7ff0000000000000ull;
}
// x >= 0 (FP64: of the two zeros only +0).
__device__ __forceinline__ bool is_nonneg(float x) { return x >= 0.0f; }
__device__ __forceinline__ bool is_nonneg(double x) { return __double2hiint(x) >= 0; }
// The smaller and the larger of two numbers (neither NaN).
__device__ __forceinline__ long long order_key(double x) {
  const long long b = __double_as_longlong(x);
  return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ float min_of(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ float max_of(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ double min_of(double a, double b) { return order_key(a) < order_key(b) ? a : b; }
__device__ __forceinline__ double max_of(double a, double b) { return order_key(a) < order_key(b) ? b : a; }

// Powers (x > 0) as exp2(y log2 x): a few ulp (FP64: relative 1e-15 at the
// exponents of the exact solver), against the accurate pow/powf, whose
// extended-precision logarithm is several times longer and dominated the
// instruction stream of the exact solver.
template <typename T> __device__ __forceinline__ T dpow(T x, T y);
template <> __device__ __forceinline__ double dpow<double>(double x, double y) { return exp2(y * log2(x)); }
template <> __device__ __forceinline__ float dpow<float>(float x, float y) { return exp2f(y * log2f(x)); }

// Quotient of the state conversions, wave speeds and the exact solver
// (pressure functions, guess, Newton step, sampling).  FP32: a times the
// reciprocal above (Newton corrects its own iterates).  FP64: a normal or 0, b
// as for rcp, the quotient normal.
template <typename T> __device__ __forceinline__ T qdiv(T a, T b);
template <> __device__ __forceinline__ float qdiv<float>(float a, float b) { return a * rcp<float>(b); }
// (quotient: a/b with r = 1/b to ~2^-36 in hand)
__device__ __forceinline__ float quotient(float a, float, float r) { return a * r; }
__device__ __forceinline__ double quotient(double a, double b, double r) {
  const double q = a * r;
  return fma(fma(-b, q, a), r, q);
}
template <> __device__ __forceinline__ double qdiv<double>(double a, double b) { return quotient(a, b, rcp_estimate(b)); }

template <typename T> __device__ __forceinline__ T temp_tol();
template <> __device__ __forceinline__ double temp_tol<double>() { return 1e-13; }
template <> __device__ __forceinline__ float temp_tol<float>() { return 1e-6f; }

// A temperature and the Newton iterations it took.
template <typename T>
struct TempIts {
  T t;
  int its;
};
// GasRad::temperature from the upper bound, for a start so far below the root
// that 60 steps do not reach it: the first then lands far above (in FP32 it
// may overflow), where each further one takes off a quarter at most.  (Of its
// own: the bound tested at each step cost the radiation wedge 2-6 %, a second
// pass of the usual loop 3 %, this 0.6 %.)
template <typename T>
static __device__ __noinline__ TempIts<T> far_temperature(T c1, T c4, T y) {
  T t = qdiv(y, c1);
  if (c4 > T(0)) t = min_of(t, dsqrt(dsqrt(qdiv(y, c4))));
  int it = 0;
  for (; it < 60; ++it) {
    const T t3 = t * t * t;
    const T tn = t - qdiv(c1 * t + c4 * t3 * t - y, c1 + T(4) * c4 * t3);
    if (!(tn < t)) break;
    t = tn;
  }
  return {t, 60 + it};
}
// The solve of GasRad::temperature.  Out of line: a step has 15 sites of it,
// and inlined they overflowed the instruction cache (1.8 stalls per issue).
template <typename T>
static __device__ __noinline__ TempIts<T> newton_temperature(T c1, T c4, T y, T t0) {
  T t = qdiv(y, c1);
  if (!is_pos(y)) return {t, 0};
  if (t0 > T(0)) t = t0;
  else if (c4 > T(0)) t = min_of(t, dsqrt(dsqrt(qdiv(y, c4))));
  bool conv = false;
  int it = 0;
  for (; it < 60; ++it) {
    const T t3 = t * t * t;
    const T tn = t - qdiv(c1 * t + c4 * t3 * t - y, c1 + T(4) * c4 * t3);
    const T ch = fabs(tn - t);
    t = tn;
    if (conv) break;
    if (ch < temp_tol<T>() * tn) {
      if constexpr (sizeof(T) == 4) break;  // FP32: this step was the last
      conv = true;
    }
  }
  if (it == 60 && t0 > T(0)) return far_temperature<T>(c1, c4, y);
  return {t, it < 60 ? it + 1 : 60};
}

// Ideal gas in equilibrium with radiation, Eq. 6-7: e = rho R T/(gamma-1) +
// a T^4, P = rho R T + a T^4/3 with R = k_b/(mu m_u), and the sound speed of
// Eq. 7.  The temperature comes from a Newton iteration (Sect. 2.3).
template <typename T>
struct GasRad : Gas<T> {
  static constexpr bool RAD = true;
  T R;    // specific gas constant k_b/(mu m_u)
  T Rg;   // R/(gamma - 1)
  T a;    // radiation constant
  T a3;   // a/3
  T c_g;  // gamma/(gamma - 1), numerator constant of Eq. 7
  T c_1;  // 1/(gamma - 1), denominator constant of Eq. 7

  // The temperature where c1 t + c4 t^4 = y (c1 > 0, c4 >= 0).  The left side
  // is increasing and convex in t > 0, so Newton from the upper bound
  // min(y/c1, (y/c4)^(1/4)) descends monotonically to the root; from any
  // other positive start t0 (a nearby temperature the caller knows) the first
  // step lands above the root and the descent follows (from that bound again
  // if 60 steps do not end it: a start below a few hundredths of the root).  It stops when the
  // relative step is below temp_tol and takes one more step; in FP32 the step
  // below temp_tol (1e-6) is the last (quadratic convergence leaves that
  // iterate ~1e-12 from the root, below FP32 resolution).  y <= 0 gives
  // y/c1 <= 0, which the positivity checks reject.
  // (its, if given, accumulates the Newton iterations taken.)
  __device__ __forceinline__ T temperature(T c1, T c4, T y, T t0 = T(0), int* its = nullptr) const {
    const TempIts<T> r = newton_temperature<T>(c1, c4, y, t0);
    if (its) *its += r.its;
    return r.t;
  }
  // Eq. 7 from the gas and radiation pressures
  __device__ __forceinline__ T sound2(T rho, T pg, T pr) const {
    const T al = qdiv(pr, pg);
    return qdiv(c_g + T(20) * al + T(16) * al * al, c_1 + T(12) * al) * qdiv(pg, rho);
  }
  // P and c^2 from (rho, e)
  __device__ __forceinline__ void from_e(T rho, T e, T& p, T& c2) const {
    const T t = temperature(rho * Rg, a, e);
    const T pg = rho * R * t, pr = a3 * t * t * t * t;
    p = pg + pr;
    c2 = sound2(rho, pg, pr);
  }
  // P, c^2 and the temperature from (rho, e) (t0: a start, see temperature)
  __device__ __forceinline__ void from_e_t(T rho, T e, T& p, T& c2, T& t, T t0 = T(0), int* its = nullptr) const {
    t = temperature(rho * Rg, a, e, t0, its);
    const T pg = rho * R * t, pr = a3 * t * t * t * t;
    p = pg + pr;
    c2 = sound2(rho, pg, pr);
  }
  // the temperature of (rho, P) (t0: a start, see temperature)
  __device__ __forceinline__ T temp_p(T rho, T p, T t0 = T(0), int* its = nullptr) const {
    return temperature(rho * R, a3, p, t0, its);
  }
  // e and c^2 of a state whose temperature is known
  __device__ __forceinline__ void from_t(T rho, T t, T& e, T& c2) const {
    const T pg = rho * R * t, pr = a3 * t * t * t * t;
    e = pg * c_1 + T(3) * pr;
    c2 = sound2(rho, pg, pr);
  }
  // e and c^2 from (rho, P)
  __device__ __forceinline__ void from_p(T rho, T p, T& e, T& c2) const {
    const T t = temperature(rho * R, a3, p);
    const T pg = rho * R * t, pr = a3 * t * t * t * t;
    e = pg * c_1 + T(3) * pr;
    c2 = sound2(rho, pg, pr);
  }
};

// The larger of two non-negative numbers (FP64: by their bit patterns).
__device__ __forceinline__ float larger_speed(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ double larger_speed(double a, double b) {
  return __double_as_longlong(a) < __double_as_longlong(b) ? b : a;
}

// sum += x z for z given as the pair z.x + z.y, the sum kept as a compensated
// pair.  (The _rn intrinsics keep the compiler from fusing these operations.)
__device__ __forceinline__ void add_column_sum(float2& sum, float x, float2 z) {
  const float p = __fmul_rn(x, z.x);
  const float e = fmaf(x, z.y, fmaf(x, z.x, -p));
  const float t = __fadd_rn(sum.x, p);
  const float bb = __fsub_rn(t, sum.x);
  const float r = __fadd_rn(__fsub_rn(sum.x, __fsub_rn(t, bb)), __fsub_rn(p, bb));
  const float lo = __fadd_rn(sum.y, __fadd_rn(r, e));
  sum.x = __fadd_rn(t, lo);
  sum.y = __fsub_rn(lo, __fsub_rn(sum.x, t));
}

// (double)x of a finite x.  FP32 by integer operations and one exact product
// (which makes a subnormal normal): a conversion occupies the FP64 pipe.
__device__ __forceinline__ double widen(float x) {
  const bool less = fabsf(x) < 1.0f;
  const unsigned b = __float_as_uint(less ? x * 0x1p100f : x);
  const unsigned h = ((b & 0x7fffffffu) >> 3) + (less ? 0x38000000u - (100u << 20) : 0x38000000u);
  return __hiloint2double((int)((b & 0x80000000u) | ((b & 0x7fffffffu) ? h : 0u)), (int)(b << 29));
}
__device__ __forceinline__ double widen(double x) { return x; }

// 0 as long as `nul` is 0 and x is finite, NaN otherwise (FP64: by the bits).
__device__ __forceinline__ float finite_or(float nul, float x) { return fmaf(x, 0.0f, nul); }
__device__ __forceinline__ double finite_or(double nul, double x) {
  return (__double2hiint(x) & 0x7ff00000) == 0x7ff00000 ? __longlong_as_double(0x7ff8000000000000ll) : nul;
}
// Whether two numbers are equal (FP64: have the same bits, so 0 and -0 differ).
__device__ __forceinline__ bool equal_values(float a, float b) { return a == b; }
__device__ __forceinline__ bool equal_values(double a, double b) {
  return __double_as_longlong(a) == __double_as_longlong(b);
}
// Whether two numbers have the same bits.
__device__ __forceinline__ bool same_bits(float a, float b) { return __float_as_int(a) == __float_as_int(b); }
__device__ __forceinline__ bool same_bits(double a, double b) {
  return __double_as_longlong(a) == __double_as_longlong(b);
}
// 1/x, correctly rounded in FP32.
__device__ __forceinline__ float one_over(float x) { return 1.0f / x; }
__device__ __forceinline__ double one_over(double x) { return rcp<double>(x); }

template <typename T> __device__ __forceinline__ T dexp(T x);
template <> __device__ __forceinline__ double dexp<double>(double x) { return exp(x); }
template <> __device__ __forceinline__ float dexp<float>(float x) { return expf(x); }
template <typename T> __device__ __forceinline__ T dlog(T x);
template <> __device__ __forceinline__ double dlog<double>(double x) { return log(x); }
template <> __device__ __forceinline__ float dlog<float>(float x) { return logf(x); }

// ---------------------------------------------------------------------------
// EoS conversions (Eq. 5 with E = e + rho|u|^2/2)
// ---------------------------------------------------------------------------
template <typename T, int D, int NSX, typename G>
__device__ __forceinline__ void to_prim(const T* U, T* W, const G& gas) {
  const T rho = U[0];
  const T ir = rcp<T>(rho);
  T ke = T(0);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    W[1 + d] = U[1 + d] * ir;
    ke += U[1 + d] * W[1 + d];
  }
  W[0] = rho;
  if constexpr (G::RAD) {
    T c2;
    gas.from_e(rho, U[1 + D] - T(0.5) * ke, W[1 + D], c2);
  } else {
    W[1 + D] = gas.gm1 * (U[1 + D] - T(0.5) * ke);
  }
#pragma unroll
  for (int s = 0; s < NSX; ++s) W[2 + D + s] = U[2 + D + s] * ir;
}

// to_prim for the gas + radiation EoS that also returns c^2 (Eq. 7) and the
// temperature of the same solve (t0: a Newton start, see GasRad::temperature).
template <typename T, int D, int NSX, typename G>
__device__ __forceinline__ void to_prim_ct(const T* U, T* W, T& c2, T& t, const G& gas, T t0 = T(0),
                                           int* its = nullptr) {
  const T rho = U[0];
  const T ir = rcp<T>(rho);
  T ke = T(0);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    W[1 + d] = U[1 + d] * ir;
    ke += U[1 + d] * W[1 + d];
  }
  W[0] = rho;
  gas.from_e_t(rho, U[1 + D] - T(0.5) * ke, W[1 + D], c2, t, t0, its);
#pragma unroll
  for (int s = 0; s < NSX; ++s) W[2 + D + s] = U[2 + D + s] * ir;
}

// Internal energy per volume of the primitive state (rho, p) (Eq. 5 or 6).
template <typename T, typename G>
__device__ __forceinline__ T eint_of(const G& gas, T rho, T p) {
  if constexpr (G::RAD) {
    T e, c2;
    gas.from_p(rho, p, e, c2);
    return e;
  } else {
    return p * gas.igm1;
  }
}

template <typename T, int D, int NSX, typename G>
__device__ __forceinline__ void to_cons(const T* W, T* U, const G& gas) {
  const T rho = W[0];
  T v2 = T(0);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    U[1 + d] = rho * W[1 + d];
    v2 += W[1 + d] * W[1 + d];
  }
  U[0] = rho;
  if constexpr (G::RAD) U[1 + D] = eint_of(gas, rho, W[1 + D]) + T(0.5) * rho * v2;
  else U[1 + D] = W[1 + D] * gas.igm1 + T(0.5) * rho * v2;
#pragma unroll
  for (int s = 0; s < NSX; ++s) U[2 + D + s] = rho * W[2 + D + s];
}

// Physical flux through a face normal to axis DIR, from primitives.
template <typename T, int D, int NSX, int DIR, typename G>
__device__ __forceinline__ void phys_flux(const T* W, T* F, const G& gas) {
  const T rho = W[0], un = W[1 + DIR], p = W[1 + D];
  T v2 = T(0);
#pragma unroll
  for (int d = 0; d < D; ++d) v2 += W[1 + d] * W[1 + d];
  T E;
  if constexpr (G::RAD) E = eint_of(gas, rho, p) + T(0.5) * rho * v2;
  else E = p * gas.igm1 + T(0.5) * rho * v2;
  const T mn = rho * un;
  F[0] = mn;
#pragma unroll
  for (int d = 0; d < D; ++d) F[1 + d] = mn * W[1 + d];
  F[1 + DIR] += p;
  F[1 + D] = un * (E + p);
#pragma unroll
  for (int s = 0; s < NSX; ++s) F[2 + D + s] = mn * W[2 + D + s];
}

// ---------------------------------------------------------------------------
// Slope limiters of Eq. 17 (minmod, van Leer, van Albada; 0 = first order),
// applied to the one-sided differences dm, dp; zero when they differ in sign.
// ---------------------------------------------------------------------------
// minmod: the argument of smaller magnitude where the signs agree.  FP32:
// the hardware minimum of magnitudes that carries the product's sign,
// clamped at 0, with dm's sign put back (3 instructions).  FP64: signs and
// magnitudes compared as integers (no FP64 operation).
__device__ __forceinline__ float minmod(float dm, float dp) {
  float m;
  asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(m) : "f"(dm), "f"(dp));
  return __int_as_float(__float_as_int(fmaxf(m, 0.0f)) | (__float_as_int(dm) & 0x80000000));
}
__device__ __forceinline__ double minmod(double dm, double dp) {
  const unsigned long long bm = (unsigned long long)__double_as_longlong(dm) & 0x7fffffffffffffffull;
  const unsigned long long bp = (unsigned long long)__double_as_longlong(dp) & 0x7fffffffffffffffull;
  const double m = bm < bp ? dm : dp;
  return (__double2hiint(dm) ^ __double2hiint(dp)) < 0 ? 0.0 : m;
}
// van Leer's 2ab/(a+b) and van Albada's ab(a+b)/(a^2+b^2) where the signs
// agree.  FP32: through the ratio s of the smaller to the larger magnitude,
// so that no product of two small slopes underflows (densities of 1e-24 have
// slopes of that size); magnitudes below 2^-125 give 0.
__device__ __forceinline__ float smooth_limit(bool vanleer, float dm, float dp) {
  const float m = fmaxf(fabsf(dm), fabsf(dp)), n = fminf(fabsf(dm), fabsf(dp));
  if ((__float_as_int(dm) ^ __float_as_int(dp)) < 0 || !(m > 2.4e-38f)) return 0.0f;
  const float s = n * rcp<float>(m);
  const float r = vanleer ? (n + n) * rcp<float>(1.0f + s) : n * (1.0f + s) * rcp<float>(1.0f + s * s);
  return __int_as_float(__float_as_int(r) | (__float_as_int(dm) & 0x80000000));
}
// (FP64: the product as the sign test; the quotients need a normal divisor,
// and slopes of less than ~1e-149 do not matter.)
__device__ __forceinline__ double smooth_limit(bool vanleer, double dm, double dp) {
  const double pr = dm * dp;
  if (__double2hiint(pr) <= 0x01d00000) return 0.0;  // 2^-994
  return vanleer ? qdiv(2.0 * pr, dm + dp) : qdiv(pr * (dm + dp), dm * dm + dp * dp);
}

// Homogeneous of degree 1: limit(k, s a, s b) = s limit(k, a, b) for s > 0.
template <typename T>
__device__ __forceinline__ T limit(int kind, T dm, T dp) {
  if (kind == LIM_MINMOD) return minmod(dm, dp);
  if (kind == LIM_FIRST) return T(0);
  return smooth_limit(kind == LIM_VANLEER, dm, dp);
}

// ---------------------------------------------------------------------------
// Approximate Riemann solvers.
// ---------------------------------------------------------------------------
// Flux through a face normal to DIR and the conserved state of a primitive
// state whose internal energy per volume e is already known.
template <typename T, int D, int NSX, int DIR>
__device__ __forceinline__ void flux_cons_e(const T* W, T e, T* F, T* U) {
  const T rho = W[0], un = W[1 + DIR], p = W[1 + D];
  T v2 = T(0);
#pragma unroll
  for (int d = 0; d < D; ++d) v2 += W[1 + d] * W[1 + d];
  const T E = e + T(0.5) * rho * v2;
  const T mn = rho * un;
  F[0] = mn;
  U[0] = rho;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    F[1 + d] = mn * W[1 + d];
    U[1 + d] = rho * W[1 + d];
  }
  F[1 + DIR] += p;
  F[1 + D] = un * (E + p);
  U[1 + D] = E;
#pragma unroll
  for (int s = 0; s < NSX; ++s) {
    F[2 + D + s] = mn * W[2 + D + s];
    U[2 + D + s] = rho * W[2 + D + s];
  }
}

// FP64: the difference of the fluxes of two limited states (ideal gas) and
// their conserved states, every fused operation written out, so that all
// instantiations round alike.
template <int D, int NSX, int DIR>
__device__ __forceinline__ void flux_diff(const double* Wl, const double* Wh, double igm1, double* dF, double* Ul,
                                          double* Uh) {
  auto conserved = [&](const double* W, double* U) {
    double v2 = __dmul_rn(W[1], W[1]);
#pragma unroll
    for (int d = 1; d < D; ++d) v2 = fma(W[1 + d], W[1 + d], v2);
    U[0] = W[0];
#pragma unroll
    for (int v = 1; v < 2 + D + NSX; ++v) U[v] = __dmul_rn(W[0], W[v]);
    U[1 + D] = fma(__dmul_rn(0.5, W[0]), v2, __dmul_rn(W[1 + D], igm1));
  };
  conserved(Wl, Ul);
  conserved(Wh, Uh);
  const double ul = Wl[1 + DIR], uh = Wh[1 + DIR], pl = Wl[1 + D], ph = Wh[1 + D];
  const double ml = Ul[1 + DIR], mh = Uh[1 + DIR];
  dF[0] = __dsub_rn(ml, mh);
#pragma unroll
  for (int v = 1; v < 2 + D + NSX; ++v) dF[v] = fma(ml, Wl[v], -__dmul_rn(mh, Wh[v]));
  dF[1 + DIR] = __dsub_rn(fma(ml, ul, pl), fma(mh, uh, ph));
  dF[1 + D] = fma(ul, __dadd_rn(Ul[1 + D], pl), -__dmul_rn(uh, __dadd_rn(Uh[1 + D], ph)));
}

// HLL flux of two states with known internal energies and sound speeds,
// Davis speeds S_L, S_R.  With S_L clamped to <= 0 and S_R to >= 0 (the
// supersonic cases included), F = a F_L + b F_R + c (U_R - U_L) with a =
// S_R/(S_R - S_L), b = -S_L/(S_R - S_L), c = S_L S_R/(S_R - S_L); and since
// F = u U + P (0, n, u), each side's conserved state enters with one factor
// k_L = a u_L - c, k_R = b u_R + c: about 45 operations instead of the ~75 of
// forming both fluxes and both conserved states.  Densities (and scalars and
// energies, by the same operations) enter as a u_L rho_L + b u_R rho_R + c (rho_R
// - rho_L): the factors carry the rounding of c even where the sides are equal,
// which raised the density's error by a third on a smooth flow (FP64; 2 % in
// FP32) and that of the energy by 2 %.
template <typename T, int D, int NSX, int DIR>
__device__ __forceinline__ void hll_flux(const T* WL, const T* WR, T eL, T eR, T cL, T cR, T* F) {
  const T uL = WL[1 + DIR], uR = WR[1 + DIR], pL = WL[1 + D], pR = WR[1 + D];
  T SL = min_of(uL - cL, uR - cR), SR = max_of(uL + cL, uR + cR);
  SL = is_nonneg(SL) ? T(0) : SL;
  SR = is_nonneg(SR) ? SR : T(0);
  const T inv = rcp<T>(SR - SL);
  const T a = SR * inv, b = -SL * inv, c = (SL * SR) * inv;
  const T auL = a * uL, buR = b * uR;
  const T kL = auL - c, kR = buR + c;
  const T mL = WL[0] * kL, mR = WR[0] * kR;
  T vL = T(0), vR = T(0);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    vL += WL[1 + d] * WL[1 + d];
    vR += WR[1 + d] * WR[1 + d];
    F[1 + d] = mL * WL[1 + d] + mR * WR[1 + d];
  }
  auto carried = [&](T qL, T qR) { return fma(c, qR - qL, fma(buR, qR, auL * qL)); };
  F[0] = carried(WL[0], WR[0]);
  F[1 + DIR] += a * pL + b * pR;
  F[1 + D] = fma(auL, pL, fma(buR, pR, carried(eL + T(0.5) * WL[0] * vL, eR + T(0.5) * WR[0] * vR)));
#pragma unroll
  for (int s = 0; s < NSX; ++s) F[2 + D + s] = carried(WL[0] * WL[2 + D + s], WR[0] * WR[2 + D + s]);
}

// HLLC flux of two states with known internal energies and sound speeds: the
// contact is restored; star states keep their side's tangential velocities
// and scalars.  The flux is that of the state on the face: V (rho, rho u_t,
// rho V, E + P, rho f) + (0, n P, 0), with V, rho, P, E those of the side
// where the flow is supersonic and of its star state (V = S*, rho* = rho (S -
// u)/(S - S*), P* = P + rho (S - u)(S* - u)) otherwise: two quotients instead
// of the four of F + S (U* - U).
template <typename T, int D, int NSX, int DIR>
__device__ __forceinline__ void hllc_flux(const T* WL, const T* WR, T eL, T eR, T cL, T cR, T* F) {
  const T uL = WL[1 + DIR], uR = WR[1 + DIR], pL = WL[1 + D], pR = WR[1 + D];
  const T SL = min_of(uL - cL, uR - cR), SR = max_of(uL + cL, uR + cR);
  const T aL = WL[0] * (SL - uL), aR = WR[0] * (SR - uR);
  const T Ss = qdiv(pR - pL + uL * aL - uR * aR, aL - aR);
  const bool supL = is_nonneg(SL), supR = !is_pos(SR);
  const bool left = supL || (!supR && is_nonneg(Ss));  // the side of the contact
  T W[2 + D + NSX];
#pragma unroll
  for (int v = 0; v < 2 + D + NSX; ++v) W[v] = left ? WL[v] : WR[v];
  const T S = left ? SL : SR, a = left ? aL : aR, e = left ? eL : eR;  // a = rho (S - u)
  const T rho = W[0], un = W[1 + DIR], p = W[1 + D];
  T v2 = T(0);
#pragma unroll
  for (int d = 0; d < D; ++d) v2 += W[1 + d] * W[1 + d];
  const T E = e + T(0.5) * rho * v2;
  const T inv = rcp<T>(S - Ss);
  const bool sup = left ? supL : supR;
  const T V = sup ? un : Ss;
  const T pS = sup ? p : p + a * (Ss - un);
  const T rS = sup ? rho : a * inv;
  const T ES = sup ? E : (E * (S - un) - p * un + pS * Ss) * inv;
  const T m = rS * V;
  F[0] = m;
#pragma unroll
  for (int d = 0; d < D; ++d) F[1 + d] = m * W[1 + d];
  F[1 + DIR] = m * V + pS;
  F[1 + D] = V * (ES + pS);
#pragma unroll
  for (int s = 0; s < NSX; ++s) F[2 + D + s] = m * W[2 + D + s];
}

// Internal energy and sound speed of a face state: from its temperature t
// where the caller knows it (gas + radiation, t > 0), else from (rho, P).
template <typename T, typename G>
__device__ __forceinline__ void face_e_c(const G& gas, T rho, T p, T t, T& e, T& c) {
  T c2;
  if constexpr (G::RAD) {
    if (t > T(0)) gas.from_t(rho, t, e, c2);
    else gas.from_p(rho, p, e, c2);
  } else {
    e = p * gas.igm1;
    c2 = qdiv(gas.g * p, rho);
  }
  c = dsqrt(c2);
}

// HLL and HLLC with Davis wave-speed bounds (TL, TR: the face states'
// temperatures, gas + radiation).
template <typename T, int D, int NSX, int DIR, typename G>
__device__ __forceinline__ void riemann_hll(const T* WL, const T* WR, T* F, const G& gas, T TL = T(0), T TR = T(0)) {
  T eL, eR, cL, cR;
  face_e_c<T>(gas, WL[0], WL[1 + D], TL, eL, cL);
  face_e_c<T>(gas, WR[0], WR[1 + D], TR, eR, cR);
  hll_flux<T, D, NSX, DIR>(WL, WR, eL, eR, cL, cR, F);
}

template <typename T, int D, int NSX, int DIR, typename G>
__device__ __forceinline__ void riemann_hllc(const T* WL, const T* WR, T* F, const G& gas, T TL = T(0), T TR = T(0)) {
  T eL, eR, cL, cR;
  face_e_c<T>(gas, WL[0], WL[1 + D], TL, eL, cL);
  face_e_c<T>(gas, WR[0], WR[1 + D], TR, eR, cR);
  hllc_flux<T, D, NSX, DIR>(WL, WR, eL, eR, cL, cR, F);
}

// ---------------------------------------------------------------------------
// Exact Riemann solver (Toro 2009 ch. 4).
// ---------------------------------------------------------------------------
// y^n, n in 4 .. 8 (the same n in all threads).
template <typename T>
__device__ __forceinline__ T power_n(T y, int n) {
  const T y2 = y * y, y4 = y2 * y2;
  if (n == 8) return y4 * y4;
  T w = y4;
  if (n & 2) w *= y2;
  if (n & 1) w *= y;
  return w;
}
// One third-order (Halley) step for y^n = x from y with relative error e:
// y + 2 y (x - y^n)/((n + 1) y^n + (n - 1) x), error ~ n^2/12 e^3.  The
// quotient is a correction of relative size e, so it needs only its leading
// digits: its divisor's reciprocal is refined once (FP64).
__device__ __forceinline__ float root_step(float y, float x, int n) {
  const float w = power_n(y, n);
  return fmaf(y * (x - w), rcp<float>(0.5f * (n + 1) * w + 0.5f * (n - 1) * x), y);
}
// FP64: the rounding of the powers is carried along (each product's exact
// remainder by a fused operation), so that the root is hi + lo, hi its nearest
// number.  With the plain residual x - y^n the last bit was wrong at times;
// that and the quotients taken as products with rounded reciprocals (here, in
// press_fn and in behind_fan) cost the exact solver 2-4 % in accuracy.  512
// FP64 tubes take 2.01 ms with all of it, 1.83 without.
struct Root {
  double hi, lo;
};
__device__ __forceinline__ Root root_step(double y, double x, int n) {
  const double y2 = y * y, e2 = fma(y, y, -y2);
  const double y4 = y2 * y2, e4 = fma(y2 + y2, e2, fma(y2, y2, -y4));
  double w = y4, e = e4;
  if (n == 8) {
    w = y4 * y4;
    e = fma(y4 + y4, e4, fma(y4, y4, -w));
  } else {
    if (n & 2) {
      w = y4 * y2;
      e = fma(y4, e2, fma(e4, y2, fma(y4, y2, -w)));
    }
    if (n & 1) {
      const double v = w * y;
      e = fma(e, y, fma(w, y, -v));
      w = v;
    }
  }
  const double d = y * ((x - w) - e) * rcp_estimate(fma(0.5 * (n + 1), w, 0.5 * (n - 1) * x));
  const double hi = y + d;
  return {hi, (y - hi) + d};
}
// x^z, z = (gamma - 1)/(2 gamma), x > 0 a ratio of pressures.  For the usual
// gammas 1/z is a small integer and x^z a root: a hardware estimate (relative
// error ~1e-6) and one root_step, correct to about 1 ulp (FP64 half of one) --
// 17 FP64 operations, against the ~43 of exp2(z log2 x), whose FP32 form is
// also twice as long and less exact.
__device__ __forceinline__ float pow_z(float x, const Gas<float>& gas) {
  if (gas.root == 0) return dpow<float>(x, gas.z);
  float t;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(t) : "f"(__log2f(x) * gas.z));
  return root_step(t, x, gas.root);
}
__device__ __forceinline__ Root root_z(double x, const Gas<double>& gas) {
  // log2 x from its exponent and leading 23 bits; 2^t scaled back by the exponent
  const int hx = __double2hiint(x), lx = __double2loint(x);
  const float m = __int_as_float(0x3f800000 | ((hx & 0xfffff) << 3) | (int)((unsigned)lx >> 29));
  const float t = ((float)((hx >> 20) - 1023) + __log2f(m)) * (float)gas.z, ti = rintf(t);
  float f;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"(t - ti));
  double y = (double)f;
  y = __hiloint2double(__double2hiint(y) + ((int)ti << 20), __double2loint(y));
  return root_step(y, x, gas.root);
}
__device__ __forceinline__ double pow_z(double x, const Gas<double>& gas) {
  return gas.root ? root_z(x, gas).hi : dpow<double>(x, gas.z);
}
// Behind a rarefaction of pressure ratio q: t = q^z, the ratio of sound
// speeds, and rho = rK q^(1/g) = rK q^(1 - 2z) (FP64: of a root, the quotient
// of the exact products, to about half an ulp).
__device__ __forceinline__ float behind_fan(float rK, float q, const Gas<float>& gas, float& t) {
  t = pow_z(q, gas);
  return qdiv(rK * q, t * t);
}
__device__ __forceinline__ double behind_fan(double rK, double q, const Gas<double>& gas, double& t) {
  if (gas.root == 0) {
    t = dpow<double>(q, gas.z);
    return rK * dpow<double>(q, gas.ig);
  }
  const Root y = root_z(q, gas);
  t = y.hi;
  const double b = t * t, eb = fma(t + t, y.lo, fma(t, t, -b));
  const double a = rK * q, ea = fma(rK, q, -a);
  const double r = rcp_estimate(b), rho = a * r;
  return fma(fma(-rho, eb, fma(-rho, b, a) + ea), r, rho);
}
// x^(1/z)
template <typename T>
__device__ __forceinline__ T pow_iz(T x, const Gas<T>& gas) {
  return gas.root ? power_n(x, gas.root) : dpow<T>(x, gas.iz);
}

// What the pressure function of one side needs at every iterate.
template <typename T>
struct PressSide {
  T p, ip;   // p_K and its reciprocal
  T A, B;    // 2/((g+1) rho_K), (g-1)/(g+1) p_K
  T f0, irc;  // 2 c_K/(g-1), 1/(rho_K c_K) = c_K/(g p_K)
  __device__ __forceinline__ PressSide(T rK, T pK, T cK, const Gas<T>& gas)
      : p(pK), ip(rcp<T>(pK)), A(qdiv(gas.A2, rK)), B(gas.Bq * pK), f0(gas.two_gm1 * cK) {
    irc = cK * ip * gas.ig;
  }
};

// One side's pressure function f_K(p) and its derivative: shock branch
// (p > p_K) with A and B; rarefaction branch (p <= p_K) from the isentrope.
// (rp = 1/p)
template <typename T>
__device__ __forceinline__ void press_fn(T p, T rp, const PressSide<T>& k, const Gas<T>& gas, T& f, T& df) {
  if (p > k.p) {
    const T d = p - k.p, s = p + k.B, r = rcp_estimate(s);
    const T q = dsqrt(quotient(k.A, s, r));
    f = d * q;
    df = q * (T(1) - T(0.5) * (d * r));
  } else {
    const T pz = pow_z(quotient(p, k.p, k.ip), gas);  // (p/pK)^((g-1)/(2g))
    f = k.f0 * (pz - T(1));
    // (p/pK)^(-(g+1)/(2g)) = (p/pK)^z / (p/pK)
    df = pz * (k.p * rp) * k.irc;
  }
}

// Toro's adaptive guess (Sect. 9.5.1 of Toro 2009): PVRS when the data are
// close (pmax/pmin <= 2 and PVRS within [pmin,pmax]); TRRS below pmin; TSRS
// otherwise.  kind: 0 PVRS, 1 TRRS, 2 TSRS.
template <typename T>
__device__ __forceinline__ T toro_guess(T rL, T uL, T pL, T cL, T rR, T uR, T pR, T cR,
                                        const Gas<T>& gas, int& kind) {
  T ppv = T(0.5) * (pL + pR) - T(0.125) * (uR - uL) * (rL + rR) * (cL + cR);
  ppv = is_pos(ppv) ? ppv : T(0);
  const T pmin = min_of(pL, pR), pmax = max_of(pL, pR);
  if (pmax <= T(2) * pmin && ppv >= pmin && ppv <= pmax) {
    kind = 0;
    return ppv;
  }
  if (ppv < pmin) {
    kind = 1;
    // p_L (num/(c_L + c_R (p_L/p_R)^z))^(1/z)
    const T num = cL + cR - T(0.5) * gas.gm1 * (uR - uL);
    const T den = cL + cR * pow_z(qdiv(pL, pR), gas);
    return pL * pow_iz(qdiv(num, den), gas);
  }
  kind = 2;
  const T gL = dsqrt(qdiv(qdiv(gas.A2, rL), ppv + gas.Bq * pL));
  const T gR = dsqrt(qdiv(qdiv(gas.A2, rR), ppv + gas.Bq * pR));
  return qdiv(gL * pL + gR * pR - (uR - uL), gL + gR);
}

// Newton on f_L(p) + f_R(p) + (u_R - u_L) = 0 from p0: stop when the
// relative change 2|dp|/(p_k + p_{k-1}) < tol, then take one more step.
// Negative iterates are clamped to 1e-14 of the mean pressure.  In FP32 the
// step whose change is below tol (1e-6) is the last: Newton converges
// quadratically, so the iterate it gives is ~1e-12 from the root, far below
// FP32 resolution, and a further step would only move it within its own
// rounding.  The FP32 iteration also stops when the residual is within 8 ulp
// of the sum of the magnitudes of its terms (then with one more step): the
// rounding of f_L + f_R + du then decides the step, and no later iterate is
// better determined (near vacuum, where the two rarefaction terms nearly
// cancel du, the 1e-6 change is never reached).
// The last step's change dp is below that tolerance (or within the residual's
// rounding), so f at its iterate is f + f' dp to O(dp^2), below the rounding of
// f: the star velocity takes that instead of a further evaluation.
template <typename T>
__device__ __forceinline__ int newton_star(T p, T rL, T uL, T pL, T cL, T rR, T uR, T pR, T cR,
                                           const Gas<T>& gas, T tol, T& ps, T& us, int& iters) {
  const T du = uR - uL;
  const T pfloor = T(1e-14) * T(0.5) * (pL + pR);
  if (!(p > pfloor)) p = pfloor;
  const PressSide<T> L(rL, pL, cL, gas), R(rR, pR, cR, gas);
  bool conv = false;
  for (int it = 1; it <= 100; ++it) {
    T fL, dfL, fR, dfR;
    const T rp = rcp_estimate(p);  // (for the derivatives)
    press_fn(p, rp, L, gas, fL, dfL);
    press_fn(p, rp, R, gas, fR, dfR);
    const T res = fL + fR + du;
    T pn = p - res * rcp_estimate(dfL + dfR);  // (a correction: its leading digits do)
    if (pn < T(0)) pn = pfloor;
    const T dp = pn - p;
    const bool small = T(2) * fabs(dp) < tol * (pn + p);
    p = pn;
    // FP64 takes one more step after convergence, FP32 after the residual's rule only
    if (conv || (sizeof(T) == 4 && small)) {
      iters = it;
      ps = p;
      us = T(0.5) * (uL + uR) + T(0.5) * ((fR + dfR * dp) - (fL + dfL * dp));
      return ST_OK;
    }
    conv = small;
    if constexpr (sizeof(T) == 4) conv = fabs(res) <= T(8 * 1.1920929e-7) * (fabs(fL) + fabs(fR) + fabs(du));
  }
  iters = 100;
  return ST_NEWTON;
}

// A primitive 1D state returned by value (a local whose address an
// out-of-line function takes lives in local memory).
template <typename T>
struct Prim3 {
  T rho, u, p;
};

// The state inside a left rarefaction fan at x/t = S (Toro ch. 4.5): c =
// 2/(g+1) (cK + (g-1)/2 (uK - S)), u = S + c; rho and P from the isentrope
// through (rK, pK).  Out of line: x/t = S lies inside a fan only near sonic
// points, and the hot solver code stays shorter.
template <typename T>
static __device__ __noinline__ Prim3<T> fan_state(T S, T rK, T uK, T pK, T cK, Gas<T> gas) {
  const T c = gas.A2 * (cK + T(0.5) * gas.gm1 * (uK - S));
  const T x = qdiv(c, cK), t = dpow(x, gas.two_gm1);
  Prim3<T> w;
  w.u = S + c;
  w.rho = rK * t;
  w.p = pK * (t * x * x);  // 2g/(g-1) = 2/(g-1) + 2
  return w;
}

// Sample the exact solution at x/t = S given the star state (Toro ch. 4.5);
// returns the (rho, u, P) there and whether it lies left of the contact
// (ties left).  A point right of the contact is sampled as the mirror image,
// so that both sides run the same code.
template <typename T>
__device__ __forceinline__ bool sample_xi(T S, T rL, T uL, T pL, T cL, T rR, T uR, T pR, T cR, T ps,
                                          T us, const Gas<T>& gas, T& rho, T& u, T& p) {
  const bool left = S <= us;
  const T rK = left ? rL : rR, uK = left ? uL : -uR, pK = left ? pL : pR, cK = left ? cL : cR;
  const T x = left ? S : -S, um = left ? us : -us;
  const T q = qdiv(ps, pK);
  rho = rK;
  u = uK;
  p = pK;
  if (ps > pK) {
    const T SK = uK - cK * dsqrt(gas.zp * q + gas.z);
    if (x > SK) {
      rho = qdiv(rK * (q + gas.Bq), gas.Bq * q + T(1));
      u = um;
      p = ps;
    }
  } else if (x > uK - cK) {
    T t;  // c*/c_K
    const T rs = behind_fan(rK, q, gas, t);
    if (x >= um - cK * t) {
      rho = rs;
      u = um;
      p = ps;
    } else {
      const Prim3<T> f = fan_state<T>(x, rK, uK, pK, cK, gas);
      rho = f.rho;
      u = f.u;
      p = f.p;
    }
  }
  if (!left) u = -u;
  return left;
}

// The same at x/t = 0, the value the Godunov flux needs.
template <typename T>
__device__ __forceinline__ bool sample0(T rL, T uL, T pL, T cL, T rR, T uR, T pR, T cR, T ps, T us,
                                        const Gas<T>& gas, T& rho, T& u, T& p) {
  return sample_xi<T>(T(0), rL, uL, pL, cL, rR, uR, pR, cR, ps, us, gas, rho, u, p);
}

// Newton tolerance per precision: 1e-10 in FP64; in FP32 the relative
// change cannot go below a few ulp, so 1e-6 is used there.
template <typename T> __device__ __forceinline__ T newton_tol();
template <> __device__ __forceinline__ double newton_tol<double>() { return 1e-10; }
template <> __device__ __forceinline__ float newton_tol<float>() { return 1e-6f; }

// Gas<double> from Gas<float> for the FP64 hard-face fallback.
__device__ __forceinline__ Gas<double> gas_double(const Gas<float>& g) {
  Gas<double> d;
  const double gg = (double)g.g;
  d.g = gg; d.gm1 = gg - 1.0; d.igm1 = 1.0 / (gg - 1.0); d.z = (gg - 1.0) / (2.0 * gg);
  d.iz = 1.0 / d.z; d.zp = (gg + 1.0) / (2.0 * gg); d.A2 = 2.0 / (gg + 1.0);
  d.Bq = (gg - 1.0) / (gg + 1.0); d.two_gm1 = 2.0 / (gg - 1.0); d.ig = 1.0 / gg;
  d.root = 0;  // (of the FP32 gamma, 1/z is no integer)
  return d;
}

// Star state of one face.  guess_in > 0 replaces Toro's guess (MLP).  In FP32
// a face near vacuum (margin below 20 %) or with a pressure ratio above 1e6
// is solved in FP64, where the FP32 pressure function loses digits.
// The FP64 Newton solve of an FP32 face near vacuum or with a pressure ratio
// above 1e6 (reading R12).  Kept out of line: it is rare, and its FP64 code
// would crowd the instruction cache of the FP32 kernels.
struct Star32 {
  float ps, us;
  int iters, st;
};
static __device__ __noinline__ Star32 newton_star_fp64(float p0, float rL, float uL, float pL, float rR, float uR,
                                                float pR, Gas<float> gas) {
  const Gas<double> g2 = gas_double(gas);
  double ps2 = 0.0, us2 = 0.0;
  const double cL2 = sqrt(g2.g * (double)pL / (double)rL), cR2 = sqrt(g2.g * (double)pR / (double)rR);
  Star32 r;
  r.iters = 0;
  r.st = newton_star<double>((double)p0, rL, uL, pL, cL2, rR, uR, pR, cR2, g2, 1e-10, ps2, us2, r.iters);
  r.ps = (float)ps2;
  r.us = (float)us2;
  return r;
}

// An FP32 face that is solved in FP64 (reading R12): pressure ratio above
// 1e6, or a velocity jump within 20 % of the vacuum limit vac =
// 2(cL+cR)/(g-1), where the FP32 residual loses more than ~5 of its bits to
// the cancellation of the two rarefaction terms against du.
template <typename T>
__device__ __forceinline__ bool hard_face(T pL, T pR, T du, T vac) {
  return max_of(pL, pR) > T(1e6) * min_of(pL, pR) || vac - du < T(0.2) * vac;
}

// Star state from a given initial guess p0 and the sound speeds cL, cR of
// the two states (vacuum check, FP32 hard-face fallback, Newton).
template <typename T>
__device__ __forceinline__ int exact_star_from(T rL, T uL, T pL, T cL, T rR, T uR, T pR, T cR,
                                               const Gas<T>& gas, T p0, T& ps, T& us, int& iters) {
  const T vac = gas.two_gm1 * (cL + cR);
  if (vac <= uR - uL) return ST_VACUUM;
  if constexpr (sizeof(T) == 4) {
    if (hard_face<T>(pL, pR, uR - uL, vac)) {
      const Star32 r = newton_star_fp64(p0, rL, uL, pL, rR, uR, pR, gas);
      ps = r.ps;
      us = r.us;
      iters = r.iters;
      return r.st;
    }
  }
  return newton_star<T>(p0, rL, uL, pL, cL, rR, uR, pR, cR, gas, newton_tol<T>(), ps, us, iters);
}

template <typename T>
__device__ __forceinline__ int exact_star(T rL, T uL, T pL, T rR, T uR, T pR, const Gas<T>& gas,
                                          T guess_in, T& ps, T& us, int& iters, int& kind) {
  const T cL = dsqrt(qdiv(gas.g * pL, rL)), cR = dsqrt(qdiv(gas.g * pR, rR));
  if (gas.two_gm1 * (cL + cR) <= uR - uL) return ST_VACUUM;
  T p0 = toro_guess(rL, uL, pL, cL, rR, uR, pR, cR, gas, kind);
  if (guess_in > T(0)) p0 = guess_in;
  return exact_star_from<T>(rL, uL, pL, cL, rR, uR, pR, cR, gas, p0, ps, us, iters);
}

// Godunov flux from the exact solution at x/t = 0; tangential velocities and
// scalars come from the side of the contact.
template <typename T, int D, int NSX, int DIR>
__device__ __forceinline__ int riemann_exact(const T* WL, const T* WR, T* F, const Gas<T>& gas,
                                             T guess_in, int& iters, int& kind) {
  constexpr int NV = 2 + D + NSX;
  // Identical states: the solution is that state (no wave), and the general
  // path returns exactly its flux (PVRS gives p = P, Newton stops at once,
  // the sample is the state) -- take it directly.
  bool same = true;
#pragma unroll
  for (int v = 0; v < NV; ++v) same = same && equal_values(WL[v], WR[v]);
  if (same) {
    iters = 0;
    kind = 0;
    phys_flux<T, D, NSX, DIR>(WL, F, gas);
    return ST_OK;
  }
  T ps, us;
  const T rL = WL[0], uL = WL[1 + DIR], pL = WL[1 + D];
  const T rR = WR[0], uR = WR[1 + DIR], pR = WR[1 + D];
  const int st = exact_star<T>(rL, uL, pL, rR, uR, pR, gas, guess_in, ps, us, iters, kind);
  if (st != ST_OK) {
#pragma unroll
    for (int v = 0; v < NV; ++v) F[v] = T(0);
    return st;
  }
  const T cL = dsqrt(qdiv(gas.g * pL, rL)), cR = dsqrt(qdiv(gas.g * pR, rR));
  T rho, u, p;
  const bool left = sample0<T>(rL, uL, pL, cL, rR, uR, pR, cR, ps, us, gas, rho, u, p);
  T W[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) W[v] = left ? WL[v] : WR[v];
  W[0] = rho;
  W[1 + DIR] = u;
  W[1 + D] = p;
  phys_flux<T, D, NSX, DIR>(W, F, gas);
  return ST_OK;
}

// The Godunov flux of two different states (1D, no scalars) from a given
// initial guess p0 and their sound speeds: the batched path has both in
// hand from choosing the guess, so neither is computed twice.
template <typename T>
__device__ __forceinline__ int riemann_exact_from(const T* WL, const T* WR, T cL, T cR, T p0, T* F,
                                                  const Gas<T>& gas, int& iters) {
  T ps, us;
  const int st = exact_star_from<T>(WL[0], WL[1], WL[2], cL, WR[0], WR[1], WR[2], cR, gas, p0, ps, us, iters);
  if (st != ST_OK) {
#pragma unroll
    for (int v = 0; v < 3; ++v) F[v] = T(0);
    return st;
  }
  T W[3];
  const bool left = sample0<T>(WL[0], WL[1], WL[2], cL, WR[0], WR[1], WR[2], cR, ps, us, gas, W[0], W[1], W[2]);
  (void)left;
  phys_flux<T, 1, 0, 0>(W, F, gas);
  return ST_OK;
}

// ---------------------------------------------------------------------------
// MLP guess network: 6 -> 64 -> 64 -> 1 with SiLU, FP32 weights.
// ---------------------------------------------------------------------------
// Faces where the network replaces Toro's guess: his rule picks the two-shock
// estimate (kind 2) and the pressure jump exceeds a factor 4 -- where that
// estimate is poor; the two-rarefaction estimate is exact for two
// rarefactions and PVRS serves nearby states.
constexpr double MLP_GATE_RATIO = 4.0;
template <typename T>
__device__ __forceinline__ bool mlp_gate(int kind, T pL, T pR) {
  return kind == 2 && max_of(pL, pR) > T(MLP_GATE_RATIO) * min_of(pL, pR);
}

constexpr int MLP_IN = 6, MLP_H = 64;
constexpr int MLP_NPARAM = MLP_H * MLP_IN + MLP_H + MLP_H * MLP_H + MLP_H + MLP_H + 1;
constexpr int MW1 = 0, MB1 = MW1 + MLP_H * MLP_IN, MW2 = MB1 + MLP_H, MB2 = MW2 + MLP_H * MLP_H,
              MW3 = MB2 + MLP_H, MB3 = MW3 + MLP_H;

__device__ __forceinline__ float silu_f(float z) { return z / (1.0f + expf(-z)); }

// Features of a face: log densities and pressures normalised by their
// geometric means, velocities by the reference sound speed; p_ref returned.
__device__ __forceinline__ void mlp_features(float g, float rL, float uL, float pL, float rR,
                                             float uR, float pR, float* x, float& pref) {
  const float rref = sqrtf(rL * rR);
  pref = sqrtf(pL * pR);
  const float icref = rsqrtf(g * pref / rref);
  x[0] = logf(rL / rref);
  x[1] = logf(rR / rref);
  x[2] = logf(pL / pref);
  x[3] = logf(pR / pref);
  x[4] = uL * icref;
  x[5] = uR * icref;
}

// Forward pass with the weights in shared (or global) memory; all lanes of a
// warp read the same weight at the same time (broadcast).
__device__ __forceinline__ float mlp_forward(const float* __restrict__ w, const float* x) {
  float h1[MLP_H];
#pragma unroll
  for (int o = 0; o < MLP_H; ++o) {
    float a = w[MB1 + o];
#pragma unroll
    for (int i = 0; i < MLP_IN; ++i) a = fmaf(w[MW1 + o * MLP_IN + i], x[i], a);
    h1[o] = silu_f(a);
  }
  float y = w[MB3];
#pragma unroll 4
  for (int o = 0; o < MLP_H; ++o) {
    float a = w[MB2 + o];
#pragma unroll
    for (int i = 0; i < MLP_H; ++i) a = fmaf(w[MW2 + o * MLP_H + i], h1[i], a);
    y = fmaf(w[MW3 + o], silu_f(a), y);
  }
  return y;
}

}  // namespace hydro
