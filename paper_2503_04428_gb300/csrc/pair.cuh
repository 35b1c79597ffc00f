// pair.cuh -- the FP32 step's arithmetic on pairs of cells.
//
// sm_100 and later execute an addition, product or fused multiply-add of two
// FP32 pairs as one instruction (PTX add/sub/mul/fma .f32x2).  The FP32 grid
// step is bound by instruction issue, so its marching kernels carry two
// independent cells per thread, one in each half of every pair: the halves
// never mix, and each half's arithmetic is that of physics.cuh.  Minima,
// comparisons and the special functions run per half.
#pragma once
#include "physics.cuh"

namespace hydro {

struct f2 {
  unsigned long long v;
};
__device__ __forceinline__ f2 make_f2(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ f2 both(float a) { return make_f2(a, a); }
__device__ __forceinline__ float lo(f2 a) { return __uint_as_float((unsigned)a.v); }
__device__ __forceinline__ float hi(f2 a) { return __uint_as_float((unsigned)(a.v >> 32)); }
__device__ __forceinline__ f2 operator+(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 operator-(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 operator*(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
// Reciprocal and reciprocal square root by the hardware approximations (1-2 ulp).
__device__ __forceinline__ f2 rcp2(f2 a) { return make_f2(rcp<float>(lo(a)), rcp<float>(hi(a))); }
__device__ __forceinline__ f2 rsqrt2(f2 a) { return make_f2(rsqrt_fast(lo(a)), rsqrt_fast(hi(a))); }
__device__ __forceinline__ f2 minmod2(f2 a, f2 b) { return make_f2(minmod(lo(a), lo(b)), minmod(hi(a), hi(b))); }
__device__ __forceinline__ f2 limit2(int kind, f2 a, f2 b) {
  return make_f2(limit<float>(kind, lo(a), lo(b)), limit<float>(kind, hi(a), hi(b)));
}
// Per half: a where the half's condition holds, else b.
__device__ __forceinline__ f2 pick(bool c0, bool c1, f2 a, f2 b) {
  return make_f2(c0 ? lo(a) : lo(b), c1 ? hi(a) : hi(b));
}
// max(a, b, 0)
__device__ __forceinline__ f2 max2_0(f2 a, f2 b) {
  return make_f2(fmaxf(fmaxf(lo(a), lo(b)), 0.f), fmaxf(fmaxf(hi(a), hi(b)), 0.f));
}

// Minima that are NaN if an argument is.
__device__ __forceinline__ float min_or_nan(float a, float b) {
  float r;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float min_or_nan(float a, float b, float c) {
  float r;
  asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// The gas constants as pairs.
struct Gas2 {
  f2 g, gm1, igm1, half, mhalf;
  __device__ __forceinline__ explicit Gas2(const Gas<float>& s)
      : g(both(s.g)), gm1(both(s.gm1)), igm1(both(s.igm1)), half(both(0.5f)), mhalf(both(-0.5f)) {}
};

// (rho, m, E, rho f) -> (rho, u, P, f), D axes.
template <int D, int NSX>
__device__ __forceinline__ void to_prim2(const f2* U, f2* W, const Gas2& gas) {
  const f2 ir = rcp2(U[0]);
  W[0] = U[0];
#pragma unroll
  for (int d = 0; d < D; ++d) W[1 + d] = U[1 + d] * ir;
  f2 ke = U[1] * W[1];
#pragma unroll
  for (int d = 1; d < D; ++d) ke = fma2(U[1 + d], W[1 + d], ke);
  W[1 + D] = fma2(gas.mhalf, ke, U[1 + D]) * gas.gm1;
#pragma unroll
  for (int s = 0; s < NSX; ++s) W[2 + D + s] = U[2 + D + s] * ir;
}

template <int D>
__device__ __forceinline__ f2 speed_sq(const f2* W) {
  f2 v = W[1] * W[1];
#pragma unroll
  for (int d = 1; d < D; ++d) v = fma2(W[1 + d], W[1 + d], v);
  return v;
}

// dU += (F(l) - F(h)) ih along DIR (FIRST: dU = ...).  (Products and
// difference rounded separately: equal states give exactly 0.)
template <int D, int NSX, int DIR, bool FIRST>
__device__ __forceinline__ void half_step2(const f2* l, const f2* h, f2 ih, f2* dU, const Gas2& gas) {
  const f2 ml = l[0] * l[1 + DIR], mh = h[0] * h[1 + DIR];
  const f2 el = fma2(l[0] * gas.half, speed_sq<D>(l), l[1 + D] * gas.igm1);
  const f2 eh = fma2(h[0] * gas.half, speed_sq<D>(h), h[1 + D] * gas.igm1);
  auto add = [&](int v, f2 t) { dU[v] = FIRST ? t * ih : fma2(t, ih, dU[v]); };
  add(0, ml - mh);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    f2 t = ml * l[1 + d] - mh * h[1 + d];
    if (d == DIR) t = t + (l[1 + D] - h[1 + D]);
    add(1 + d, t);
  }
  add(1 + D, l[1 + DIR] * (el + l[1 + D]) - h[1 + DIR] * (eh + h[1 + D]));
#pragma unroll
  for (int s = 0; s < NSX; ++s) add(2 + D + s, ml * l[2 + D + s] - mh * h[2 + D + s]);
}

// The predicted state of the limited state l with the increment dU.  A half
// that is not physical falls back to Wc and is counted by count(bad0, bad1);
// the test is one vote, so every lane of the warp has to take part.
template <int D, int NSX, typename Count>
__device__ __forceinline__ void face_state2(const f2* l, const f2* dU, const f2* Wc, f2* w, const Gas2& gas,
                                            Count count) {
  constexpr int NV = 2 + D + NSX;
  f2 u[NV];
  u[0] = l[0] + dU[0];
#pragma unroll
  for (int d = 0; d < D; ++d) u[1 + d] = fma2(l[0], l[1 + d], dU[1 + d]);
  u[1 + D] = fma2(l[0] * gas.half, speed_sq<D>(l), fma2(l[1 + D], gas.igm1, dU[1 + D]));
#pragma unroll
  for (int s = 0; s < NSX; ++s) u[2 + D + s] = fma2(l[0], l[2 + D + s], dU[2 + D + s]);
  to_prim2<D, NSX>(u, w, gas);
  // (the usual outcome costs two minima and one comparison)
  if (__any_sync(0xffffffffu, !(min_or_nan(min_or_nan(lo(w[0]), lo(w[1 + D]), hi(w[0])), hi(w[1 + D])) > 0.f))) {
    const bool bad0 = !(min_or_nan(lo(w[0]), lo(w[1 + D])) > 0.f), bad1 = !(min_or_nan(hi(w[0]), hi(w[1 + D])) > 0.f);
#pragma unroll
    for (int v = 0; v < NV; ++v) w[v] = pick(bad0, bad1, Wc[v], w[v]);
    count(bad0, bad1);
  }
}

__device__ __forceinline__ f2 sound2(f2 rho, f2 p, const Gas2& gas) {
  const f2 c2 = (gas.g * p) * rcp2(rho);
  return c2 * rsqrt2(c2);
}

// hll_flux of physics.cuh on pairs (l = -S_L >= 0).
template <int D, int NSX, int DIR>
__device__ __forceinline__ void hll2(const f2* WL, const f2* WR, f2* F, const Gas2& gas) {
  const f2 uL = WL[1 + DIR], uR = WR[1 + DIR], pL = WL[1 + D], pR = WR[1 + D];
  const f2 cL = sound2(WL[0], pL, gas), cR = sound2(WR[0], pR, gas);
  const f2 l = max2_0(cL - uL, cR - uR), r = max2_0(uL + cL, uR + cR);
  const f2 inv = rcp2(r + l);
  const f2 a = r * inv, b = l * inv, c = (l * r) * inv;
  const f2 auL = a * uL, buR = b * uR;
  const f2 kL = auL + c, kR = buR - c;
  const f2 mL = WL[0] * kL, mR = WR[0] * kR;
  auto carried = [&](f2 qL, f2 qR) { return fma2(c, qL - qR, fma2(buR, qR, auL * qL)); };
  F[0] = carried(WL[0], WR[0]);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    F[1 + d] = fma2(mR, WR[1 + d], mL * WL[1 + d]);
    if (d == DIR) F[1 + d] = F[1 + d] + fma2(b, pR, a * pL);
  }
  const f2 q = fma2(mR, speed_sq<D>(WR), mL * speed_sq<D>(WL));
  F[1 + D] = fma2(gas.half, q, fma2(fma2(kR, gas.igm1, buR), pR, fma2(kL, gas.igm1, auL) * pL));
#pragma unroll
  for (int s = 0; s < NSX; ++s) F[2 + D + s] = carried(WL[0] * WL[2 + D + s], WR[0] * WR[2 + D + s]);
}

// hllc_flux of physics.cuh on pairs.
template <int D, int NSX, int DIR>
__device__ __forceinline__ void hllc2(const f2* WL, const f2* WR, f2* F, const Gas2& gas) {
  const f2 uL = WL[1 + DIR], uR = WR[1 + DIR], pL = WL[1 + D], pR = WR[1 + D];
  const f2 cL = sound2(WL[0], pL, gas), cR = sound2(WR[0], pR, gas);
  const f2 l0 = uL - cL, l1 = uR - cR, r0 = uL + cL, r1 = uR + cR;
  const f2 SL = make_f2(fminf(lo(l0), lo(l1)), fminf(hi(l0), hi(l1)));
  const f2 SR = make_f2(fmaxf(lo(r0), lo(r1)), fmaxf(hi(r0), hi(r1)));
  const f2 aL = WL[0] * (SL - uL), aR = WR[0] * (SR - uR);
  const f2 Ss = (fma2(uL, aL, pR) - fma2(uR, aR, pL)) * rcp2(aL - aR);
  const bool sl0 = lo(SL) >= 0.f, sl1 = hi(SL) >= 0.f, sr0 = !(lo(SR) > 0.f), sr1 = !(hi(SR) > 0.f);
  const bool left0 = sl0 || (!sr0 && lo(Ss) >= 0.f), left1 = sl1 || (!sr1 && hi(Ss) >= 0.f);
  const bool sup0 = sl0 || sr0, sup1 = sl1 || sr1;  // (the side's own: left if sl, right otherwise)
  const f2 rho = pick(left0, left1, WL[0], WR[0]), un = pick(left0, left1, uL, uR), p = pick(left0, left1, pL, pR);
  const f2 S = pick(left0, left1, SL, SR), a = pick(left0, left1, aL, aR);
  f2 W[D];
#pragma unroll
  for (int d = 0; d < D; ++d) W[d] = d == DIR ? un : pick(left0, left1, WL[1 + d], WR[1 + d]);
  f2 v2 = W[0] * W[0];
#pragma unroll
  for (int d = 1; d < D; ++d) v2 = fma2(W[d], W[d], v2);
  const f2 E = fma2(rho * gas.half, v2, p * gas.igm1);
  const f2 inv = rcp2(S - Ss);
  const f2 ps = fma2(a, Ss - un, p);
  const f2 V = pick(sup0, sup1, un, Ss), pS = pick(sup0, sup1, p, ps), rS = pick(sup0, sup1, rho, a * inv);
  const f2 ES = pick(sup0, sup1, E, fma2(E, S - un, ps * Ss - p * un) * inv);
  const f2 m = rS * V;
  F[0] = m;
#pragma unroll
  for (int d = 0; d < D; ++d) F[1 + d] = d == DIR ? fma2(m, V, pS) : m * W[d];
  F[1 + D] = V * (ES + pS);
#pragma unroll
  for (int s = 0; s < NSX; ++s) F[2 + D + s] = m * pick(left0, left1, WL[2 + D + s], WR[2 + D + s]);
}

}  // namespace hydro
