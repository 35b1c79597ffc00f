// march.cuh -- what the marching FP32 steps (march2.cuh, march3.cuh) share:
// asynchronous staging copies and the update of a pair of cells.
#pragma once
#include <type_traits>

#include "pair.cuh"
#include "sweep.cuh"

namespace hydro {

__device__ __forceinline__ unsigned shared_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned smem_addr(const f2* p) { return shared_addr(p); }
// Asynchronous 4-byte copies to shared memory (PTX cp.async), waited for in
// groups: at most N groups still in flight after copies_wait<N>.
__device__ __forceinline__ void copy4_async(unsigned dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copies_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// The element `bytes` bytes after a (uniform) address.
template <typename P>
__device__ __forceinline__ P* at_byte(P* p, unsigned bytes) {
  using C = std::conditional_t<std::is_const_v<P>, const char, char>;
  return reinterpret_cast<P*>(reinterpret_cast<C*>(p) + bytes);
}

// One thread of a CTA: the launch's dt (0: nothing to do) and Ni-56 factor.
__device__ __forceinline__ void step_start(const SweepArgs<float>& a, double& dt, float& hfac) {
  const volatile Ctrl* vc = a.ctrl;
  dt = vc->status != 0 ? 0.0 : step_dt(vc, a.dt_host, a.cfl, a.t_end);
  hfac = 0.f;
  if (a.heating == HEAT_NI56) {
    const double t = vc->t;
    hfac = (float)(a.ni_lambda * (a.ni_a * exp(-t / a.ni_tni) + a.ni_qco * exp(-t / a.ni_tco)));
  }
}

// a6-a8: U^n + dt acc plus gravity and heating (gr: the radial acceleration
// of point-mass and monopole gravity).
template <int D, int NSX>
__device__ __forceinline__ void new_state2(const SweepArgs<float>& a, f2 dt, f2 gr, float hfac, const f2* Uo,
                                           const f2* acc, f2* Un) {
#pragma unroll
  for (int v = 0; v < 2 + D + NSX; ++v) Un[v] = fma2(dt, acc[v], Uo[v]);
  if (a.gravity == GRAV_UNIFORM) {
    f2 work = both(0.f);
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const f2 g = both(a.g0[d]);
      Un[1 + d] = fma2(dt * Uo[0], g, Un[1 + d]);
      work = fma2(Uo[1 + d], g, work);
    }
    Un[1 + D] = fma2(dt, work, Un[1 + D]);
  } else if (a.gravity != GRAV_NONE) {
    Un[1] = fma2(dt * Uo[0], gr, Un[1]);
    Un[1 + D] = fma2(dt, Uo[1] * gr, Un[1 + D]);
  }
  if (a.heating == HEAT_CONST) {
    Un[1 + D] = fma2(dt, both(a.heat_q), Un[1 + D]);
  } else if (a.heating == HEAT_NI56) {
    f2 rf = both(0.f);
#pragma unroll
    for (int s = 0; s < NSX; ++s)
      if (s == a.ni_index) rf = Uo[2 + D + s];
    Un[1 + D] = fma2(dt * both(hfac), rf, Un[1 + D]);
  }
}

// a9: the signal speed sum_d (|u_d| + c) ih_d and the validity of the new
// states (of the high half only if it is written).
template <int D, int NSX>
__device__ __forceinline__ void check_state2(const Gas2& gas, const f2* Un, const f2* ih, bool high, float& smax,
                                             int& err) {
  f2 Wn[2 + D + NSX];
  to_prim2<D, NSX>(Un, Wn, gas);
  const f2 cs = sound2(Wn[0], Wn[1 + D], gas);
  auto absolute = [](f2 x) { return make_f2(fabsf(lo(x)), fabsf(hi(x))); };
  f2 sp = (absolute(Wn[1]) + cs) * ih[0];
#pragma unroll
  for (int d = 1; d < D; ++d) sp = fma2(absolute(Wn[1 + d]) + cs, ih[d], sp);
  f2 nul = both(0.f);  // 0 unless a value is infinite or NaN
#pragma unroll
  for (int v = 0; v < 2 + D + NSX; ++v) nul = fma2(Un[v], both(0.f), nul);
  smax = fmaxf(smax, lo(sp));
  if (high) smax = fmaxf(smax, hi(sp));
  const bool bad0 = !(lo(nul) == 0.f && lo(Wn[0]) > 0.f && lo(Wn[1 + D]) > 0.f);
  const bool bad1 = high && !(hi(nul) == 0.f && hi(Wn[0]) > 0.f && hi(Wn[1 + D]) > 0.f);
  if (bad0 || bad1) {
    if (err == 0 && bad0) err = lo(nul) == 0.f ? ST_NEG : ST_NONFINITE;
    if (err == 0 && bad1) err = hi(nul) == 0.f ? ST_NEG : ST_NONFINITE;
  }
}

}  // namespace hydro
