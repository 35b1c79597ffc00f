// march2.cuh -- the fused 2D time step of the FP32 ideal-gas forms (HLL, HLLC).
//
// The same step as sweep.cuh's (a1-a10) on pairs of cells (pair.cuh), with
// nothing shared between warps: a warp owns a strip of 28 columns (32 lanes
// with a halo of two on either side) and marches two runs of rows along axis
// 1 at once, one in each half of every pair.  Axis 0 neighbours, states and
// fluxes pass between lanes by shuffles; on axis 1 the row below's upper
// state, the slope difference and the open cell stay in registers.  So a step
// has no barrier and each state value is staged once, by asynchronous copies
// into the thread's own slots one row ahead of use.  The general sweep it
// replaces was bound by its phases: a 608-thread CTA per SM waiting at
// barriers (31 % of issue slots busy, ~1570 thread instructions per
// cell-update).  Rayleigh-Taylor 512 x 1536 (HLLC, one scalar): 84 -> 35 us
// per step, 567 thread instructions per cell-update, half of the issue slots
// busy with 11 warps per SM; bound by dependent arithmetic at that occupancy
// (128-226 registers; the CTAs per SM below leave no spills).
#pragma once
#include <algorithm>

#include "march.cuh"
#include "pair.cuh"
#include "sweep.cuh"

namespace hydro {

template <int NSX, bool SPH>
struct March2Shape {
  static constexpr int NV = 4 + NSX, NW = 4, NT = 32 * NW, MB = NSX == 0 ? 4 : NSX == 1 ? 3 : 2;
  static constexpr int TX = 28;        // owned columns of a warp
  static constexpr int MAXLEN = 64;    // rows of a half at most
  // per warp: geometry of the lanes' columns and of the rows -1 .. len (of both halves)
  enum { GX_SQ, GX_SF, GX_IW, GX_G, GX_IR, GX_AF, GX_INVA, GX_GA, GX_QR, GX_GR, GX_SPH };
  enum { GY_SQ, GY_SF, GY_IW, GY_IB, GY_BF, GY_GT, GY_SPH };
  static constexpr int GX_N = SPH ? (int)GX_SPH : (int)GX_IR, GY_N = SPH ? (int)GY_SPH : (int)GY_BF;
  static constexpr int GYL = MAXLEN + 3;
  static constexpr int off_gx = 4 * NV * NT;                 // [ring row][v][thread] conserved
  static constexpr int off_gy = off_gx + NW * GX_N * 33;
  static constexpr int elems = off_gy + NW * GY_N * GYL;
  static constexpr size_t smem_bytes = ((size_t)elems * sizeof(f2) + 15) / 16 * 16;
  static constexpr size_t tot_bytes = (size_t)NV * NT * sizeof(double);
};

template <int NSX, int RS, bool SPH>
__global__ void __launch_bounds__(March2Shape<NSX, SPH>::NT, March2Shape<NSX, SPH>::MB)
    march2_kernel(const SweepArgs<float> a) {
  using S = March2Shape<NSX, SPH>;
  constexpr int NV = S::NV, NT = S::NT, TX = S::TX;
  constexpr unsigned FULL = 0xffffffffu;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  f2* const Ws = reinterpret_cast<f2*>(smem_raw);
  double* const tsum = a.tot_part ? reinterpret_cast<double*>(smem_raw + S::smem_bytes) : nullptr;  // [v][thread]
  __shared__ double s_dt;
  __shared__ float s_hfac;
  const volatile Ctrl* vc = a.ctrl;
  const int cur = vc->cur;
  const float* const Uin = cur ? a.B : a.A;
  float* const Uout = cur ? a.Aw : a.B;
  if (threadIdx.x == 0) step_start(a, s_dt, s_hfac);
  int tid = threadIdx.x;
  asm volatile("" : "+r"(tid));  // (kept in a register: re-reading the special register costs more)
  const int lane = tid & 31;
  const int n0 = a.n[0], n1 = a.n[1];
  // the warp's strip and rows: z0 .. z0+len-1 (low half) and zb .. zb+lenb-1
  // (high half; lenb is len or len - 1: of its last row nothing is then written)
  const int strips = (n0 + TX - 1) / TX;
  const int chunks = (n1 + a.zchunk - 1) / a.zchunk;
  const int job = blockIdx.x * S::NW + (tid >> 5);
  const bool live = job < strips * chunks;
  const int x0 = (live ? job % strips : 0) * TX, z0 = (live ? job / strips : 0) * a.zchunk;
  const int count = min(a.zchunk, n1 - z0);
  const int len = (count + 1) / 2, lenb = count - len, zb = z0 + len;
  const int gi = x0 - 2 + lane;
  const bool lown = live && lane >= 2 && lane < 2 + TX && gi < n0;  // this lane holds owned cells
  auto active = [&](int v) { return NSX < 3 || v < NV - 1 || a.ns == NSX; };

  f2* const gx = Ws + S::off_gx + (tid >> 5) * (S::GX_N * 33) + lane;
  f2* const gyb = Ws + S::off_gy + (tid >> 5) * (S::GY_N * S::GYL);
  for (int q = lane; q < 33; q += 32) {
    const int g = x0 - 2 + q, ge = min(max(g, -2), n0 + 1) + 2, gc = min(max(g, 0), n0 - 1), gf = min(max(g, 0), n0);
    f2* const p = gx - lane + q;
    p[S::GX_SQ * 33] = both(a.geo.sq[0][ge]);
    p[S::GX_SF * 33] = both(a.geo.sf[0][ge]);
    p[S::GX_IW * 33] = both(a.geo.inv_w[0][ge]);
    p[S::GX_G * 33] = both(a.gravity == GRAV_POINT ? a.geo.gpt[gc] : a.gravity == GRAV_MONO ? a.gmono[gc] : 0.f);
    if constexpr (SPH) {
      p[S::GX_IR * 33] = both(a.geo.inv_r[ge]);
      p[S::GX_AF * 33] = both(a.geo.Af[gf]);
      p[S::GX_INVA * 33] = both(a.geo.inva[gc]);
      p[S::GX_GA * 33] = both(a.geo.ga[gc]);
      p[S::GX_QR * 33] = both(a.geo.qr[gc]);
      p[S::GX_GR * 33] = both(a.geo.gr[gc]);
    }
  }
  for (int q = lane; q < len + 2; q += 32) {  // row q - 1 of both halves
    const int e0 = z0 - 1 + q, e1 = min(zb - 1 + q, n1);
    const int c0 = min(max(e0, 0), n1 - 1), c1 = min(max(e1, 0), n1 - 1);
    f2* const p = gyb + q;
    p[S::GY_SQ * S::GYL] = make_f2(a.geo.sq[1][e0 + 2], a.geo.sq[1][e1 + 2]);
    p[S::GY_SF * S::GYL] = make_f2(a.geo.sf[1][e0 + 2], a.geo.sf[1][e1 + 2]);
    p[S::GY_IW * S::GYL] = make_f2(a.geo.inv_w[1][e0 + 2], a.geo.inv_w[1][e1 + 2]);
    p[S::GY_IB * S::GYL] = make_f2(a.geo.invb[c0], a.geo.invb[c1]);
    if constexpr (SPH) {
      p[S::GY_BF * S::GYL] = make_f2(a.geo.Bf[max(e0, 0)], a.geo.Bf[max(e1, 0)]);
      p[S::GY_GT * S::GYL] = make_f2(a.geo.gt[c0], a.geo.gt[c1]);
    }
  }
  auto gy = [&](int f, int i) { return gyb[f * S::GYL + i + 1]; };
  f2* const ring = Ws + tid;  // own slots: row i at ((i + 2) & 3) * NV * NT, variable v at v * NT
  if (tsum)
#pragma unroll
    for (int v = 0; v < NV; ++v) tsum[v * NT + tid] = 0.0;
  if (!active(NV - 1))
#pragma unroll
    for (int r = 0; r < 4; ++r) ring[(r * NV + NV - 1) * NT] = both(0.f);

  // a1: the lane's source column (mirrored normal momentum: fx)
  bool fx;
  const unsigned si = (unsigned)map_axis(min(gi, n0 + 1), n0, a.bc[0][0], a.bc[0][1], fx);
  auto source = [&](int k, bool& flip) { return map_axis(min(k, n1 + 1), n1, a.bc[1][0], a.bc[1][1], flip); };
  auto ghosts = [&](int i) { return z0 + i < 0 || zb + i >= n1; };
  // row i of both halves (may be ghosts) starts to arrive in the own slots
  auto fetch = [&](int i) {
    int k0 = z0 + i, k1 = zb + i;
    if (ghosts(i)) {
      bool f;
      k0 = source(k0, f);
      k1 = source(k1, f);
    }
    const float* s0 = Uin + (long long)k0 * n0 + si;
    const float* s1 = Uin + (long long)k1 * n0 + si;
    const unsigned d = smem_addr(ring + ((i + 2) & 3) * (NV * NT));
#pragma unroll
    for (int v = 0; v < NV; ++v)
      if (active(v)) {
        copy4_async(d + v * NT * 8, s0 + v * a.ncell);
        copy4_async(d + v * NT * 8 + 4, s1 + v * a.ncell);
      }
  };
  const Gas2 gas(a.gas);
  // a2: the primitives of row i
  auto row = [&](int i, f2* w) {
    f2 u[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) u[v] = ring[(((i + 2) & 3) * NV + v) * NT];
    if (fx) u[1] = both(0.f) - u[1];
    if (ghosts(i)) {
      bool f0, f1;
      source(z0 + i, f0);
      source(zb + i, f1);
      u[2] = make_f2(f0 ? -lo(u[2]) : lo(u[2]), f1 ? -hi(u[2]) : hi(u[2]));
    }
    to_prim2<2, NSX>(u, w, gas);
  };
  auto slopes = [&](const f2* dm, const f2* dp, f2 q, f2 f, f2* s) {
    if (a.limiter == LIM_MINMOD) {
#pragma unroll
      for (int v = 0; v < NV; ++v) s[v] = f * minmod2(dm[v], dp[v] * q);
    } else {
#pragma unroll
      for (int v = 0; v < NV; ++v) s[v] = f * limit2(a.limiter, dm[v], dp[v] * q);
    }
  };
  unsigned n_fb = 0;
  float smax = 0.f;
  int err = 0;
  f2 Wc[NV], Wn[NV], dU[NV];  // rows i and i + 1; the Hancock increment of row i
  f2 dy[NV];                  // W(i) - W(i-1)
  f2 yhi[NV];                 // predicted upper state of row i - 1
  f2 acc[NV];                 // the open cell's flux differences
  auto half_step = [&](auto dir, const f2* s, f2 ih) {
    constexpr int DIR = decltype(dir)::value;
    f2 l[NV], h[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      l[v] = Wc[v] - s[v];
      h[v] = Wc[v] + s[v];
    }
    half_step2<2, NSX, DIR, DIR == 0>(l, h, ih, dU, gas);
  };
  auto state = [&](const f2* s, bool up, f2* w, auto owned) {
    f2 l[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) l[v] = up ? Wc[v] + s[v] : Wc[v] - s[v];
    face_state2<2, NSX>(l, dU, Wc, w, gas, [&](bool bad0, bool bad1) {
      n_fb += (bad0 && owned(0) ? 1u : 0u) + (bad1 && owned(1) ? 1u : 0u);
    });
  };
  auto solve = [&](auto dir, const f2* WL, const f2* WR, f2* F) {
    constexpr int DIR = decltype(dir)::value;
    if constexpr (RS == RS_HLL) hll2<2, NSX, DIR>(WL, WR, F, gas);
    else hllc2<2, NSX, DIR>(WL, WR, F, gas);
  };
  using D0 = std::integral_constant<int, 0>;
  using D1 = std::integral_constant<int, 1>;

  __syncthreads();  // (dt)
  const double dtd = s_dt;
  if (!(dtd > 0.0)) return;
  const f2 dt = both((float)dtd), half_dt = both(0.5f * (float)dtd);
  if (live) {
    for (int i = -2; i <= 0; ++i) fetch(i);
    copies_commit();
    copies_wait<0>();
    {
      f2 w[NV];
      row(-2, w);
      row(-1, Wc);
      row(0, Wn);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        dy[v] = Wc[v] - w[v];
        yhi[v] = acc[v] = both(0.f);
      }
    }
    for (int i = -1;; ++i) {
      const bool inner = i >= 0 && i < len;  // a row whose cells are updated
      if (i < len) fetch(i + 2);
      copies_commit();
      // a3 + a4: limited slopes and the Hancock increment of the cells of row i
      f2 sx[NV], sy[NV];
      {
        f2 dm[NV], dp[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          f2 r;
          r.v = __shfl_down_sync(FULL, Wc[v].v, 1);
          dp[v] = r - Wc[v];
          dm[v].v = __shfl_up_sync(FULL, dp[v].v, 1);
        }
        slopes(dm, dp, gx[S::GX_SQ * 33], gx[S::GX_SF * 33], sx);
        half_step(D0(), sx, gx[S::GX_IW * 33] * half_dt);
      }
      {
        f2 dp[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) dp[v] = Wn[v] - Wc[v];
        slopes(dy, dp, gy(S::GY_SQ, i), gy(S::GY_SF, i), sy);
        f2 ih = gy(S::GY_IW, i) * half_dt;
        if constexpr (SPH) ih = ih * gx[S::GX_IR * 33];
        half_step(D1(), sy, ih);
#pragma unroll
        for (int v = 0; v < NV; ++v) dy[v] = dp[v];
      }
#pragma unroll
      for (int v = 0; v < NV; ++v) {  // (see march3.cuh: the states are formed again from the slopes)
        asm volatile("" : "+l"(sx[v].v));
        asm volatile("" : "+l"(sy[v].v));
      }
      // axis 1: the face below row i closes the cell of row i-1 and opens that of row i
      if (i >= 0) {
        f2 wl[NV], F[NV];
        state(sy, false, wl, [&](int h) {
          return lown && (h ? i < lenb || (i <= lenb && zb + i == n1) : i < len || z0 + i == n1);
        });
        solve(D1(), yhi, wl, F);
        if constexpr (SPH) {
          const f2 Bf = gy(S::GY_BF, i);
#pragma unroll
          for (int v = 0; v < NV; ++v) wl[v] = F[v] * Bf;  // area times flux
        } else {
#pragma unroll
          for (int v = 0; v < NV; ++v) wl[v] = F[v];
        }
        if (i > 0) {
          f2 cy = gy(S::GY_IB, i - 1);
          if constexpr (SPH) cy = cy * gx[S::GX_GA * 33];
#pragma unroll
          for (int v = 0; v < NV; ++v) acc[v] = acc[v] - wl[v] * cy;
          if constexpr (SPH) acc[1] = fma2(both(0.25f) * gx[S::GX_GR * 33], F[2], acc[1]);
          // a6-a9: the new states of the cells of row i-1
          if (lown) {
            const bool w1 = i - 1 < lenb;  // the high half is written too
            f2 Uo[NV], Un[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) Uo[v] = ring[(((i + 1) & 3) * NV + v) * NT];
            new_state2<2, NSX>(a, dt, gx[S::GX_G * 33], s_hfac, Uo, acc, Un);
            if (tsum) {
              // the thread's sums of U dvol[1] in FP64 (512 x 1536: 38.2 us per
              // step; with conversions 42.5; compensated FP32 pairs took 36.7
              // and lost their low words at densities below ~1e-31)
              const double t0 = a.dvol[1][z0 + i - 1], t1 = w1 ? a.dvol[1][zb + i - 1] : 0.0;
#pragma unroll
              for (int v = 0; v < NV; ++v)
                if (active(v)) {
                  double t = fma(widen(lo(Un[v])), t0, tsum[v * NT + tid]);
                  if (w1) t = fma(widen(hi(Un[v])), t1, t);
                  tsum[v * NT + tid] = t;
                }
            }
            f2 ih[2] = {gx[S::GX_IW * 33], gy(S::GY_IW, i - 1)};
            if constexpr (SPH) ih[1] = ih[1] * gx[S::GX_IR * 33];
            check_state2<2, NSX>(gas, Un, ih, w1, smax, err);
            float* const o = Uout + (long long)(z0 + i - 1) * n0 + gi;
#pragma unroll
            for (int v = 0; v < NV; ++v)
              if (active(v)) {
                o[v * a.ncell] = lo(Un[v]);
                if (w1) o[v * a.ncell + (long long)len * n0] = hi(Un[v]);
              }
          }
        }
        f2 cy = gy(S::GY_IB, i);
        if constexpr (SPH) cy = cy * gx[S::GX_GA * 33];
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] = wl[v] * cy;
        if constexpr (SPH) acc[1] = fma2(both(0.25f) * gx[S::GX_GR * 33], F[2], acc[1]);
      }
      if (i == len) break;
      state(sy, true, yhi, [&](int h) {
        return lown && (h ? i + 1 < lenb || (i < lenb && zb + i + 1 == n1) : i + 1 < len || z0 + i + 1 == n1);
      });
      if (inner) {
        // axis 0: states and fluxes by shuffles along the row
        f2 wh[NV], wl[NV], F[NV];
        state(sx, true, wh, [&](int h) {
          return ((lane >= 1 && lane < 1 + TX && gi + 1 < n0) || (lane >= 2 && lane < 2 + TX && gi + 1 == n0)) &&
                 (h == 0 || i < lenb);
        });
#pragma unroll
        for (int v = 0; v < NV; ++v) wh[v].v = __shfl_up_sync(FULL, wh[v].v, 1);
        state(sx, false, wl, [&](int h) { return (lown || (gi == n0 && lane <= 2 + TX)) && (h == 0 || i < lenb); });
        solve(D0(), wh, wl, F);
        if constexpr (SPH) {
          const f2 Afl = gx[S::GX_AF * 33], Afh = gx[S::GX_AF * 33 + 1], ia = gx[S::GX_INVA * 33];
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            f2 Fh;
            Fh.v = __shfl_down_sync(FULL, F[v].v, 1);
            Fh = Fh * Afh;
            const f2 Fl = F[v] * Afl;
            acc[v] = fma2(Fl - Fh, ia, acc[v]);
            if (v == 2) acc[2] = acc[2] - gx[S::GX_QR * 33] * (Fh + Fl);
          }
          // the absent axis: the pressure of the half-step cell state (of the
          // cell's if that one is not physical)
          f2 Uh[NV], Wh[NV];
#pragma unroll
          for (int v = 0; v < NV; ++v) Uh[v] = ring[(((i + 2) & 3) * NV + v) * NT] + dU[v];
          to_prim2<2, NSX>(Uh, Wh, gas);
          const f2 P = pick(lo(Wh[0]) > 0.f && lo(Wh[3]) > 0.f, hi(Wh[0]) > 0.f && hi(Wh[3]) > 0.f, Wh[3], Wc[3]);
          acc[1] = fma2(gas.half * gx[S::GX_GR * 33], P, acc[1]);
          acc[2] = fma2(gx[S::GX_GA * 33] * gy(S::GY_GT, i), P, acc[2]);
        } else {
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            f2 Fh;
            Fh.v = __shfl_down_sync(FULL, F[v].v, 1);
            acc[v] = fma2(F[v] - Fh, gx[S::GX_IW * 33], acc[v]);
          }
        }
      }
      copies_wait<0>();  // row i + 2
#pragma unroll
      for (int v = 0; v < NV; ++v) Wc[v] = Wn[v];
      row(i + 2, Wn);
    }
  }
  __syncthreads();
  if (tsum) {
    // the threads' sums times dvol[0] (and the absent axis's dvol[2]), then a
    // tree in a fixed order per variable
    const double w = lown ? a.dvol[0][gi] * a.dvol[2][0] : 0.0;
#pragma unroll
    for (int v = 0; v < NV; ++v) tsum[v * NT + tid] *= w;
    __syncthreads();
    reduce_totals<NV, NT, NT>(tsum);
    if (tid < NV) a.tot_part[(long long)tid * gridDim.x + blockIdx.x] = tsum[tid * NT];
  }
  finish_step<NT>(a.ctrl, (double)smax, err, (unsigned long long)n_fb, 0ull, dtd, a.mirror);
}

template <int NSX, int RS, bool SPH>
cudaError_t launch_march2(const SweepArgs<float>& args, cudaStream_t s, LaunchShape* sh) {
  using S = March2Shape<NSX, SPH>;
  SweepArgs<float> a = args;
  const void* fn = (const void*)march2_kernel<NSX, RS, SPH>;
  cudaError_t e = smem_attr_once(fn, (int)(S::smem_bytes + S::tot_bytes));
  if (e != cudaSuccess) return e;
  long long slots;
  if ((e = kernel_slots(fn, S::NT, S::smem_bytes + S::tot_bytes, &slots)) != cudaSuccess) return e;
  const int strips = (a.n[0] + S::TX - 1) / S::TX;
  a.zchunk = plan_zchunk(strips, a.n[1], slots * S::NW, 2, 1.8, 2 * S::MAXLEN);
  const long long jobs = (long long)strips * ((a.n[1] + a.zchunk - 1) / a.zchunk);
  sh->tx = S::TX;
  sh->ty = a.zchunk;
  sh->zchunk = 1;
  sh->threads = S::NT;
  sh->ctas = (jobs + S::NW - 1) / S::NW;
  march2_kernel<NSX, RS, SPH><<<(unsigned)sh->ctas, S::NT, S::smem_bytes + (a.tot_part ? S::tot_bytes : 0), s>>>(a);
  return cudaGetLastError();
}

}  // namespace hydro
