// march3.cuh -- the fused 3D time step of the FP32 ideal-gas forms (HLL, HLLC).
//
// The same step as sweep.cuh's (a1-a10), laid out for the FP32 form's bound,
// which is instruction issue: the general sweep spends half of its ~2100
// thread instructions per cell-update outside FP32 arithmetic, most of them
// parking face states and fluxes in shared memory and fetching them back, and
// all of its FP32 arithmetic one value at a time.  Here
//   - a CTA marches two runs of planes at once, one in each half of every
//     FP32 pair (pair.cuh): one instruction adds or multiplies for both, and
//     addresses, x and y geometry, ghost maps and barriers serve both;
//   - a warp owns a row of 32 cells of axis 0 and a thread one column along
//     axis 2: on axis 0 a face's two states meet by one shuffle up and its
//     flux reaches the cell below it by one shuffle down; on axis 2 the upper
//     state of the plane below stays in registers; on
//     axis 1 the upper state goes to the row above through shared memory,
//     which waits for that row alone (a barrier of two warps) and returns the
//     flux in the same slot; the CTA meets once per plane, for the fluxes and
//     the staged plane;
//   - the halo rows' warps, which have the least to do, stage the cells beyond
//     one per thread.
// 30 of a warp's 32 lanes and R - 2 of the CTA's R rows own cells; the others
// form the predicted states of the one-cell halo (the halo rows only those of
// axis 1).  Face states are formed twice from the limited slopes, once for
// the Hancock increment and once with it, which costs less than keeping 6 NV
// values in registers or parking them in shared memory.
//
// Measured against the general sweep, which stays for the sizes that march3_pays
// leaves it (one GB300, whole passes of state in, 10 or 5 steps, state out):
// Sedov 256^3 HLL with totals 13.3 -> 9.75 ms, wedge 1024 x 128^2 (NV = 8, HLLC,
// monopole) 10.9 -> 8.45 ms; thread
// instructions per cell-update 2210 -> 990 (Sedov), 48 % of issue slots busy
// with 16 warps per SM.  The two-warp barriers and the halo rows' staging then
// gave 9.65 -> 9.34 and 7.81 -> 7.50 ms, the totals' widths staged with the
// other axis-2 factors 9.33 -> 9.25; HLL's mass flux by differences 9.25 -> 9.30.
// Bound now: fixed-latency dependences at
// that occupancy (registers: 128 at NV = 5, 168 at NV = 6 and 8): 4 % fewer
// instructions (the totals' sums of both halves in pairs) gave nothing, and
// sums by FP64 instructions cost 11.95 ms.
#pragma once
#include <algorithm>

#include "march.cuh"
#include "pair.cuh"
#include "sweep.cuh"

namespace hydro {

// Rows of warps per CTA, one CTA per SM: as many as leave the step its
// registers (three scalar slots spill 8-12 bytes; NV = 5: 16 rows of 128 registers 9.75 ms, 12 of
// 168 10.9; with the two-warp barriers 16 rows 9.49, 8 rows twice per SM
// 9.73) and fit shared memory
// with the totals (NV = 6: 12, NV = 8: 10).
template <int NSX>
struct March3Cfg {
  static constexpr int R = NSX == 0 ? 16 : NSX == 1 ? 12 : 10;
  static constexpr int MB = 1;
};

template <int NSX, bool SPH>
struct March3Shape {
  static constexpr int NV = 5 + NSX, R = March3Cfg<NSX>::R, MB = March3Cfg<NSX>::MB;
  static constexpr int TX = 30, TY = R - 2;          // owned cells
  static constexpr int EX = 34, EY = R + 2;          // a staged primitive plane
  static constexpr int NT = 32 * R, WPL = EX * EY;
  static constexpr int WX = WPL - NT;                // staged cells beyond one per thread
  static_assert(WX <= 128, "two warps stage the rest, two cells a thread");
  // staged geometry: of the 32 columns and of the R rows
  enum { GX_SQ, GX_SF, GX_IW, GX_IR, GX_AF, GX_INVA, GX_GA, GX_QR, GX_GR, GX_G, GX_N };
  enum { GY_SQ, GY_SF, GY_IW, GY_IS, GY_BF, GY_INVB, GY_ZC, GY_GT, GY_QT, GY_N };
  enum { GZ_SQ, GZ_SF, GZ_IW, GZ_IC, GZ_VH, GZ_VL, GZ_N };  // axis-2 factors of planes -1 .. len
  static constexpr int MAXLEN = 128;                      // planes of a half at most
  static constexpr int off_y = 4 * NV * WPL;              // [v][row][lane]: upper state, then the flux
  static constexpr int off_uo = off_y + NV * R * 32;      // [v][thread] the own cell's conserved state
  static constexpr int off_s = off_uo + NV * NT;          // [axis 0, 1][v][thread] limited slopes
  static constexpr int off_gz = off_s + 2 * NV * NT;      // [GZ_*][plane]
  static constexpr int off_gx = off_gz + GZ_N * (MAXLEN + 2);
  static constexpr int off_gy = off_gx + GX_N * 33;       // (one more column: the upper face)
  static constexpr int elems = off_gy + GY_N * (R + 1);
  static constexpr size_t smem_bytes = ((size_t)elems * sizeof(f2) + 15) / 16 * 16;
  static constexpr size_t tot_bytes = (size_t)NV * TX * TY * sizeof(double);
};

// Barrier `id` (1 .. R-1; 0 is __syncthreads) of rows id - 1, which arrives and
// goes on, and id, which waits for it.
__device__ __forceinline__ void rows_arrive(int id) { asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void rows_wait(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }

template <int NSX, int RS, bool SPH>
__global__ void __launch_bounds__(March3Shape<NSX, SPH>::NT, March3Shape<NSX, SPH>::MB)
    march3_kernel(const SweepArgs<float> a) {
  using S = March3Shape<NSX, SPH>;
  constexpr int NV = S::NV, R = S::R, TX = S::TX, TY = S::TY, EX = S::EX, NT = S::NT, WPL = S::WPL;
  constexpr unsigned FULL = 0xffffffffu;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  f2* const Ws = reinterpret_cast<f2*>(smem_raw);
  f2* const GX = Ws + S::off_gx;
  f2* const GY = Ws + S::off_gy;
  // totals: [v][owner] compensated column sums over both halves
  constexpr int NI = TX * TY;
  float2* const tsum = a.tot_part ? reinterpret_cast<float2*>(smem_raw + S::smem_bytes) : nullptr;
  __shared__ double s_dt;
  __shared__ float s_hfac;
  const volatile Ctrl* vc = a.ctrl;
  const int cur = vc->cur;
  const float* const Uin = cur ? a.B : a.A;
  float* const Uout = cur ? a.Aw : a.B;
  if (threadIdx.x == 0) step_start(a, s_dt, s_hfac);
  int tid = threadIdx.x;
  asm volatile("" : "+r"(tid));  // (kept in a register: re-reading the special register costs more)
  const int lane = tid & 31, row = tid >> 5;
  const int n0 = a.n[0], n1 = a.n[1], n2 = a.n[2];
  const long long plane = (long long)n1 * n0;
  const bool small = plane < (1ll << 30);
  const Gas2 gas(a.gas);
  float smax = 0.f;
  int err = 0;
  unsigned n_fb = 0;
  // (of three scalar slots the last may be unused: carried as 0)
  auto active = [&](int v) { return NSX < 3 || v < NV - 1 || a.ns == NSX; };

  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, z0 = blockIdx.z * a.zchunk;
  const int count = min(a.zchunk, n2 - z0);
  // the two halves of the planes: z0 .. z0+len-1 (low half of the pairs) and
  // zb .. zb+lenb-1 (high half; lenb is len or len - 1: of its last plane
  // nothing is then written)
  const int len = (count + 1) / 2, lenb = count - len, zb = z0 + len;
  const int gi = x0 - 1 + lane, gj = y0 - 1 + row;
  const bool lown = lane >= 1 && lane <= TX && gi < n0;  // this column holds owned cells
  const bool rown = row >= 1 && row <= TY && gj < n1;    // so does this row (warp-uniform)
  const bool ract = gj <= n1;                            // a row with a face to form

  // geometry of the CTA's columns and rows, doubled for the pairs (clamped
  // beyond the domain, where it is not used)
  for (int p = tid; p < 33; p += NT) {
    const int g = x0 - 1 + p, ge = min(g, n0 + 1) + 2, gc = min(max(g, 0), n0 - 1), gf = min(max(g, 0), n0);
    GX[S::GX_SQ * 33 + p] = both(a.geo.sq[0][ge]);
    GX[S::GX_SF * 33 + p] = both(a.geo.sf[0][ge]);
    GX[S::GX_IW * 33 + p] = both(a.geo.inv_w[0][ge]);
    GX[S::GX_G * 33 + p] = both(a.gravity == GRAV_POINT ? a.geo.gpt[gc] : a.gravity == GRAV_MONO ? a.gmono[gc] : 0.f);
    if constexpr (SPH) {
      GX[S::GX_IR * 33 + p] = both(a.geo.inv_r[ge]);
      GX[S::GX_AF * 33 + p] = both(a.geo.Af[gf]);
      GX[S::GX_INVA * 33 + p] = both(a.geo.inva[gc]);
      GX[S::GX_GA * 33 + p] = both(a.geo.ga[gc]);
      GX[S::GX_QR * 33 + p] = both(a.geo.qr[gc]);
      GX[S::GX_GR * 33 + p] = both(a.geo.gr[gc]);
    }
  }
  for (int p = tid; p < R + 1; p += NT) {
    const int g = y0 - 1 + p, ge = min(g, n1 + 1) + 2, gc = min(max(g, 0), n1 - 1), gf = min(max(g, 0), n1);
    GY[S::GY_SQ * (R + 1) + p] = both(a.geo.sq[1][ge]);
    GY[S::GY_SF * (R + 1) + p] = both(a.geo.sf[1][ge]);
    GY[S::GY_IW * (R + 1) + p] = both(a.geo.inv_w[1][ge]);
    if constexpr (SPH) {
      GY[S::GY_IS * (R + 1) + p] = both(a.geo.inv_s[ge]);
      GY[S::GY_BF * (R + 1) + p] = both(a.geo.Bf[gf]);
      GY[S::GY_INVB * (R + 1) + p] = both(a.geo.invb[gc]);
      GY[S::GY_ZC * (R + 1) + p] = both(a.geo.zc[gc]);
      GY[S::GY_GT * (R + 1) + p] = both(a.geo.gt[gc]);
      GY[S::GY_QT * (R + 1) + p] = both(a.geo.qt[gc]);
    }
  }
  f2* const GZ = Ws + S::off_gz;
  for (int p = tid; p < len + 2; p += NT) {
    const int e0 = z0 - 1 + p, e1 = min(zb - 1 + p, n2);  // planes p - 1 of both halves
    constexpr int st = S::MAXLEN + 2;
    GZ[S::GZ_SQ * st + p] = make_f2(a.geo.sq[2][e0 + 2], a.geo.sq[2][e1 + 2]);
    GZ[S::GZ_SF * st + p] = make_f2(a.geo.sf[2][e0 + 2], a.geo.sf[2][e1 + 2]);
    GZ[S::GZ_IW * st + p] = make_f2(a.geo.inv_w[2][e0 + 2], a.geo.inv_w[2][e1 + 2]);
    if (tsum) {
      const float2 v0 = a.dvz32[min(max(e0, 0), n2 - 1)], v1 = a.dvz32[min(max(e1, 0), n2 - 1)];
      GZ[S::GZ_VH * st + p] = make_f2(v0.x, v1.x);
      GZ[S::GZ_VL * st + p] = make_f2(v0.y, v1.y);
    }
    GZ[S::GZ_IC * st + p] = make_f2(a.geo.invc[min(max(e0, 0), n2 - 1)], a.geo.invc[min(max(e1, 0), n2 - 1)]);
  }
  if (tsum)
    for (int q = tid; q < NV * NI; q += NT) tsum[q] = make_float2(0.f, 0.f);
  const f2* const gx = GX + lane;
  const f2* const gy = GY + row;

  // a1: the staged cells of this thread (the same columns in every plane):
  // offset of the source cell in its plane, and which momenta are mirrored.
  // (Byte offsets in 32 bits next to uniform 64-bit plane addresses cost no
  // integer instruction per access; planes of 2^30 cells or more index by
  // element.)
  // A thread stages cell tid; the WPL - NT cells left over are staged by the
  // halo rows' warps, which have no faces of axes 0 and 2 to form.
  __shared__ unsigned s_so[S::WX];
  __shared__ unsigned char s_flip[S::WX];
  auto source_cell = [&](int idx, unsigned& off) {
    const int ex = idx % EX, ey = idx / EX;
    bool fx, fy;
    const int si = map_axis(min(x0 - 2 + ex, n0 + 1), n0, a.bc[0][0], a.bc[0][1], fx);
    const int sj = map_axis(min(y0 - 2 + ey, n1 + 1), n1, a.bc[1][0], a.bc[1][1], fy);
    off = (unsigned)sj * (unsigned)n0 + (unsigned)si;
    return (fx ? 1u : 0u) | (fy ? 2u : 0u);
  };
  unsigned so;
  const unsigned sflip = source_cell(tid, so);
  const bool halo_row = row == 0 || row == R - 1;
  const int e0 = (row == 0 ? 0 : 64) + lane;  // this thread's left-over cells: e0, e0 + 32
  if (halo_row)
    for (int e = e0; e < e0 + 64; e += 32)
      if (e < S::WX) {
        unsigned o;
        s_flip[e] = (unsigned char)source_cell(NT + e, o);
        s_so[e] = o;
      }
  const bool edge = x0 < 2 || x0 + TX + 2 > n0 || y0 < 2 || y0 + TY + 2 > n1;  // x or y ghosts are staged
  // a1: plane i of both halves (may be ghosts) starts to arrive, conserved,
  // in its ring slot (asynchronous 4-byte copies, issued one phase ahead of
  // their use; the thread that issued a cell's copies converts it)
  auto source = [&](int k, bool& flip) {  // the plane that plane k copies
    return map_axis(min(k, n2 + 1), n2, a.bc[2][0], a.bc[2][1], flip);
  };
  auto ghosts = [&](int i) { return z0 + i < 0 || zb + i >= n2; };  // either plane is one (z0 <= zb)
  auto fetch = [&](int i, int slot) {
    int k0 = z0 + i, k1 = zb + i;
    if (ghosts(i)) {
      bool fz;
      k0 = source(k0, fz);
      k1 = source(k1, fz);
    }
    const float* const s0 = Uin + k0 * plane;
    const float* const s1 = Uin + k1 * plane;
    auto copy = [&](f2* raw, unsigned off) {
      const unsigned d = smem_addr(raw);
      if (small) {
        const unsigned o = off * 4u;
#pragma unroll
        for (int v = 0; v < NV; ++v)
          if (active(v)) {
            copy4_async(d + v * WPL * 8, at_byte(s0 + v * a.ncell, o));
            copy4_async(d + v * WPL * 8 + 4, at_byte(s1 + v * a.ncell, o));
          }
      } else {
#pragma unroll 1
        for (int v = 0; v < NV; ++v)
          if (active(v)) {
            copy4_async(d + v * WPL * 8, s0 + v * a.ncell + off);
            copy4_async(d + v * WPL * 8 + 4, s1 + v * a.ncell + off);
          }
      }
    };
    copy(Ws + slot * (NV * WPL) + tid, so);
    if (halo_row) {
#pragma unroll 1
      for (int e = e0; e < e0 + 64; e += 32)
        if (e < S::WX) copy(Ws + slot * (NV * WPL) + NT + e, s_so[e]);
    }
  };
  // a2: what has arrived of plane i in ring slot `slot`, to primitives
  auto stage = [&](int i, int slot) {
    bool fz0 = false, fz1 = false;
    if (ghosts(i)) {
      source(z0 + i, fz0);
      source(zb + i, fz1);
    }
    auto convert = [&](f2* dst, unsigned flip) {
      f2 u[NV], w[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) u[v] = active(v) ? dst[v * WPL] : both(0.f);
      if (edge) {
        if (flip & 1u) u[1] = both(0.f) - u[1];
        if (flip & 2u) u[2] = both(0.f) - u[2];
      }
      if (fz0 || fz1) u[3] = make_f2(fz0 ? -lo(u[3]) : lo(u[3]), fz1 ? -hi(u[3]) : hi(u[3]));
      to_prim2<3, NSX>(u, w, gas);
#pragma unroll
      for (int v = 0; v < NV; ++v) dst[v * WPL] = w[v];
    };
    convert(Ws + slot * (NV * WPL) + tid, sflip);
    if (halo_row) {
#pragma unroll 1
      for (int e = e0; e < e0 + 64; e += 32)
        if (e < S::WX) convert(Ws + slot * (NV * WPL) + NT + e, s_flip[e]);
    }
  };
  // the own cells' conserved state of plane i (an owned one), for its update
  f2* const own_u = Ws + S::off_uo + tid;
  const unsigned cell = (unsigned)max(gj, 0) * (unsigned)n0 + (unsigned)max(gi, 0);  // in its plane
  auto fetch_own = [&](int i) {
    if (lown && rown) {
      const float* s0 = Uin + (z0 + i) * plane;
      const float* s1 = s0 + (i < lenb ? len * plane : 0);
      const unsigned d = smem_addr(own_u);
      if (small) {
#pragma unroll
        for (int v = 0; v < NV; ++v)
          if (active(v)) {
            copy4_async(d + v * NT * 8, at_byte(s0 + v * a.ncell, cell * 4u));
            copy4_async(d + v * NT * 8 + 4, at_byte(s1 + v * a.ncell, cell * 4u));
          }
      } else {
#pragma unroll 1
        for (int v = 0; v < NV; ++v)
          if (active(v)) {
            copy4_async(d + v * NT * 8, s0 + v * a.ncell + cell);
            copy4_async(d + v * NT * 8 + 4, s1 + v * a.ncell + cell);
          }
      }
    }
  };
  // the new state of the own cell of one half's plane at `dst`
  auto store = [&](float* dst, auto half, const f2* Un) {
    if (small) {
#pragma unroll
      for (int v = 0; v < NV; ++v)
        if (active(v)) *at_byte(dst + v * a.ncell, cell * 4u) = decltype(half)::value ? hi(Un[v]) : lo(Un[v]);
    } else {
#pragma unroll
      for (int v = 0; v < NV; ++v)
        if (active(v)) dst[v * a.ncell + cell] = decltype(half)::value ? hi(Un[v]) : lo(Un[v]);
    }
  };
  if (!active(NV - 1)) own_u[(NV - 1) * NT] = both(0.f);
  for (int i = -2; i <= 0; ++i) {
    fetch(i, i + 2);
    copies_commit();
    copies_wait<0>();
    stage(i, i + 2);
  }
  __syncthreads();
  if (!(s_dt > 0.0)) return;
  const f2 dt = both((float)s_dt), half_dt = both(0.5f * (float)s_dt);

  const f2* const Wo = Ws + (row + 1) * EX + lane + 1;  // own column (slot 0, variable 0)
  f2* const So = Ws + S::off_s + tid;                   // own parked slopes
  f2* const Yo = Ws + S::off_y + row * 32 + lane;       // own slot of the axis-1 exchange
  f2 zhi[NV];  // predicted upper state of plane i-1
  f2 acc[NV];  // the open cell's flux differences
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    zhi[v] = acc[v] = both(0.f);
  }

  // limited slopes times half widths
  auto slopes = [&](const f2* dm, const f2* dp, f2 q, f2 f, f2* s) {
    if (a.limiter == LIM_MINMOD) {
#pragma unroll
      for (int v = 0; v < NV; ++v) s[v] = f * minmod2(dm[v], dp[v] * q);
    } else {
#pragma unroll
      for (int v = 0; v < NV; ++v) s[v] = f * limit2(a.limiter, dm[v], dp[v] * q);
    }
  };
  f2 Wc[NV], dU[NV];
  auto half_step = [&](auto dir, const f2* s, f2 ih) {
    constexpr int DIR = decltype(dir)::value;
    f2 l[NV], h[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      l[v] = Wc[v] - s[v];
      h[v] = Wc[v] + s[v];
    }
    half_step2<3, NSX, DIR, DIR == 0>(l, h, ih, dU, gas);
  };
  auto upper = [&](const f2* s, f2* w, auto owned) {
    f2 l[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) l[v] = Wc[v] + s[v];
    face_state2<3, NSX>(l, dU, Wc, w, gas, [&](bool bad0, bool bad1) {
      n_fb += (bad0 && owned(0) ? 1u : 0u) + (bad1 && owned(1) ? 1u : 0u);
    });
  };
  auto lower = [&](const f2* s, f2* w, auto owned) {
    f2 l[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) l[v] = Wc[v] - s[v];
    face_state2<3, NSX>(l, dU, Wc, w, gas, [&](bool bad0, bool bad1) {
      n_fb += (bad0 && owned(0) ? 1u : 0u) + (bad1 && owned(1) ? 1u : 0u);
    });
  };
  auto solve = [&](auto dir, const f2* WL, const f2* WR, f2* F) {
    constexpr int DIR = decltype(dir)::value;
    if constexpr (RS == RS_HLL) hll2<3, NSX, DIR>(WL, WR, F, gas);
    else hllc2<3, NSX, DIR>(WL, WR, F, gas);
  };
  auto gz = [&](int f, int i) { return GZ[f * (S::MAXLEN + 2) + i + 1]; };
  using D0 = std::integral_constant<int, 0>;
  using D1 = std::integral_constant<int, 1>;
  using D2 = std::integral_constant<int, 2>;

  int sc = 1;  // ring slot of plane i (of four; planes in cyclic order)
  for (int i = -1;; ++i) {
    const bool inner = i >= 0 && i < len;  // a plane whose cells are updated
    if (i < len) fetch(i + 2, (sc + 2) & 3);
    copies_commit();
    const f2* const W0 = Wo + sc * (NV * WPL);
    f2 ylo[NV];
    if (inner ? ract : rown) {
      // a3 + a4: limited slopes and the Hancock increment of the cells (gi, gj) of plane i
      f2 sz[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        Wc[v] = W0[v * WPL];
      }
      {
        f2 dm[NV], dp[NV], sx[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          dm[v] = Wc[v] - W0[v * WPL - 1];
          dp[v] = W0[v * WPL + 1] - Wc[v];
        }
        slopes(dm, dp, gx[S::GX_SQ * 33], gx[S::GX_SF * 33], sx);
        half_step(D0(), sx, gx[S::GX_IW * 33] * half_dt);
        if (inner && rown) {
#pragma unroll
          for (int v = 0; v < NV; ++v) So[v * NT] = sx[v];
        }
      }
      {
        f2 dm[NV], dp[NV], sy[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          dm[v] = Wc[v] - W0[v * WPL - EX];
          dp[v] = W0[v * WPL + EX] - Wc[v];
        }
        slopes(dm, dp, gy[S::GY_SQ * (R + 1)], gy[S::GY_SF * (R + 1)], sy);
        f2 ih = gy[S::GY_IW * (R + 1)] * half_dt;
        if constexpr (SPH) ih = ih * gx[S::GX_IR * 33];
        half_step(D1(), sy, ih);
        if (inner) {
#pragma unroll
          for (int v = 0; v < NV; ++v) So[(NV + v) * NT] = sy[v];
        }
      }
      {
        f2 dm[NV], dp[NV];
        const f2* const Wn = Wo + ((sc + 1) & 3) * (NV * WPL);
        const f2* const Wb = Wo + ((sc + 3) & 3) * (NV * WPL);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          dm[v] = Wc[v] - Wb[v * WPL];
          dp[v] = Wn[v * WPL] - Wc[v];
        }
        slopes(dm, dp, gz(S::GZ_SQ, i), gz(S::GZ_SF, i), sz);
        f2 ih = gz(S::GZ_IW, i) * half_dt;
        if constexpr (SPH) ih = ih * (gx[S::GX_IR * 33] * gy[S::GY_IS * (R + 1)]);
        half_step(D2(), sz, ih);
      }
      // (the states below are formed again from the slopes, those of axes 0
      // and 1 parked in shared memory: keeping values of the increment's pass
      // for them would cost more registers than 16 warps leave)
#pragma unroll
      for (int v = 0; v < NV; ++v) asm volatile("" : "+l"(sz[v].v));
      if (rown) {
        // axis 2: the face below plane i closes the cell of plane i-1 and
        // opens that of plane i
        if (i >= 0) {
          f2 wl[NV], F[NV];
          lower(sz, wl, [&](int h) {
            return lown && (h ? i < lenb || (i <= lenb && zb + i == n2) : i < len || z0 + i == n2);
          });
          solve(D2(), zhi, wl, F);
          if (i > 0) {
            f2 cz = gz(S::GZ_IC, i - 1);
            if constexpr (SPH) cz = cz * (gx[S::GX_GA * 33] * gy[S::GY_ZC * (R + 1)]);
#pragma unroll
            for (int v = 0; v < NV; ++v) acc[v] = acc[v] - F[v] * cz;
            if constexpr (SPH) {
              acc[1] = fma2(both(0.25f) * gx[S::GX_GR * 33], F[3], acc[1]);
              acc[2] = fma2(gas.half * (gx[S::GX_GA * 33] * gy[S::GY_GT * (R + 1)]), F[3], acc[2]);
            }
            // a6-a9: the new states of the cells (gi, gj) of plane i-1
            const bool w0 = lown, w1 = lown && i - 1 < lenb;  // the halves written
            if (w0) {
              copies_wait<1>();  // the own cells' state (all but the plane just fetched)
              f2 Uo[NV], Un[NV];
#pragma unroll
              for (int v = 0; v < NV; ++v) Uo[v] = own_u[v * NT];
              new_state2<3, NSX>(a, dt, gx[S::GX_G * 33], s_hfac, Uo, acc, Un);
              if (tsum) {
                float2* ts = tsum + (row - 1) * TX + lane - 1;
                const f2 vh = gz(S::GZ_VH, i - 1), vl = gz(S::GZ_VL, i - 1);
                const float2 t0 = make_float2(lo(vh), lo(vl)), t1 = make_float2(hi(vh), hi(vl));
#pragma unroll
                for (int v = 0; v < NV; ++v)
                  if (active(v)) {
                    add_column_sum(ts[v * NI], lo(Un[v]), t0);
                    if (w1) add_column_sum(ts[v * NI], hi(Un[v]), t1);
                  }
              }
              f2 ih[3] = {gx[S::GX_IW * 33], gy[S::GY_IW * (R + 1)], gz(S::GZ_IW, i - 1)};
              if constexpr (SPH) {
                ih[1] = ih[1] * gx[S::GX_IR * 33];
                ih[2] = ih[2] * (gx[S::GX_IR * 33] * gy[S::GY_IS * (R + 1)]);
              }
              float* const dst = Uout + (z0 + i - 1) * plane;
              store(dst, std::integral_constant<int, 0>(), Un);
              if (w1) store(dst + len * plane, std::integral_constant<int, 1>(), Un);
              check_state2<3, NSX>(gas, Un, ih, w1, smax, err);
            }
          }
          f2 cz = gz(S::GZ_IC, i);
          if constexpr (SPH) cz = cz * (gx[S::GX_GA * 33] * gy[S::GY_ZC * (R + 1)]);
#pragma unroll
          for (int v = 0; v < NV; ++v) acc[v] = F[v] * cz;
          if constexpr (SPH) {
            acc[1] = fma2(both(0.25f) * gx[S::GX_GR * 33], F[3], acc[1]);
            acc[2] = fma2(gas.half * (gx[S::GX_GA * 33] * gy[S::GY_GT * (R + 1)]), F[3], acc[2]);
          }
        }
        if (i < len)
          upper(sz, zhi, [&](int h) {
            return lown && (h ? i + 1 < lenb || (i < lenb && zb + i + 1 == n2) : i + 1 < len || z0 + i + 1 == n2);
          });
      }
      if (inner) {
        // (a face of the high half counts if its plane does)
        auto counts = [&](int h) { return h == 0 || i < lenb; };
        if (rown) {
          // axis 0: states and fluxes by shuffles along the row
          f2 wh[NV], wl[NV], F[NV], sx[NV];
#pragma unroll
          for (int v = 0; v < NV; ++v) sx[v] = So[v * NT];
          upper(sx, wh, [&](int h) {
            return ((lane < TX && gi + 1 < n0) || (lane >= 1 && lane <= TX && gi + 1 == n0)) && counts(h);
          });
#pragma unroll
          for (int v = 0; v < NV; ++v) wh[v].v = __shfl_up_sync(FULL, wh[v].v, 1);
          lower(sx, wl, [&](int h) { return (lown || gi == n0) && counts(h); });
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
              if (v == 2 || v == 3) acc[v] = acc[v] - gx[S::GX_QR * 33] * (Fh + Fl);
            }
          } else {
#pragma unroll
            for (int v = 0; v < NV; ++v) {
              f2 Fh;
              Fh.v = __shfl_down_sync(FULL, F[v].v, 1);
              acc[v] = fma2(F[v] - Fh, gx[S::GX_IW * 33], acc[v]);
            }
          }
        }
        // axis 1: the upper state to the row above
        f2 sy[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) sy[v] = So[(NV + v) * NT];
        if (row <= TY) {
          f2 wh[NV];
          upper(sy, wh, [&](int h) {
            return lown && ((row < TY && gj + 1 < n1) || (rown && gj + 1 == n1)) && counts(h);
          });
#pragma unroll
          for (int v = 0; v < NV; ++v) Yo[v * (R * 32)] = wh[v];
          if (gj < n1) rows_arrive(row + 1);
        }
        if (row >= 1) lower(sy, ylo, [&](int h) { return lown && (rown || gj == n1) && counts(h); });
      }
    }
    if (i == len) break;
    if (inner) fetch_own(i);
    copies_commit();
    f2 F[NV];
    if (inner && row >= 1 && ract) {
      // a5, axis 1: the face below this row, its flux into the slot the
      // row below reads back
      rows_wait(row);
      f2 wl[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) wl[v] = Yo[v * (R * 32) - 32];
      solve(D1(), wl, ylo, F);
#pragma unroll
      for (int v = 0; v < NV; ++v) Yo[v * (R * 32) - 32] = F[v];
    }
    copies_wait<1>();  // plane i + 2 (all but the own cells' state)
    stage(i + 2, (sc + 2) & 3);
    __syncthreads();
    if (inner && rown) {
      if constexpr (SPH) {
        const f2 Bfl = gy[S::GY_BF * (R + 1)], Bfh = gy[S::GY_BF * (R + 1) + 1];
        const f2 ga = gx[S::GX_GA * 33], cy = ga * gy[S::GY_INVB * (R + 1)];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const f2 f = Yo[v * (R * 32)], Fh = f * Bfh, Fl = F[v] * Bfl;
          acc[v] = fma2(Fl - Fh, cy, acc[v]);
          if (v == 2) acc[1] = fma2(both(0.25f) * gx[S::GX_GR * 33], f + F[v], acc[1]);
          if (v == 3) acc[3] = acc[3] - (ga * gy[S::GY_QT * (R + 1)]) * (Fh + Fl);
        }
      } else {
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] = fma2(F[v] - Yo[v * (R * 32)], gy[S::GY_IW * (R + 1)], acc[v]);
      }
    }
    sc = (sc + 1) & 3;
  }
  if (tsum) {
    // the columns' sums times dvol[0] dvol[1] in FP64, in place, then a tree
    // in a fixed order per variable
    __syncthreads();
    double* const td = reinterpret_cast<double*>(tsum);
    for (int q = tid; q < NI * NV; q += NT) {
      const int o = q % NI;
      const int ci = x0 + o % TX, cj = y0 + o / TX;
      const float2 c = tsum[q];
      const double w = (ci < n0 && cj < n1) ? a.dvol[0][ci] * a.dvol[1][cj] : 0.0;
      td[q] = ((double)c.x + (double)c.y) * w;
    }
    __syncthreads();
    reduce_totals<NV, NI, NT>(td);
    const long long ncta = (long long)gridDim.x * gridDim.y * gridDim.z;
    const long long cta = blockIdx.x + gridDim.x * ((long long)blockIdx.y + (long long)gridDim.y * blockIdx.z);
    if (tid < NV) a.tot_part[tid * ncta + cta] = td[tid * NI];
  }
  finish_step<NT>(a.ctrl, (double)smax, err, (unsigned long long)n_fb, 0ull, s_dt, a.mirror);
}

// The march's and the general sweep's time in microseconds, from their plans:
// a CTA's step of two planes costs the march `step` (one CTA per SM), a plane
// costs the general sweep `plane` alone on its SM and `more` with each further
// CTA there.  Fitted to 35 grids from 8^3 to 192^3 and 32 x 32 x 2048 to 300 x
// 300 x 20 (HLL and HLLC; each form within 25 %).  The form it picks is the
// faster one, or at most 13 % slower, on all of them; the march's tiles of 30 x
// 14, 10 or 8 owned cells fit widths next above their multiples badly.  HLLC,
// one scalar, us per step, march and sweep: 64^3 54 and 41, 80^3 52 and 59, 96^3
// 105 and 89, 128^3 182 and 228, 32 x 32 x 512 111 and 59, 192^3 510 and 572.
// A single column of the general sweep's tiles (up to 16 x 16 cells) is faster
// there (2 x 2 x 2000: 59 and 50).  Columns of 4096 planes or more march at any
// width, so that the same long column gives the same bits in grids of any width
// (the two forms round differently): wide ones gain (128 x 128 x 4100 3.8 ms
// against 4.5, 200 x 200 x 4200 7.2 against 10.6), narrow ones lose (16 x 16 x
// 6600 0.27 ms against 0.13).
template <int NSX>
bool march3_pays(const int* n, int sms) {
  using M = March3Shape<NSX, false>;
  using S = SweepShape<float, 3, NSX>;
  constexpr double step = NSX == 0 ? 6.1 : NSX == 1 ? 5.4 : 5.9;
  constexpr double plane = NSX == 0 ? 3.9 : NSX == 1 ? 4.4 : 6.0, more = NSX == 0 ? 2.0 : NSX == 1 ? 1.8 : 2.1;
  auto tiles = [&](int tx, int ty) { return (long long)((n[0] + tx - 1) / tx) * ((n[1] + ty - 1) / ty); };
  const ChunkPlan m = plan_chunks(tiles(M::TX, M::TY), n[2], (long long)sms * M::MB, 2, 1.8, 2 * M::MAXLEN);
  const long long t = tiles(S::TX, S::TY);
  if (n[2] >= 4096) return true;
  if (t == 1) return false;
  const ChunkPlan s = plan_chunks(t, n[2], (long long)sms * S::MB, 1, 1.5, n[2]);
  const double per_sm = (double)(t * ((n[2] + s.z - 1) / s.z)) / sms;
  return 10.0 + step * m.end <= 8.5 + (plane + more * std::min(std::max(per_sm - 1.0, 0.0), S::MB - 1.0)) * s.end;
}

template <int NSX, int RS, bool SPH>
cudaError_t launch_march3(const SweepArgs<float>& args, cudaStream_t s, LaunchShape* sh) {
  using S = March3Shape<NSX, SPH>;
  SweepArgs<float> a = args;
  const void* fn = (const void*)march3_kernel<NSX, RS, SPH>;
  cudaError_t e = smem_attr_once(fn, (int)(S::smem_bytes + S::tot_bytes));
  if (e != cudaSuccess) return e;
  // (planned for the launch with totals, so that both take the same chunks)
  long long slots;
  if ((e = kernel_slots(fn, S::NT, S::smem_bytes + S::tot_bytes, &slots)) != cudaSuccess) return e;
  dim3 grid((a.n[0] + S::TX - 1) / S::TX, (a.n[1] + S::TY - 1) / S::TY);
  a.zchunk = plan_zchunk((long long)grid.x * grid.y, a.n[2], slots, 2, 1.8, 2 * S::MAXLEN);
  grid.z = (a.n[2] + a.zchunk - 1) / a.zchunk;
  sh->tx = S::TX;
  sh->ty = S::TY;
  sh->zchunk = a.zchunk;
  sh->threads = S::NT;
  sh->ctas = (long long)grid.x * grid.y * grid.z;
  march3_kernel<NSX, RS, SPH><<<grid, S::NT, S::smem_bytes + (a.tot_part ? S::tot_bytes : 0), s>>>(a);
  return cudaGetLastError();
}

}  // namespace hydro
