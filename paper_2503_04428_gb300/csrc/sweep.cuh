// sweep.cuh -- fused MUSCL-Hancock time step for 1D/2D/3D grids.
//
// One kernel launch is one full time step (HERACLES++ Sect. 3.2):
//   a1 ghost cells, synthesised at load time from the boundary kinds;
//   a2 primitive recovery (Eq. 5) of every staged cell;
//   a3/a4 limited slopes (Eq. 17) and the unsplit Hancock predictor (Eq. 18);
//         every predicted face state is formed once, by the cell it belongs
//         to, and parked in a shared-memory slot of its face;
//   a5 one Riemann solve per face (HLL, HLLC or exact), whose flux is written
//      over the face's left state;
//   a6 conservative update with dS/dV and the spherical sources (Eq. 13-16);
//   a7/a8 gravity (Eq. 2-4) and heating (Sect. 2.4) from the t^n state;
//   a9 the signal speed of the new state (max over cells) for the next CFL
//      time step, committed by the last CTA through the control block.
//
// Tiling: a CTA owns TX x TY cells of the (axis0, axis1) plane and, in 3D,
// marches along axis 2 over `zchunk` planes.  Shared memory holds a ring of
// three primitive planes (halo 2 on axes 0/1), the left/right states of the
// current plane's x and y faces, and the z-face states (lower side: two
// planes, upper side: one).  Thread t < TX*TY owns tile cell t for the whole
// march and keeps the partial update of its cell in the plane below in
// registers until that plane's upper z flux is known.  Each state value is
// read from HBM once per CTA (halo re-reads hit L2) and written once.
#pragma once
#include <algorithm>

#include "common.cuh"

namespace hydro {

// Tile shape per (precision, dimension, scalar slots) and the CTAs per SM
// the register budget is sized for (MB; see sweep_ctas).  The CTA has one
// thread per predictor cell (the tile plus a one-cell halo without corners),
// rounded up to whole warps.  SMALL: the 1D and 2D tiles of grids whose large
// tiles would leave SMs idle (see small_tile): 28 cells and their halo fill
// one warp, 8 x 8 three (FP64: twice as many, see Sweep::predictor_split).
template <typename T, int DIM, int NSX, bool SMALL>
struct TileCfg {
  static constexpr int TX = DIM == 1 ? (SMALL ? 28 : 254) : (SMALL ? 8 : 16);
  static constexpr int TY = DIM == 1 ? 1 : SMALL ? 8 : (DIM == 3 && NSX == 3 && sizeof(T) == 8) ? 8 : 16;
  // (FP32 3D without scalars: three CTAs of 64 registers)
  static constexpr int MB = DIM == 1 || SMALL ? 1 : DIM == 2 ? 2 : sizeof(T) == 8 ? 1 : NSX == 0 ? 3 : 2;
};

// The smallest power of two >= n (n >= 1).
__host__ __device__ constexpr int pow2_ceil(int n) { return n <= 1 ? 1 : 2 * pow2_ceil((n + 1) / 2); }

template <typename T, int DIM, int NSX, bool SMALL = false>
struct SweepShape {
  static constexpr int NV = 2 + DIM + NSX;
  static constexpr int TX = TileCfg<T, DIM, NSX, SMALL>::TX;
  static constexpr int TY = TileCfg<T, DIM, NSX, SMALL>::TY;
  static constexpr int HY = DIM >= 2 ? 2 : 0;              // primitive halo along axis 1
  static constexpr int EX = TX + 4, EY = TY + 2 * HY;      // primitive plane extents
  static constexpr int QY = DIM >= 2 ? 1 : 0;              // predictor halo along axis 1
  static constexpr int WP = DIM == 3 ? 3 : 1;              // primitive planes in flight
  static constexpr int NI = TX * TY;                        // tile cells, one owner thread each
  static constexpr int NH = 2 * TY + (DIM >= 2 ? 2 * TX : 0);  // halo predictor cells
  static constexpr int NP = NI + NH;                        // predictor cells
  static constexpr int NPT = (NP + 31) / 32 * 32;
  // threads per CTA: one per predictor cell, for the small FP64 tiles two (see
  // Sweep::predictor_split)
  static constexpr bool TWO = SMALL && sizeof(T) == 8;
  static constexpr int NT = TWO ? 2 * NPT : NPT;
  static constexpr int MB = TileCfg<T, DIM, NSX, SMALL>::MB;       // resident CTAs per SM (register budget)
  static constexpr int WPL = EX * EY;
  static constexpr int NFX = (TX + 1) * TY;
  static constexpr int NFY = DIM >= 2 ? TX * (TY + 1) : 0;
  static constexpr int NFZ = DIM == 3 ? TX * TY : 0;
  static constexpr size_t smem_elems = (size_t)WP * NV * WPL + (size_t)2 * NV * NFX +
                                       (size_t)2 * NV * NFY + (size_t)3 * NV * NFZ;
  static constexpr size_t dual_elems = (size_t)2 * (NFX + NFY + NFZ);  // dual-energy face terms
  // radiation EoS: face-state temperatures and those of the primitive planes
  static constexpr size_t rad_elems = (size_t)2 * NFX + 2 * NFY + 3 * NFZ + (size_t)WP * WPL;
  // FP64, ideal gas: the face states' sound speeds, in the temperatures' place
  static constexpr size_t snd_elems = (size_t)2 * NFX + 2 * NFY + 3 * NFZ;
  __host__ __device__ static constexpr size_t face_elems(int mode) {
    return (mode & 1) ? rad_elems : sizeof(T) == 8 ? snd_elems : 0;
  }
  // the x and y geometry factors of the CTA's cells, staged once per CTA
  // (GX_N arrays over the TX + 2 predictor columns, GY_N over the TY + 2 rows)
  enum { GX_SQ, GX_SF, GX_IW, GX_IR, GX_AF, GX_INVA, GX_GA, GX_QR, GX_GR, GX_G, GX_N };
  enum { GY_SQ, GY_SF, GY_IW, GY_IS, GY_BF, GY_INVB, GY_ZC, GY_GT, GY_QT, GY_N };
  static constexpr size_t geo_elems = (size_t)GX_N * (TX + 2) + (DIM >= 2 ? (size_t)GY_N * (TY + 2) : 0);
  static constexpr size_t split_elems = TWO && DIM == 2 ? (size_t)2 * NV * NPT : 0;  // what the two exchange
  __host__ __device__ static constexpr size_t smem_bytes_for(int mode) {
    return (smem_elems + ((mode & 2) ? dual_elems : 0) + face_elems(mode) + geo_elems + split_elems) * sizeof(T);
  }
  // conserved totals accumulated in the step: one FP64 sum per owner and
  // variable, after the rest (16-byte aligned)
  __host__ __device__ static constexpr size_t tot_offset(int mode) { return (smem_bytes_for(mode) + 15) / 16 * 16; }
  static constexpr size_t tot_bytes = (size_t)NI * NV * sizeof(double);
};

// Ghost mapping of one axis (periodic wrap, transmissive copy of the edge
// cell, reflective mirror with the normal momentum negated).  g in [-2, n+1].
__device__ __forceinline__ int map_axis(int g, int n, int lo, int hi, bool& flip) {
  flip = false;
  if (g < 0) {
    if (lo == BC_PERIODIC) return g + n;
    if (lo == BC_TRANSMISSIVE) return 0;
    flip = true;
    return -1 - g;
  }
  if (g >= n) {
    if (hi == BC_PERIODIC) return g - n;
    if (hi == BC_TRANSMISSIVE) return n - 1;
    flip = true;
    return 2 * n - 1 - g;
  }
  return g;
}

// The same with exchanged sides (domain decomposition): a ghost of an
// exchanged side sets `layer` to its distance - 1 from the side and returns
// 0; layer stays -1 otherwise.
__device__ __forceinline__ int map_axis(int g, int n, int lo, int hi, bool& flip, int& layer) {
  flip = false;
  if ((g < 0 && lo == BC_EXCHANGED) || (g >= n && hi == BC_EXCHANGED)) {
    layer = g < 0 ? -1 - g : g - n;
    return 0;
  }
  if (g < 0) {
    if (lo == BC_PERIODIC) return g + n;
    if (lo == BC_TRANSMISSIVE) return 0;
    flip = true;
    return -1 - g;
  }
  if (g >= n) {
    if (hi == BC_PERIODIC) return g - n;
    if (hi == BC_TRANSMISSIVE) return n - 1;
    flip = true;
    return 2 * n - 1 - g;
  }
  return g;
}

// Asynchronous copy of one element to shared memory (PTX cp.async).
template <typename T>
__device__ __forceinline__ void copy_async(T* dst, const T* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "n"(sizeof(T))
               : "memory");
}

// The CTA's totals of its NI owners' sums [v][owner], by a tree in a fixed
// order per variable (so the result does not depend on scheduling), left in
// sums[v][0].
template <int NV, int NI, int NT>
__device__ void reduce_totals(double* sums) {
  for (int w = pow2_ceil(NI) / 2; w > 0; w >>= 1) {
    for (int q = threadIdx.x; q < NV * w; q += NT) {
      const int v = q / w, o = q - v * w;
      if (o + w < NI) sums[v * NI + o] += sums[v * NI + o + w];
    }
    __syncthreads();
  }
}

// Which face states a predictor pass writes.
enum { PRED_ALL = 0, PRED_ZHI = 1, PRED_ZLO = 2 };

// MODE bit 0: gas + radiation EoS (Eq. 6-7); bit 1: dual-energy correction
// (Sect. 2.5); bit 2: a slab of a decomposed grid or a moving grid (exchanged
// ghosts, moving faces; ideal gas only).  Each combination is its own
// instantiation, so the plain step carries none of the optional work.
// SMALL: the small tiles; MULTI: several steps in one launch (sweep_steps_kernel).
template <typename T, int DIM, int NSX, int RS, int MODE, bool SMALL, bool MULTI = false>
struct Sweep {
  static constexpr int EOS = MODE & 1;
  static constexpr bool DUAL = (MODE & 2) != 0;
  // A face state's sound speed is formed with the state, whose 1/rho is at
  // hand (FP64: three operations of its pipe per state; FP32 reciprocals are
  // cheaper than the exchange).
  static constexpr bool SND = EOS == 0 && sizeof(T) == 8 && RS != RS_EXACT;
  static constexpr bool XM = (MODE & 4) != 0;
  // in-step totals as compensated FP32 column sums (FP32, 3D) instead of FP64 sums per cell
  static constexpr bool COLSUM = sizeof(T) == 4 && DIM == 3;
  using S = SweepShape<T, DIM, NSX, SMALL>;
  static constexpr int NV = S::NV, TX = S::TX, TY = S::TY, EX = S::EX, EY = S::EY, HY = S::HY,
                       QY = S::QY, NT = S::NT, NI = S::NI, NP = S::NP, NFX = S::NFX,
                       NFY = S::NFY, NFZ = S::NFZ;

  const SweepArgs<T>& a;
  T* Ws;  // primitive planes [slot][v][ey][ex]
  T* XL;  // x faces [v][row*(TX+1)+f]: left state, then the flux
  T* XR;  // x faces: right state
  T* YL;  // y faces [v][fy*TX+col]: left (lower) state, then the flux
  T* YR;
  T* ZL;  // [2][v][j*TX+i]: state below the z face above plane (slot = plane & 1)
  T* ZR;  // [v][j*TX+i]: state above the z face below the current plane, then the flux
  T* XQ;  // dual energy (Sect. 2.5): [2][face] u_f e_f and u_f of the x faces
  T* YQ;  //   ... of the y faces
  T* ZQ;  //   ... of the z face below the current plane
  // radiation EoS: temperatures of the parked face states (same indices as
  // XL/XR, YL/YR, ZL (two planes), ZR)
  T* XTL;
  T* XTR;
  T* YTL;
  T* YTR;
  T* ZTL;
  T* ZTR;
  T* WT;  // [slot][ey][ex] temperatures of the primitive planes
  T* GXs;  // [GX_*][px] geometry of predictor column px (cell x0 - 1 + px)
  T* GYs;  // [GY_*][py] geometry of predictor row py (cell y0 - 1 + py)
  double* tsum;  // [v][owner] sums of U dV of the owner's new cells (FP32 3D: float2 column sums
                 // until the end of the CTA, see close_cell), or null (totals off)
  int x0, y0, z1, n2;
  T dt, half_dt;
  const T* Uin;
  T* Uout;
  unsigned long long n_fallback = 0, n_iters = 0;
  int t_iters = 0;  // radiation EoS: temperature Newton iterations of this thread (reported as n_iters)
  int err = 0;
  T smax = T(0);  // max of the new states' signal speeds (FP32: the FP64 max of
                  // the same values, converted once at the end: the conversion is exact)
  T hfac = T(0);
  // owner registers: partial update of the owned cell, its predictor
  // increment (1D/2D) and the spherical partial sums of Eq. 13-16
  T acc[NV];
  T dUo[NV];
  T fzb3 = T(0), tth = T(0), x2 = T(0), s3 = T(0);
  T Ucell[MULTI ? NV : 1];  // several steps per launch: the owned cell's conserved state
  T aq1 = T(0), aq2 = T(0);  // dual energy: divergences of u e and of u (times dt^-1)
  T topen = T(0);            // radiation EoS: the open cell's temperature (its plane's slot is refilled before it closes)

  __device__ Sweep(const SweepArgs<T>& args, T* smem) : a(args) {
    Ws = smem;
    tsum = args.tot_part ? reinterpret_cast<double*>(reinterpret_cast<unsigned char*>(smem) + S::tot_offset(MODE))
                         : nullptr;
    XL = Ws + S::WP * NV * S::WPL;
    XR = XL + NV * NFX;
    YL = XR + NV * NFX;
    YR = YL + NV * NFY;
    ZL = YR + NV * NFY;
    ZR = ZL + 2 * NV * NFZ;
    // the dual-energy and temperature arrays exist only in the instantiations
    // that use them
    XQ = ZR + NV * NFZ;
    YQ = XQ + 2 * NFX;
    ZQ = YQ + 2 * NFY;
    XTL = DUAL ? ZQ + 2 * NFZ : XQ;
    XTR = XTL + NFX;
    YTL = XTR + NFX;
    YTR = YTL + NFY;
    ZTL = YTR + NFY;
    ZTR = ZTL + 2 * NFZ;
    WT = ZTR + NFZ;
    GXs = Ws + S::smem_elems + (DUAL ? S::dual_elems : 0) + S::face_elems(MODE);
    GYs = GXs + S::GX_N * (TX + 2);
  }

  __device__ __forceinline__ T gx(int k, int px) const { return GXs[k * (TX + 2) + px]; }
  __device__ __forceinline__ T gy(int k, int py) const { return GYs[k * (TY + 2) + py]; }

  // Stage the x and y geometry factors of the CTA's cells (constant over
  // the march; read after the first barrier).  Indices are clamped to the
  // arrays' ranges: entries of columns or rows beyond the domain are never
  // used.
  __device__ void stage_geometry() {
    const int n0 = a.n[0], n1 = a.n[1];
    for (int p = threadIdx.x; p < TX + 2; p += NT) {
      const int gi = x0 - 1 + p;              // >= -1
      const int ge = min(gi, n0 + 1) + 2;     // extended (ghost) index
      const int gc = min(max(gi, 0), n0 - 1);  // interior cell
      const int gf = min(max(gi, 0), n0);      // interior face
      T* g = GXs + p;
      constexpr int st = TX + 2;
      g[S::GX_SQ * st] = a.geo.sq[0][ge];
      g[S::GX_SF * st] = a.geo.sf[0][ge];
      g[S::GX_IW * st] = a.geo.inv_w[0][ge];
      g[S::GX_IR * st] = a.spherical ? a.geo.inv_r[ge] : T(1);
      g[S::GX_AF * st] = a.geo.Af[gf];
      g[S::GX_INVA * st] = a.geo.inva[gc];
      g[S::GX_GA * st] = a.geo.ga[gc];
      g[S::GX_QR * st] = a.geo.qr[gc];
      g[S::GX_GR * st] = a.geo.gr[gc];
      g[S::GX_G * st] = a.gravity == GRAV_POINT ? a.geo.gpt[gc] : a.gravity == GRAV_MONO ? a.gmono[gc] : T(0);
    }
    if constexpr (DIM >= 2) {
      for (int p = threadIdx.x; p < TY + 2; p += NT) {
        const int gj = y0 - 1 + p;
        const int ge = min(gj, n1 + 1) + 2;
        const int gc = min(max(gj, 0), n1 - 1);
        const int gf = min(max(gj, 0), n1);
        T* g = GYs + p;
        constexpr int st = TY + 2;
        g[S::GY_SQ * st] = a.geo.sq[1][ge];
        g[S::GY_SF * st] = a.geo.sf[1][ge];
        g[S::GY_IW * st] = a.geo.inv_w[1][ge];
        g[S::GY_IS * st] = a.spherical ? a.geo.inv_s[ge] : T(1);
        g[S::GY_BF * st] = a.geo.Bf[gf];
        g[S::GY_INVB * st] = a.geo.invb[gc];
        g[S::GY_ZC * st] = a.geo.zc[gc];
        g[S::GY_GT * st] = a.geo.gt[gc];
        g[S::GY_QT * st] = a.geo.qt[gc];
      }
    }
  }

  // Dual energy (Sect. 2.5, reading R15): the advected internal energy
  // u_f e_f = F_rho (e/rho)_upwind and the face velocity u_f = F_rho/rho_upwind,
  // upwind by the sign of the mass flux.
  __device__ __forceinline__ void dual_terms(const T* WL, const T* WR, const T* F, T* q, int st,
                                             int idx) const {
    const T* Wu = F[0] >= T(0) ? WL : WR;
    const T eu = eint_of(gas(), Wu[0], Wu[1 + DIM]);
    q[idx] = F[0] * eu / Wu[0];
    q[st + idx] = F[0] / Wu[0];
  }

  // the EoS of this instantiation: ideal gas (Eq. 5) or gas + radiation (Eq. 6-7)
  __device__ __forceinline__ const auto& gas() const {
    if constexpr (EOS == 1) return a.grad;
    else return a.gas;
  }

  // State loads: several steps per launch read other CTAs' fresh cells, from L2.
  static __device__ __forceinline__ T load(const T* p) {
    if constexpr (MULTI) return __ldcg(p);
    else return __ldg(p);
  }

  __device__ __forceinline__ T& W(int slot, int v, int ey, int ex) {
    return Ws[((slot * NV + v) * EY + ey) * EX + ex];
  }
  static __device__ __forceinline__ int wslot(int gz) { return DIM == 3 ? (gz + 6) % 3 : 0; }

  // a1 + a2: stage plane gz (axis-2 index, may be a ghost) as primitives.
  __device__ void load_plane(int gz) {
    const int n0 = a.n[0], n1 = a.n[1];
    bool fz = false;
    int lz = -1;
    int sz = 0;
    if constexpr (DIM == 3) {
      if constexpr (XM) sz = map_axis(gz, a.n[2], a.bc[2][0], a.bc[2][1], fz, lz);
      else sz = map_axis(gz, a.n[2], a.bc[2][0], a.bc[2][1], fz);
    }
    const int slot = wslot(gz);
    const int nvact = NSX < 3 ? NV : 2 + DIM + a.ns;
    // a staged region inside the domain on every axis: no ghost mapping
    const bool inner = !XM && x0 >= 2 && x0 + TX + 2 <= n0 &&
                       (DIM < 2 || (y0 >= HY && y0 + TY + HY <= n1)) && (DIM < 3 || (gz >= 0 && gz < a.n[2]));
    if (inner) {
      const long long zoff = (long long)gz * n1 * n0;
      for (int idx = threadIdx.x; idx < S::WPL; idx += NT) {
        const int ex = idx % EX, ey = idx / EX;
        const long long c = zoff + (long long)(y0 - HY + ey) * n0 + (x0 - 2 + ex);
        T u[NV], w[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) u[v] = v < nvact ? load(Uin + (long long)v * a.ncell + c) : T(0);
        if constexpr (EOS == 1) {
          T c2, t;
          int k = 0;
          to_prim_ct<T, DIM, NSX>(u, w, c2, t, a.grad, T(0), &k);
          t_iters += k;
          WT[(slot * EY + ey) * EX + ex] = t;
        } else {
          to_prim<T, DIM, NSX>(u, w, gas());
        }
#pragma unroll
        for (int v = 0; v < NV; ++v) W(slot, v, ey, ex) = w[v];
      }
      return;
    }
    for (int idx = threadIdx.x; idx < S::WPL; idx += NT) {
      const int ex = idx % EX, ey = idx / EX;
      const int gi = min(x0 - 2 + ex, n0 + 1);
      bool fx, fy = false;
      int lx = -1, ly = -1;
      int si, sj = 0, gj = 0;
      if constexpr (XM) si = map_axis(gi, n0, a.bc[0][0], a.bc[0][1], fx, lx);
      else si = map_axis(gi, n0, a.bc[0][0], a.bc[0][1], fx);
      if (DIM >= 2) {
        gj = min(y0 - HY + ey, n1 + 1);
        if constexpr (XM) sj = map_axis(gj, n1, a.bc[1][0], a.bc[1][1], fy, ly);
        else sj = map_axis(gj, n1, a.bc[1][0], a.bc[1][1], fy);
      }
      T u[NV], w[NV];
      const int layer = XM ? max(lx, max(ly, lz)) : -1;  // >= 0: a ghost of an exchanged side
      if (layer < 0) {
        const long long c = ((long long)sz * n1 + sj) * n0 + si;
#pragma unroll
        for (int v = 0; v < NV; ++v) u[v] = v < nvact ? load(Uin + (long long)v * a.ncell + c) : T(0);
      } else {
        // the neighbour subdomain's cell, from the halo of that side; the
        // other axes are mapped (and flipped) as for any ghost
        const int side = (lx >= 0 ? gi : ly >= 0 ? gj : gz) < 0 ? 0 : 1;
        const long long nx = a.xaxis == 0 ? (long long)n1 * a.n[2] : a.xaxis == 1 ? (long long)n0 * a.n[2]
                                                                                 : (long long)n0 * n1;
        const long long q = a.xaxis == 0 ? (long long)sz * n1 + sj : a.xaxis == 1 ? (long long)sz * n0 + si
                                                                                 : (long long)sj * n0 + si;
        const T* hp = a.halo[side] + (long long)layer * nx + q;
#pragma unroll
        for (int v = 0; v < NV; ++v) u[v] = v < nvact ? hp[(long long)v * 2 * nx] : T(0);
      }
      if (fx) u[1] = -u[1];
      if (DIM >= 2 && fy) u[2] = -u[2];
      if (DIM == 3 && fz) u[3] = -u[3];
      if constexpr (EOS == 1) {
        T c2, t;
        int k = 0;  // (a local counter: a register after inlining)
        to_prim_ct<T, DIM, NSX>(u, w, c2, t, a.grad, T(0), &k);
        t_iters += k;
        WT[(slot * EY + ey) * EX + ex] = t;
      } else {
        to_prim<T, DIM, NSX>(u, w, gas());
      }
#pragma unroll
      for (int v = 0; v < NV; ++v) W(slot, v, ey, ex) = w[v];
    }
  }

  // load_plane in two parts (3D; exchanged halos: all in the second):
  // asynchronous copies of the conserved state into the plane's slot, and
  // their conversion in place by the threads that issued them, with the faces
  // of an earlier plane between.  Threads count from the CTA's end, as the
  // cells beyond one per thread then fall to warps that have fewer faces to
  // solve.  (Loads waited for at once: wedge with radiation 512 x 96^2 4.54
  // ms per 5 steps against 4.45, Sedov 128^3 FP64 9.35 per 3 against 9.14.)
  template <typename F>
  __device__ __forceinline__ void staged_cells(int gz, F&& each) {
    const int n0 = a.n[0], n1 = a.n[1];
    bool fz;
    const int sz = map_axis(gz, a.n[2], a.bc[2][0], a.bc[2][1], fz);
    const bool inner = x0 >= 2 && x0 + TX + 2 <= n0 && y0 >= HY && y0 + TY + HY <= n1;
    const long long zoff = (long long)sz * n1 * n0;
    for (int idx = NT - 1 - (int)threadIdx.x; idx < S::WPL; idx += NT) {
      int si = x0 - 2 + idx % EX, sj = y0 - HY + idx / EX;
      bool fx = false, fy = false;
      if (!inner) {
        si = map_axis(min(si, n0 + 1), n0, a.bc[0][0], a.bc[0][1], fx);
        sj = map_axis(min(sj, n1 + 1), n1, a.bc[1][0], a.bc[1][1], fy);
      }
      each(idx, zoff + (long long)sj * n0 + si, fx, fy, fz);
    }
  }
  __device__ __forceinline__ void fetch_plane(int gz) {
    if constexpr (!XM) {
      T* const dst = Ws + wslot(gz) * (NV * S::WPL);
      const int nvact = NSX < 3 ? NV : 2 + DIM + a.ns;
      staged_cells(gz, [&](int idx, long long c, bool, bool, bool) {
#pragma unroll
        for (int v = 0; v < NV; ++v)
          if (v < nvact) copy_async(dst + v * S::WPL + idx, Uin + (long long)v * a.ncell + c);
      });
      asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
  }
  __device__ __forceinline__ void finish_plane(int gz) {
    if constexpr (!XM) {
      T* const dst = Ws + wslot(gz) * (NV * S::WPL);
      const int nvact = NSX < 3 ? NV : 2 + DIM + a.ns;
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
      staged_cells(gz, [&](int idx, long long, bool fx, bool fy, bool fz) {
        T u[NV], w[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) u[v] = v < nvact ? dst[v * S::WPL + idx] : T(0);
        if (fx) u[1] = -u[1];
        if (fy) u[2] = -u[2];
        if (fz) u[3] = -u[3];
        if constexpr (EOS == 1) {
          T c2, t;
          int k = 0;
          to_prim_ct<T, DIM, NSX>(u, w, c2, t, a.grad, T(0), &k);
          t_iters += k;
          WT[wslot(gz) * S::WPL + idx] = t;
        } else {
          to_prim<T, DIM, NSX>(u, w, gas());
        }
#pragma unroll
        for (int v = 0; v < NV; ++v) dst[v * S::WPL + idx] = w[v];
      });
    } else {
      load_plane(gz);
    }
  }

  // 1/h_d of the cell in predictor column px, row py, plane gk (physical
  // width: h_r = dr, h_th = r dth, h_ph = r s dph).
  __device__ __forceinline__ T inv_h(int d, int px, int py, int gk) const {
    if (d == 0) return gx(S::GX_IW, px);
    if (d == 1) {
      const T w = gy(S::GY_IW, py);
      return a.spherical ? w * gx(S::GX_IR, px) : w;
    }
    const T w = a.geo.inv_w[2][gk + 2];
    if constexpr (DIM >= 2) return a.spherical ? w * gx(S::GX_IR, px) * gy(S::GY_IS, py) : w;
    else return w;
  }

  // Limited low/high face states along DIR of the cell with centre Wc and
  // neighbours Wm/Wp; l = the cell's predictor column (DIR 0), row (DIR 1)
  // or plane index (DIR 2).
  template <int DIR>
  __device__ __forceinline__ void faces_of(const T* Wm, const T* Wc, const T* Wp, int l, T* Wlo,
                                           T* Whi) const {
    // the limiters are homogeneous: (dm idm, dp idp) -> idm limit(dm, dp q)
    T q, f;
    if constexpr (DIR == 0) {
      q = gx(S::GX_SQ, l);
      f = gx(S::GX_SF, l);
    } else if constexpr (DIR == 1) {
      q = gy(S::GY_SQ, l);
      f = gy(S::GY_SF, l);
    } else {
      q = a.geo.sq[DIR][l + 2];
      f = a.geo.sf[DIR][l + 2];
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const T sig = limit<T>(a.limiter, Wc[v] - Wm[v], (Wp[v] - Wc[v]) * q);
      Wlo[v] = Wc[v] - f * sig;
      Whi[v] = Wc[v] + f * sig;
    }
  }

  // Predictor cell of item t: (px, py) in the (TX+2) x (TY+2QY) region around
  // the tile.  Items 0..NI-1 are the tile cells in owner order, then the
  // axis-0 halo columns, then the axis-1 halo rows (corners are never needed).
  static __device__ __forceinline__ void item_cell(int t, int& px, int& py) {
    if (t < NI) {
      px = 1 + t % TX;
      py = QY + t / TX;
      return;
    }
    int h = t - NI;
    if (h < 2 * TY) {
      px = h < TY ? 0 : TX + 1;
      py = QY + (h < TY ? h : h - TY);
      return;
    }
    h -= 2 * TY;
    px = 1 + (h < TX ? h : h - TX);
    py = h < TX ? 0 : TY + 1;
  }

  // Turn the limited state parked at p (stride `st`) into the predicted face
  // state: W -> U, + dU, U -> W; a non-physical result falls back to Wc.
  // The radiation EoS parks the conserved state (the flux evaluation already
  // solved for its energy) and records the temperature of the result at tp;
  // SND: its sound speed.
  __device__ __forceinline__ void finish_state(T* p, int st, const T* Wc, const T* dU, bool owned,
                                               T* tp = nullptr) {
    T w[NV], u[NV];
    if constexpr (EOS == 1) {
#pragma unroll
      for (int v = 0; v < NV; ++v) u[v] = p[v * st] + dU[v];
      const T rho = u[0], ir = T(1) / rho;
      T ke = T(0);
#pragma unroll
      for (int d = 0; d < DIM; ++d) {
        w[1 + d] = u[1 + d] * ir;
        ke += u[1 + d] * w[1 + d];
      }
      w[0] = rho;
      T c2, t;
      int k = 0;
      a.grad.from_e_t(rho, u[1 + DIM] - T(0.5) * ke, w[1 + DIM], c2, t, *tp, &k);
#pragma unroll
      for (int s = 0; s < NSX; ++s) w[2 + DIM + s] = u[2 + DIM + s] * ir;
      if (!is_pos(w[0]) || !is_pos(w[1 + DIM])) {
#pragma unroll
        for (int v = 0; v < NV; ++v) w[v] = Wc[v];
        t = a.grad.temp_p(Wc[0], Wc[1 + DIM], *tp, &k);
        if (owned) ++n_fallback;
      }
      *tp = t;
      t_iters += k;
    } else {
      // the slot holds the limited state's conserved form (limited_fluxes)
#pragma unroll
      for (int v = 0; v < NV; ++v) u[v] = p[v * st] + dU[v];
      to_prim<T, DIM, NSX>(u, w, gas());
      T e, c = T(0);
      if constexpr (SND) face_e_c<T>(a.gas, w[0], w[1 + DIM], T(0), e, c);
      if (!is_pos(w[0]) || !is_pos(w[1 + DIM])) {
#pragma unroll
        for (int v = 0; v < NV; ++v) w[v] = Wc[v];
        if constexpr (SND) face_e_c<T>(a.gas, w[0], w[1 + DIM], T(0), e, c);
        if (owned) ++n_fallback;
      }
      if constexpr (SND) *tp = c;
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) p[v * st] = w[v];
  }

  // Physical fluxes of the two limited states of one direction and what is
  // parked in their face slots: their conserved states (for the radiation
  // EoS from the same temperature solve).
  // (radiation EoS: tc = the cell's temperature, the Newton start; tl/th
  // receive the limited states' temperatures)
  template <int DIR>
  __device__ __forceinline__ void limited_fluxes(const T* Wl, const T* Wh, T* Fl, T* Fh, T* Pl, T* Ph,
                                                 T tc = T(0), T* tl = nullptr, T* th = nullptr) {
    if constexpr (EOS == 1) {
      T c2;
      int k = 0;
      *tl = a.grad.temp_p(Wl[0], Wl[1 + DIM], tc, &k);
      *th = a.grad.temp_p(Wh[0], Wh[1 + DIM], tc, &k);
      t_iters += k;
      T el, eh;
      a.grad.from_t(Wl[0], *tl, el, c2);
      a.grad.from_t(Wh[0], *th, eh, c2);
      flux_cons_e<T, DIM, NSX, DIR>(Wl, el, Fl, Pl);
      flux_cons_e<T, DIM, NSX, DIR>(Wh, eh, Fh, Ph);
    } else {
      // the fluxes and the conserved states together (the same operations
      // as phys_flux and to_cons, each done once)
      flux_cons_e<T, DIM, NSX, DIR>(Wl, Wl[1 + DIM] * a.gas.igm1, Fl, Pl);
      flux_cons_e<T, DIM, NSX, DIR>(Wh, Wh[1 + DIM] * a.gas.igm1, Fh, Ph);
    }
  }

  // Moving grid (reading R16): along the moving axis the predictor uses the
  // fluxes through faces that move with the grid, F - w U (ideal gas).
  // (ul, uh: the limited states' conserved forms, as parked by limited_fluxes)
  __device__ __forceinline__ void moving_fluxes(const T* ul, const T* uh, T* Fl, T* Fh) const {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      Fl[v] -= a.wg * ul[v];
      Fh[v] -= a.wg * uh[v];
    }
  }

  // The difference of the physical fluxes of the two limited states along
  // DIR (see limited_fluxes).
  template <int DIR>
  __device__ __forceinline__ void limited_diff(const T* Wl, const T* Wh, T* dF, T* Pl, T* Ph, T tc, T* tl, T* th) {
    if constexpr (EOS == 0 && sizeof(T) == 8) {
      flux_diff<DIM, NSX, DIR>(Wl, Wh, a.gas.igm1, dF, Pl, Ph);
      if constexpr (XM) {
        if (a.maxis == DIR) {
#pragma unroll
          for (int v = 0; v < NV; ++v) dF[v] -= a.wg * (Pl[v] - Ph[v]);
        }
      }
    } else {
      T Fl[NV], Fh[NV];
      limited_fluxes<DIR>(Wl, Wh, Fl, Fh, Pl, Ph, tc, tl, th);
      if constexpr (XM) {
        if (a.maxis == DIR) moving_fluxes(Pl, Ph, Fl, Fh);
      }
#pragma unroll
      for (int v = 0; v < NV; ++v) dF[v] = Fl[v] - Fh[v];
    }
  }

  // a3 + a4 for plane gz: the predictor increment dU = sum_d
  // (F_d(W_lo) - F_d(W_hi)) dt/(2 h_d) of every needed cell, and its predicted face
  // states.  PRED_ALL: tile plus halo, every face state of the plane;
  // PRED_ZHI / PRED_ZLO: tile cells only, the upper / lower z state.
  template <int PM>
  __device__ void predictor(int gz) {
    if constexpr (S::TWO && EOS == 0 && !XM) {
      predictor_split();
      return;
    }
    const int t = threadIdx.x;
    if (t >= (PM == PRED_ALL ? NP : NI)) return;
    const int n0 = a.n[0], n1 = a.n[1];
    int px, py;
    item_cell(t, px, py);
    const int gi = x0 - 1 + px;
    const int gj = DIM >= 2 ? y0 - 1 + py : 0;
    if (gi > n0 || (DIM >= 2 && gj > n1)) return;
    const int slot = wslot(gz);
    const int ex = px + 1, ey = py + (HY - QY);
    const bool trow = DIM < 2 || (py >= 1 && py <= TY);  // a tile row
    const bool tcol = px >= 1 && px <= TX;               // a tile column
    const bool rreal = DIM < 2 || gj < n1;               // a domain row
    const bool creal = gi < n0;                          // a domain column
    const int row = py - QY, col = px - 1;
    // face-state slots written by this cell
    const bool xlo = PM == PRED_ALL && px >= 1 && trow && rreal;
    const bool xhi = PM == PRED_ALL && px <= TX && trow && rreal && creal;
    const bool ylo = DIM >= 2 && PM == PRED_ALL && py >= 1 && tcol && creal;
    const bool yhi = DIM >= 2 && PM == PRED_ALL && py <= TY && tcol && creal && rreal;
    const bool zin = DIM == 3 && tcol && trow && creal && rreal;
    const bool zlo = zin && PM != PRED_ZHI;
    const bool zhi = zin && PM != PRED_ZLO;
    const int ixlo = row * (TX + 1) + px - 1, ixhi = ixlo + 1;
    const int iylo = (py - 1) * TX + col, iyhi = iylo + TX;
    const int iz = row * TX + col;
    T* zhp = ZL + (gz & 1) * NV * NFZ;

    T Wc[NV], dU[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      Wc[v] = W(slot, v, ey, ex);
      dU[v] = T(0);
    }
    const T tcell = EOS == 1 ? WT[(slot * EY + ey) * EX + ex] : T(0);
    {
      T Wm[NV], Wp[NV], Wl[NV], Wh[NV], dF[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        Wm[v] = W(slot, v, ey, ex - 1);
        Wp[v] = W(slot, v, ey, ex + 1);
      }
      faces_of<0>(Wm, Wc, Wp, px, Wl, Wh);
      T Pl[NV], Ph[NV], tl = T(0), th = T(0);
      limited_diff<0>(Wl, Wh, dF, Pl, Ph, tcell, &tl, &th);
      if constexpr (EOS == 1) {
        if (xlo) XTR[ixlo] = tl;
        if (xhi) XTL[ixhi] = th;
      }
      const T ih = inv_h(0, px, py, gz) * half_dt;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        dU[v] += dF[v] * ih;
        if (xlo) XR[v * NFX + ixlo] = Pl[v];
        if (xhi) XL[v * NFX + ixhi] = Ph[v];
      }
    }
    if constexpr (DIM >= 2) {
      T Wm[NV], Wp[NV], Wl[NV], Wh[NV], dF[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        Wm[v] = W(slot, v, ey - 1, ex);
        Wp[v] = W(slot, v, ey + 1, ex);
      }
      faces_of<1>(Wm, Wc, Wp, py, Wl, Wh);
      T Pl[NV], Ph[NV], tl = T(0), th = T(0);
      limited_diff<1>(Wl, Wh, dF, Pl, Ph, tcell, &tl, &th);
      if constexpr (EOS == 1) {
        if (ylo) YTR[iylo] = tl;
        if (yhi) YTL[iyhi] = th;
      }
      const T ih = inv_h(1, px, py, gz) * half_dt;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        dU[v] += dF[v] * ih;
        if (ylo) YR[v * NFY + iylo] = Pl[v];
        if (yhi) YL[v * NFY + iyhi] = Ph[v];
      }
    }
    if constexpr (DIM == 3) {
      T Wm[NV], Wp[NV], Wl[NV], Wh[NV], dF[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        Wm[v] = W(wslot(gz - 1), v, ey, ex);
        Wp[v] = W(wslot(gz + 1), v, ey, ex);
      }
      faces_of<2>(Wm, Wc, Wp, gz, Wl, Wh);
      T Pl[NV], Ph[NV], tl = T(0), th = T(0);
      limited_diff<2>(Wl, Wh, dF, Pl, Ph, tcell, &tl, &th);
      if constexpr (EOS == 1) {
        if (zlo) ZTR[iz] = tl;
        if (zhi) ZTL[(gz & 1) * NFZ + iz] = th;
      }
      const T ih = inv_h(2, px, py, gz) * half_dt;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        dU[v] += dF[v] * ih;
        if (zlo) ZR[v * NFZ + iz] = Pl[v];
        if (zhi) zhp[v * NFZ + iz] = Ph[v];
      }
    }
    if constexpr (DIM < 3) {
      if (t < NI) {
#pragma unroll
        for (int v = 0; v < NV; ++v) dUo[v] = dU[v];
      }
    }
    // A face is counted (fallbacks, Newton iterations) by the one CTA that
    // owns it: its tile's faces except the upper edge, unless that is the
    // domain's last face.
    T* ztl = ZTL + (gz & 1) * NFZ;
    if (xlo) finish_state(XR + ixlo, NFX, Wc, dU, px - 1 < TX || gi == n0, XTR + ixlo);
    if (xhi) finish_state(XL + ixhi, NFX, Wc, dU, px < TX || gi + 1 == n0, XTL + ixhi);
    if constexpr (DIM >= 2) {
      if (ylo) finish_state(YR + iylo, NFY, Wc, dU, py - 1 < TY || gj == n1, YTR + iylo);
      if (yhi) finish_state(YL + iyhi, NFY, Wc, dU, py < TY || gj + 1 == n1, YTL + iyhi);
    }
    if constexpr (DIM == 3) {
      if (zlo) finish_state(ZR + iz, NFZ, Wc, dU, gz < z1 || gz == n2, ZTR + iz);
      if (zhi) finish_state(zhp + iz, NFZ, Wc, dU, gz + 1 < z1 || gz + 1 == n2, ztl + iz);
    }
  }

  // predictor for the small FP64 tiles, of two threads per cell: in 2D one
  // takes axis 0 and the other axis 1, and they exchange the flux differences;
  // in 1D both evaluate these, and one finishes the lower and the other the
  // upper state.  A warp's FP64 operation occupies its scheduler for 64 cycles
  // whatever its active lanes and however few other warps there are, so the
  // longest chain of one warp is what counts: Sod 1000 FP64 9.6 -> 8.8 us per
  // step, 64 x 128 FP64 HLLC 42.7 -> 41.7 per cfl_dt + step.
  __device__ void predictor_split() {
    const int part = threadIdx.x / S::NPT, t = threadIdx.x % S::NPT;  // (part: the same in a warp)
    const int n0 = a.n[0], n1 = a.n[1];
    T* const mine = GXs + S::geo_elems + part * (NV * S::NPT) + t;
    const T* const parts = GXs + S::geo_elems + t;
    int px = 0, py = 0;
    if (t < NP) item_cell(t, px, py);
    const int gi = x0 - 1 + px, gj = DIM >= 2 ? y0 - 1 + py : 0;
    const bool cell = t < NP && gi <= n0 && (DIM < 2 || gj <= n1);
    const int ex = px + 1, ey = py + (HY - QY), row = py - QY, col = px - 1;
    const bool rreal = DIM < 2 || gj < n1, creal = gi < n0;
    const bool trow = DIM < 2 || (py >= 1 && py <= TY), tcol = px >= 1 && px <= TX;
    T Wc[NV], Wl[NV], Wh[NV], dF[NV], Pl[NV], Ph[NV];
    if (cell) {
#pragma unroll
      for (int v = 0; v < NV; ++v) Wc[v] = W(0, v, ey, ex);
      T Wm[NV], Wp[NV];
      if constexpr (DIM == 1) {
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          Wm[v] = W(0, v, ey, ex - 1);
          Wp[v] = W(0, v, ey, ex + 1);
        }
        faces_of<0>(Wm, Wc, Wp, px, Wl, Wh);
        flux_diff<DIM, NSX, 0>(Wl, Wh, a.gas.igm1, dF, Pl, Ph);
      } else {
        const int dx = part == 0 ? 1 : 0, dy = 1 - dx;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          Wm[v] = W(0, v, ey - dy, ex - dx);
          Wp[v] = W(0, v, ey + dy, ex + dx);
        }
        if (part == 0) {
          faces_of<0>(Wm, Wc, Wp, px, Wl, Wh);
          flux_diff<DIM, NSX, 0>(Wl, Wh, a.gas.igm1, dF, Pl, Ph);
        } else {
          faces_of<1>(Wm, Wc, Wp, py, Wl, Wh);
          flux_diff<DIM, NSX, (DIM >= 2 ? 1 : 0)>(Wl, Wh, a.gas.igm1, dF, Pl, Ph);
        }
#pragma unroll
        for (int v = 0; v < NV; ++v) mine[v * S::NPT] = dF[v];
      }
    }
    if constexpr (DIM >= 2) __syncthreads();
    if (!cell) return;
    T dU[NV];
    const T ix = inv_h(0, px, py, 0) * half_dt;
    if constexpr (DIM == 1) {
#pragma unroll
      for (int v = 0; v < NV; ++v) dU[v] = dF[v] * ix;
    } else {
      const T iy = inv_h(1, px, py, 0) * half_dt;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        dU[v] = fma(parts[(NV + v) * S::NPT], iy, __dmul_rn(parts[v * S::NPT], ix));
      }
    }
    if (threadIdx.x < NI) {
#pragma unroll
      for (int v = 0; v < NV; ++v) dUo[v] = dU[v];
    }
    auto finish = [&](bool needed, T* p, int st, const T* P, bool owned, T* tp) {
      if (!needed) return;
#pragma unroll
      for (int v = 0; v < NV; ++v) p[v * st] = P[v];
      finish_state(p, st, Wc, dU, owned, tp);
    };
    // (faces as in predictor: needed, slot, counted by this CTA)
    const int ixlo = row * (TX + 1) + px - 1, iylo = (py - 1) * TX + col, iyhi = iylo + TX;
    const bool xlo = px >= 1 && trow && rreal, xhi = px <= TX && trow && rreal && creal;
    const bool lo_owned = px - 1 < TX || gi == n0, hi_owned = px < TX || gi + 1 == n0;
    if constexpr (DIM == 1) {
      if (part == 0) finish(xlo, XR + ixlo, NFX, Pl, lo_owned, XTR + ixlo);
      else finish(xhi, XL + ixlo + 1, NFX, Ph, hi_owned, XTL + ixlo + 1);
    } else if (part == 0) {
      finish(xlo, XR + ixlo, NFX, Pl, lo_owned, XTR + ixlo);
      finish(xhi, XL + ixlo + 1, NFX, Ph, hi_owned, XTL + ixlo + 1);
    } else {
      finish(py >= 1 && tcol && creal, YR + iylo, NFY, Pl, py - 1 < TY || gj == n1, YTR + iylo);
      finish(py <= TY && tcol && creal && rreal, YL + iyhi, NFY, Ph, py < TY || gj + 1 == n1, YTL + iyhi);
    }
  }

  // Riemann flux of a face along DIR.  On the moving axis (reading R16) the
  // flux through the moving face, F - w U on the face path x/t = w, is the
  // fixed-face flux of the same two states seen from the frame that moves
  // with the face (normal velocities minus w; every solver here is Galilean
  // invariant), taken back to the lab frame: mass flux unchanged, normal
  // momentum flux + w F_rho, energy flux + w F_m + w^2/2 F_rho.
  // (One call site of the solver: on a fixed axis w = 0 and the shift is
  // exact, so the fixed grid computes what it computed without this.)
  template <int DIR>
  __device__ __forceinline__ void riemann(const T* WL, const T* WR, T* F, bool owned, T TL = T(0),
                                          T TR = T(0)) {
    if constexpr (!XM) {
      riemann_fixed<DIR>(WL, WR, F, owned, TL, TR);
      return;
    }
    const bool mv = a.maxis == DIR;
    const T w = mv ? a.wg : T(0);
    T wl[NV], wr[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      wl[v] = WL[v];
      wr[v] = WR[v];
    }
    wl[1 + DIR] -= w;
    wr[1 + DIR] -= w;
    riemann_fixed<DIR>(wl, wr, F, owned, TL, TR);
    if (mv) {
      F[1 + DIM] += w * F[1 + DIR] + T(0.5) * w * w * F[0];
      F[1 + DIR] += w * F[0];
    }
  }

  template <int DIR>
  __device__ __forceinline__ void riemann_fixed(const T* WL, const T* WR, T* F, bool owned, T TL = T(0),
                                                T TR = T(0)) {
    if constexpr (SND) {
      const T eL = WL[1 + DIM] * a.gas.igm1, eR = WR[1 + DIM] * a.gas.igm1;
      if constexpr (RS == RS_HLL) hll_flux<T, DIM, NSX, DIR>(WL, WR, eL, eR, TL, TR, F);
      else hllc_flux<T, DIM, NSX, DIR>(WL, WR, eL, eR, TL, TR, F);
    } else if constexpr (RS == RS_HLL) {
      riemann_hll<T, DIM, NSX, DIR>(WL, WR, F, gas(), TL, TR);
    } else if constexpr (RS == RS_HLLC) {
      riemann_hllc<T, DIM, NSX, DIR>(WL, WR, F, gas(), TL, TR);
    } else {
      int it = 0, kind = 0;
      const int st = riemann_exact<T, DIM, NSX, DIR>(WL, WR, F, a.gas, T(0), it, kind);
      if (owned) n_iters += it;
      if (st != ST_OK && err == 0) err = st;
    }
  }

  // a5: one Riemann solve per face, the flux written over the left state.
  // XY: the x and y faces of the current plane; Z: the z face below plane gz.
  template <bool XY, bool Z>
  __device__ void faces(int gz) {
    const int n0 = a.n[0], n1 = a.n[1];
    constexpr int NXY = XY ? NFX + NFY : 0;
    constexpr int NALL = NXY + (Z ? NFZ : 0);
    const T* zlp = ZL + ((gz - 1) & 1) * NV * NFZ;
    constexpr bool dual = DUAL, FT = EOS == 1 || SND;
    for (int idx = threadIdx.x; idx < NALL; idx += NT) {
      T WL[NV], WR[NV], F[NV];
      if (XY && idx < NFX) {
        const int f = idx % (TX + 1), row = idx / (TX + 1);
        if (x0 + f > n0 || (DIM >= 2 && y0 + row >= n1)) continue;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          WL[v] = XL[v * NFX + idx];
          WR[v] = XR[v * NFX + idx];
        }
        riemann<0>(WL, WR, F, f < TX || x0 + f == n0, FT ? XTL[idx] : T(0), FT ? XTR[idx] : T(0));
        if constexpr (dual) dual_terms(WL, WR, F, XQ, NFX, idx);
#pragma unroll
        for (int v = 0; v < NV; ++v) XL[v * NFX + idx] = F[v];
      } else if (XY && DIM >= 2 && idx < NXY) {
        const int k = idx - NFX;
        const int col = k % TX, fy = k / TX;
        if (x0 + col >= n0 || y0 + fy > n1) continue;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          WL[v] = YL[v * NFY + k];
          WR[v] = YR[v * NFY + k];
        }
        riemann<(DIM >= 2 ? 1 : 0)>(WL, WR, F, fy < TY || y0 + fy == n1, FT ? YTL[k] : T(0),
                                    FT ? YTR[k] : T(0));
        if constexpr (dual) dual_terms(WL, WR, F, YQ, NFY, k);
#pragma unroll
        for (int v = 0; v < NV; ++v) YL[v * NFY + k] = F[v];
      } else if (DIM == 3 && Z) {
        const int k = idx - NXY;
        const int i = k % TX, j = k / TX;
        if (x0 + i >= n0 || y0 + j >= n1) continue;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          WL[v] = zlp[v * NFZ + k];
          WR[v] = ZR[v * NFZ + k];
        }
        riemann<(DIM == 3 ? 2 : 0)>(WL, WR, F, gz < z1 || gz == n2,
                                    FT ? ZTL[((gz - 1) & 1) * NFZ + k] : T(0), FT ? ZTR[k] : T(0));
        if constexpr (dual) dual_terms(WL, WR, F, ZQ, NFZ, k);
#pragma unroll
        for (int v = 0; v < NV; ++v) ZR[v * NFZ + k] = F[v];
      }
    }
  }

  // a6 flux differences of the owned cell (i, j) from the x and y faces of
  // the current plane, plus (3D) the lower z face of plane gz; also the
  // spherical partial sums that use these fluxes.
  __device__ __forceinline__ void open_cell(int gz, int i, int j, int gi, int gj) {
    const int fx = j * (TX + 1) + i;
    const T Afl = gx(S::GX_AF, i + 1), Afh = gx(S::GX_AF, i + 2), ia = gx(S::GX_INVA, i + 1);
    constexpr bool dual = DUAL;
    const bool sph = a.spherical;  // (Cartesian area factors are 1)
    if constexpr (EOS == 1) topen = WT[(wslot(gz) * EY + j + HY) * EX + i + 2];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const T fl = XL[v * NFX + fx], fh = XL[v * NFX + fx + 1];
      acc[v] = (sph ? fl * Afl - fh * Afh : fl - fh) * ia;
    }
    if constexpr (dual) {
      aq1 = (XQ[fx] * Afl - XQ[fx + 1] * Afh) * ia;
      aq2 = (XQ[NFX + fx] * Afl - XQ[NFX + fx + 1] * Afh) * ia;
    }
    if constexpr (DIM >= 2) {
      const T Bfl = gy(S::GY_BF, j + 1), Bfh = gy(S::GY_BF, j + 2);
      const T cy = gx(S::GX_GA, i + 1) * gy(S::GY_INVB, j + 1);
      const int fy = j * TX + i;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const T fl = YL[v * NFY + fy], fh = YL[v * NFY + fy + TX];
        acc[v] += (sph ? fl * Bfl - fh * Bfh : fl - fh) * cy;
      }
      if constexpr (dual) {
        aq1 += (YQ[fy] * Bfl - YQ[fy + TX] * Bfh) * cy;
        aq2 += (YQ[NFY + fy] * Bfl - YQ[NFY + fy + TX] * Bfh) * cy;
      }
      if (a.spherical) {
        tth = T(0.5) * (YL[2 * NFY + fy] + YL[2 * NFY + fy + TX]);
        x2 = XL[2 * NFX + fx + 1] * Afh + XL[2 * NFX + fx] * Afl;
        if constexpr (DIM == 3) {
          const T frl = XL[3 * NFX + fx], frh = XL[3 * NFX + fx + 1];
          const T ftl = YL[3 * NFY + fy], fth = YL[3 * NFY + fy + TX];
          s3 = -gx(S::GX_QR, i + 1) * (frh * Afh + frl * Afl) -
               gx(S::GX_GA, i + 1) * gy(S::GY_QT, j + 1) * (fth * Bfh + ftl * Bfl);
        }
      }
    }
    if constexpr (DIM == 3) {
      const int iz = j * TX + i;
      const T cz = gx(S::GX_GA, i + 1) * gy(S::GY_ZC, j + 1) * a.geo.invc[gz];
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] += ZR[v * NFZ + iz] * cz;
      fzb3 = ZR[3 * NFZ + iz];
      if constexpr (dual) {
        aq1 += ZQ[iz] * cz;
        aq2 += ZQ[NFZ + iz] * cz;
      }
    }
  }

  // a6-a9: the new state of the owned cell (i, j) of plane gz from acc, the
  // sources, the validity checks and the signal speed.  fzt3 = the axis-2
  // momentum flux of the upper z face (3D).
  __device__ void close_cell(int gz, int i, int j, int gi, int gj, T fzt3) {
    const int n0 = a.n[0], n1 = a.n[1];
    const int nvact = NSX < 3 ? NV : 2 + DIM + a.ns;
    const long long c = ((long long)gz * n1 + gj) * n0 + gi;
    T Uo[NV], Un[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      if constexpr (MULTI) Uo[v] = Ucell[v];
      else Uo[v] = v < nvact ? Uin[(long long)v * a.ncell + c] : T(0);
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) Un[v] = Uo[v] + dt * acc[v];

    if (a.spherical) {
      // Geometric momentum sources, Eq. 13-16 (face-flux forms).  An absent
      // axis uses the pressure of the half-step cell state U + dU (or of U
      // if that state is not physical).
      T P = T(0);
      if constexpr (DIM < 3) {
        T Uh[NV], Wh[NV], Wo[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) Uh[v] = Uo[v] + dUo[v];
        to_prim<T, DIM, NSX>(Uh, Wh, gas());
        to_prim<T, DIM, NSX>(Uo, Wo, gas());
        P = (is_pos(Wh[0]) && is_pos(Wh[1 + DIM])) ? Wh[1 + DIM] : Wo[1 + DIM];
      }
      T Tth = P, Tph = P;
      if constexpr (DIM >= 2) Tth = tth;
      if constexpr (DIM == 3) Tph = T(0.5) * (fzb3 + fzt3);
      Un[1] += dt * T(0.5) * (Tth + Tph) * gx(S::GX_GR, i + 1);
      if constexpr (DIM >= 2)
        Un[2] += dt * (-gx(S::GX_QR, i + 1) * x2 + Tph * gx(S::GX_GA, i + 1) * gy(S::GY_GT, j + 1));
      if constexpr (DIM == 3) Un[3] += dt * s3;
    }
    if (a.gravity != GRAV_NONE) {
      T g[3] = {T(0), T(0), T(0)};
      if (a.gravity == GRAV_UNIFORM) {
#pragma unroll
        for (int d = 0; d < DIM; ++d) g[d] = a.g0[d];
      } else {
        g[0] = gx(S::GX_G, i + 1);  // point mass or monopole
      }
      T work = T(0);
#pragma unroll
      for (int d = 0; d < DIM; ++d) {
        Un[1 + d] += dt * Uo[0] * g[d];
        work += Uo[1 + d] * g[d];
      }
      Un[1 + DIM] += dt * work;
    }
    T dheat = T(0);
    if (a.heating == HEAT_CONST) {
      dheat = dt * a.heat_q;
      Un[1 + DIM] += dheat;
    } else if (a.heating == HEAT_NI56) {
      T rf = T(0);
#pragma unroll
      for (int s = 0; s < NSX; ++s)
        if (s == a.ni_index) rf = Uo[2 + DIM + s];
      dheat = dt * hfac * rf;
      Un[1 + DIM] += dheat;
    }

    // Dual energy (Sect. 2.5): where e is small against the kinetic energy
    // of the t^n state, blend the internal-energy change of the total-energy
    // update with that of de/dt + div(u e) + P div(u) = 0 (plus heating).
    if constexpr (DUAL) {
      T ke0 = T(0), ke1 = T(0);
#pragma unroll
      for (int d = 0; d < DIM; ++d) {
        ke0 += T(0.5) * Uo[1 + d] * Uo[1 + d] / Uo[0];
        ke1 += T(0.5) * Un[1 + d] * Un[1 + d] / Un[0];
      }
      const T e0 = Uo[1 + DIM] - ke0;
      const T crit = a.eps_dual * ke0;
      const T alpha = e0 >= crit ? T(1) : (e0 > T(0.1) * crit ? (e0 / crit) * (e0 / crit) : T(0));
      if (alpha < T(1)) {
        T Wo[NV];
        to_prim<T, DIM, NSX>(Uo, Wo, gas());
        const T d1 = (Un[1 + DIM] - ke1) - e0;
        const T d2 = dt * (aq1 + Wo[1 + DIM] * aq2) + dheat;
        Un[1 + DIM] = e0 + alpha * d1 + (T(1) - alpha) * d2 + ke1;
      }
    }

    // moving radial grid: the old cell's content spread over the new volume
    if (XM && a.vr) {
      const T q = a.vr[gi];
#pragma unroll
      for (int v = 0; v < NV; ++v) Un[v] *= q;
    }

    // the new cell's share of the conserved totals, in the owner's sum
    if (tsum) {
      const int o = j * TX + i;
      if constexpr (COLSUM) {
        // FP32 3D: per owner and variable a compensated FP32 sum (hi, lo) of
        // U dz along the owner's column, dz = dvol[2][gz] given as the FP32
        // pair hi + lo.  Each product is split exactly by an FMA, the sum
        // kept as an unevaluated pair (TwoSum, then renormalised), so each
        // term costs ~2^-48 of the sum; the column's sum is multiplied by
        // dvol[0] dvol[1] in FP64 at the end of the CTA.
        const float2 z = a.dvz32[gz];
        float2* ts = reinterpret_cast<float2*>(tsum);
#pragma unroll
        for (int v = 0; v < NV; ++v)
          if (v < nvact) add_column_sum(ts[v * NI + o], (float)Un[v], z);
      } else {
        // FP64 sums of U dV
        // (an absent axis has one factor: 1, or the angle it spans)
        const double dV = a.dvol[0][gi] * a.dvol[1][DIM >= 2 ? gj : 0] * a.dvol[2][DIM == 3 ? gz : 0];
#pragma unroll
        for (int v = 0; v < NV; ++v)
          if (v < nvact) tsum[v * NI + o] += (double)Un[v] * dV;
      }
    }

    // validity and the signal speed of the new state
    T Wn[NV], c2n;
    if constexpr (EOS == 1) {
      T tn;
      int k = 0;
      to_prim_ct<T, DIM, NSX>(Un, Wn, c2n, tn, a.grad, topen, &k);
      t_iters += k;
    } else {
      to_prim<T, DIM, NSX>(Un, Wn, a.gas);
      c2n = qdiv(a.gas.g * Wn[1 + DIM], Wn[0]);
    }
    bool finite = true;
#pragma unroll
    for (int v = 0; v < NV; ++v) finite = finite && isfinite(Un[v]);
    if (!finite) err = err ? err : ST_NONFINITE;
    else if (!is_pos(Wn[0]) || !is_pos(Wn[1 + DIM])) err = err ? err : ST_NEG;
    const T cs = dsqrt(c2n);
    T sp = T(0);
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
      T ih = inv_h(d, i + 1, j + 1, gz);
      T ud = Wn[1 + d];
      if constexpr (XM) {
        // a moving radial grid: the new state lives in the moved cell, whose
        // angular widths scale with its new radius; on the moving axis the
        // speed counts relative to the faces
        if (d >= 1 && a.ir_new) ih *= a.ir_new[gi] / a.geo.inv_r[gi + 2];
        if (d == a.maxis) ud -= a.wg;
      }
      sp += (fabs(ud) + cs) * ih;
    }
    smax = larger_speed(smax, sp);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      if (v < nvact) Uout[(long long)v * a.ncell + c] = Un[v];
      if constexpr (MULTI) Ucell[v] = Un[v];
    }
  }

  // The owner's work after the face solves of plane gz: in 3D, close the
  // cell of plane gz-1 with the flux of the z face between them and open
  // the cell of plane gz; in 1D/2D both in one go.
  __device__ void owner_step(int gz, bool close_prev, bool open_cur) {
    const int t = threadIdx.x;
    if (t >= NI) return;
    const int i = t % TX, j = t / TX;
    const int gi = x0 + i, gj = y0 + j;
    if (gi >= a.n[0] || (DIM >= 2 && gj >= a.n[1])) return;
    if constexpr (DIM == 3) {
      if (close_prev) {
        const T cz = gx(S::GX_GA, i + 1) * gy(S::GY_ZC, j + 1) * a.geo.invc[gz - 1];
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] -= ZR[v * NFZ + t] * cz;
        if constexpr (DUAL) {
          aq1 -= ZQ[t] * cz;
          aq2 -= ZQ[NFZ + t] * cz;
        }
        close_cell(gz - 1, i, j, gi, gj, ZR[3 * NFZ + t]);
      }
      if (open_cur) open_cell(gz, i, j, gi, gj);
    } else {
      open_cell(0, i, j, gi, gj);
      close_cell(0, i, j, gi, gj, T(0));
    }
  }
};

// Block-wide reductions into the control block, then the last-CTA commit and,
// where the host waits for this launch alone, the control block to the host.
// (The maximum of the non-negative speeds is taken on their bit patterns:
// integer compares, where an FP64 compare would occupy the FP64 pipe.)
template <int NT>
__device__ void finish_step(Ctrl* ctrl, double speed, int err, unsigned long long fb,
                            unsigned long long it, double dt, Ctrl* mirror) {
  __shared__ unsigned long long red_s[NT / 32];
  __shared__ int red_e[NT / 32];
  __shared__ unsigned long long red_f[NT / 32], red_i[NT / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  unsigned long long smax = dbits(speed);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long s2 = __shfl_xor_sync(0xffffffffu, smax, o);
    smax = smax > s2 ? smax : s2;
  }
  if (__any_sync(0xffffffffu, err != 0 || fb != 0 || it != 0)) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const int e2 = __shfl_xor_sync(0xffffffffu, err, o);
      err = err ? err : e2;
      fb += __shfl_xor_sync(0xffffffffu, fb, o);
      it += __shfl_xor_sync(0xffffffffu, it, o);
    }
  }
  if (lane == 0) {
    red_s[wid] = smax;
    red_e[wid] = err;
    red_f[wid] = fb;
    red_i[wid] = it;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < NT / 32; ++w) {
      smax = smax > red_s[w] ? smax : red_s[w];
      err = err ? err : red_e[w];
      fb += red_f[w];
      it += red_i[w];
    }
    const long long step = ((volatile Ctrl*)ctrl)->step;  // (constant until the commit below)
    if (smax) atomicMax(&ctrl->smax_next, smax);
    if (fb) atomicAdd(&ctrl->fallbacks, fb);
    if (it) atomicAdd(&ctrl->iters, it);
    if (err) {
      if (atomicCAS(&ctrl->status, 0, err) == 0) ctrl->err_step = step;
    }
    __threadfence();
    const unsigned int total = gridDim.x * gridDim.y * gridDim.z;
    const unsigned int ticket = atomicAdd(&ctrl->done, 1u);
    if (ticket == total - 1) {
      __threadfence();
      volatile Ctrl* vc = ctrl;
      if (vc->status == 0) {
        const unsigned long long nb = atomicExch(&ctrl->smax_next, 0ull);
        vc->smax_cur = __longlong_as_double((long long)nb);
        vc->t = vc->t + dt;
        vc->last_dt = dt;
        vc->step = step + 1;
        vc->cur = vc->cur ^ 1;
      }
      vc->done = 0;
      if (mirror) {
        // (a copy by the copy engine after the kernel takes 4 us longer)
        const volatile unsigned long long* const from = reinterpret_cast<const volatile unsigned long long*>(ctrl);
        volatile unsigned long long* const to = reinterpret_cast<volatile unsigned long long*>(mirror);
#pragma unroll
        for (int i = 0; i < (int)(sizeof(Ctrl) / 8); ++i) to[i] = from[i];
      }
      __threadfence();
    }
  }
}

// Time step of a launch: the host's dt, or the CFL step clipped to t_end (0
// or less: nothing to do).  One thread computes it for the CTA: an FP64
// operation costs a warp 19 cycles of an SM's FP64 pipe whatever its active
// lanes, so a division in every warp kept that pipe a quarter busy.
__device__ __forceinline__ double step_dt(const volatile Ctrl* vc, double dt_host, double cfl, double t_end) {
  if (dt_host > 0.0) return dt_host;
  double dt = cfl / vc->smax_cur;
  if (t_end > 0.0) dt = fmin(dt, t_end - vc->t);
  return dt;
}

// CTAs per SM that an instantiation's registers are sized for.  The FP32 3D
// forms of the radiation EoS and the exact solver wait on their Newton chains:
// two CTAs of 96 registers instead of one of 130-144 (wedge with radiation
// 512 x 96^2 8.22 -> 5.6 ms per 5 steps, exact 101 x 67 x 53 2.15 -> 1.49 ms
// per 10 steps, both with the chunks of plan_zchunk; the exact form spills 48-88
// bytes for it).
template <typename T, int DIM, int NSX, int RS, int MODE, bool SMALL>
__host__ __device__ constexpr int sweep_ctas() {
  if (SMALL) return 1;
  if (RS == RS_EXACT || (MODE & 1)) return DIM >= 2 && sizeof(T) == 4 ? 2 : 1;
  return SweepShape<T, DIM, NSX>::MB;
}

template <typename T, int DIM, int NSX, int RS, int MODE, bool SMALL>
__global__ void __launch_bounds__(SweepShape<T, DIM, NSX, SMALL>::NT,
                                  sweep_ctas<T, DIM, NSX, RS, MODE, SMALL>())
    sweep_kernel(const SweepArgs<T> args) {
  using S = SweepShape<T, DIM, NSX, SMALL>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // dt (and the heating factor) come from thread 0 and are read after the
  // barrier that ends the staging; a launch behind a failed one (dt 0)
  // writes nothing.
  __shared__ double s_dt;
  __shared__ T s_hfac;
  const volatile Ctrl* vc = args.ctrl;
  const int cur = vc->cur;
  if (threadIdx.x == 0) {
    s_dt = vc->status != 0 ? 0.0 : step_dt(vc, args.dt_host, args.cfl, args.t_end);
    if (args.heating == HEAT_NI56) {
      const double t = vc->t;
      s_hfac = (T)(args.ni_lambda * (args.ni_a * exp(-t / args.ni_tni) + args.ni_qco * exp(-t / args.ni_tco)));
    }
  }

  Sweep<T, DIM, NSX, RS, MODE, SMALL> sw(args, reinterpret_cast<T*>(smem_raw));
  if (sw.tsum)
    for (int q = threadIdx.x; q < S::NI * S::NV; q += S::NT) sw.tsum[q] = 0.0;  // (read after later barriers)
  sw.x0 = blockIdx.x * S::TX;
  sw.y0 = blockIdx.y * S::TY;
  sw.stage_geometry();  // (read after the first barrier below)
  sw.n2 = DIM == 3 ? args.n[2] : 1;
  sw.Uin = cur ? args.B : args.A;
  sw.Uout = cur ? args.Aw : args.B;
  auto set_dt = [&]() {
    sw.dt = (T)s_dt;
    sw.half_dt = T(0.5) * sw.dt;
    sw.hfac = args.heating == HEAT_NI56 ? s_hfac : T(0);
  };

  if constexpr (DIM == 3) {
    const int z0 = blockIdx.z * args.zchunk;
    const int z1 = min(z0 + args.zchunk, args.n[2]);
    sw.z1 = z1;
    for (int q = z0 - 2; q <= z0; ++q) sw.load_plane(q);
    __syncthreads();
    if (!(s_dt > 0.0)) return;
    set_dt();
    sw.template predictor<PRED_ZHI>(z0 - 1);
    __syncthreads();
    sw.load_plane(z0 + 1);
    // Plane k: its face states, then its x/y faces and the z face below it,
    // while plane k + 2 arrives; the owners close plane k-1 and open plane k.
    // k = z1 only supplies the z face above the chunk's last plane.
    for (int k = z0; k <= z1; ++k) {
      __syncthreads();
      if (k < z1) sw.template predictor<PRED_ALL>(k);
      else sw.template predictor<PRED_ZLO>(k);
      __syncthreads();
      if (k < z1) {
        sw.fetch_plane(k + 2);
        sw.template faces<true, true>(k);
        sw.finish_plane(k + 2);
      } else {
        sw.template faces<false, true>(k);
      }
      __syncthreads();
      sw.owner_step(k, k > z0, k < z1);
    }
  } else {
    sw.z1 = 1;
    sw.load_plane(0);
    __syncthreads();
    if (!(s_dt > 0.0)) return;
    set_dt();
    sw.template predictor<PRED_ALL>(0);
    __syncthreads();
    sw.template faces<true, false>(0);
    __syncthreads();
    sw.owner_step(0, false, true);
  }
  __syncthreads();
  if (sw.tsum) {
    if constexpr (decltype(sw)::COLSUM) {
      // each owner's compensated column sums, times its column's dvol[0]
      // dvol[1], in FP64 and in place
      for (int q = threadIdx.x; q < S::NI * S::NV; q += S::NT) {
        const int o = q % S::NI;
        const int gi = sw.x0 + o % S::TX, gj = sw.y0 + o / S::TX;
        const float2 c = reinterpret_cast<const float2*>(sw.tsum)[q];
        const double w = (gi < args.n[0] && gj < args.n[1]) ? args.dvol[0][gi] * args.dvol[1][gj] : 0.0;
        sw.tsum[q] = ((double)c.x + (double)c.y) * w;
      }
      __syncthreads();
    }
    reduce_totals<S::NV, S::NI, S::NT>(sw.tsum);
    const long long ncta = (long long)gridDim.x * gridDim.y * gridDim.z;
    const long long cta = blockIdx.x + gridDim.x * ((long long)blockIdx.y + (long long)gridDim.y * blockIdx.z);
    if (threadIdx.x < S::NV) args.tot_part[threadIdx.x * ncta + cta] = sw.tsum[threadIdx.x * S::NI];
  }
  finish_step<S::NT>(args.ctrl, (double)sw.smax, sw.err, sw.n_fallback,
                     (MODE & 1) ? (unsigned long long)sw.t_iters : sw.n_iters, s_dt, args.mirror);
}

// Several steps of a small 1D or 2D grid in one cooperative launch.  A step of
// such a grid is a chain of latencies (launch, control block, loads, atomics
// of the commit: ~9 of the 14.5 us of a 1000-cell FP64 step), so here the CTAs
// stay, the owners keep their cells in registers, and one word per CTA and
// step replaces the commit: a CTA publishes its speed maximum (release, after
// its stores), waits (bounded) for every CTA's and takes their maximum itself.
// A word's sign bit says which use of it is meant: the words of even and odd
// steps are apart, zeroed before the launch, and each use flips the sign, so
// none is overwritten before all have read it (8.8 us per step; a counter
// beside the words cost 0.2 more).  A step that fails in a CTA
// publishes NaN: every CTA ends with the state before it.  (A wait that
// expires ends its CTA alone, and the others may be a step further by the
// time they miss its word: the host takes the state for lost.)  The buffers
// alternate as between launches.
constexpr int ST_STEP_TIMEOUT = -6;  // HYDRO_ERR_TIMEOUT

template <typename T, int DIM, int NSX, int RS>
__global__ void __launch_bounds__(SweepShape<T, DIM, NSX, true>::NT, 1)
    sweep_steps_kernel(const SweepArgs<T> args, const StepsArgs sa) {
  using S = SweepShape<T, DIM, NSX, true>;
  constexpr int NT = S::NT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double s_dt;
  __shared__ T s_hfac;
  __shared__ unsigned long long s_speed[NT / 32];
  __shared__ int s_err[NT / 32], s_go;
  Ctrl* const ctrl = args.ctrl;
  const volatile Ctrl* vc = ctrl;
  const int cur0 = vc->cur;
  const long long step0 = vc->step;
  const unsigned int ctas = gridDim.x * gridDim.y, cta = blockIdx.x + gridDim.x * blockIdx.y;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;

  Sweep<T, DIM, NSX, RS, 0, true, true> sw(args, reinterpret_cast<T*>(smem_raw));
  sw.x0 = blockIdx.x * S::TX;
  sw.y0 = blockIdx.y * S::TY;
  sw.stage_geometry();  // (read after the first barrier below)
  sw.n2 = sw.z1 = 1;
  {
    const T* U = cur0 ? args.B : args.A;
    const int t = threadIdx.x, gi = sw.x0 + t % S::TX, gj = DIM >= 2 ? sw.y0 + t / S::TX : 0;
    const bool own = t < S::NI && gi < args.n[0] && (DIM < 2 || gj < args.n[1]);
    const int nvact = NSX < 3 ? S::NV : 2 + DIM + args.ns;
#pragma unroll
    for (int v = 0; v < S::NV; ++v)
      sw.Ucell[v] = own && v < nvact ? __ldcg(U + (long long)v * args.ncell + (long long)gj * args.n[0] + gi) : T(0);
  }
  // thread 0: the state's speed, its time, and the steps done
  double smax = vc->smax_cur, t = vc->t, last_dt = vc->last_dt;
  constexpr unsigned long long FAILED = 0x7ff8000000000000ull;
  const bool idle = vc->status != 0;  // (an earlier failure: written by this launch only after all have read it)
  int done = 0;
  for (;;) {
    if (threadIdx.x == 0) {
      double dt = 0.0;
      if (!idle && done < sa.nsteps) {
        dt = args.cfl / smax;
        if (args.t_end > 0.0) dt = fmin(dt, args.t_end - t);
      }
      s_dt = dt;
      if (args.heating == HEAT_NI56)
        s_hfac = (T)(args.ni_lambda * (args.ni_a * exp(-t / args.ni_tni) + args.ni_qco * exp(-t / args.ni_tco)));
    }
    const bool odd = ((cur0 ^ done) & 1) != 0;
    sw.Uin = odd ? args.B : args.A;
    sw.Uout = odd ? args.Aw : args.B;
    sw.load_plane(0);
    __syncthreads();
    const double dtd = s_dt;
    if (!(dtd > 0.0)) break;
    sw.dt = (T)dtd;
    sw.half_dt = T(0.5) * sw.dt;
    sw.hfac = args.heating == HEAT_NI56 ? s_hfac : T(0);
    sw.smax = T(0);
    sw.template predictor<PRED_ALL>(0);
    __syncthreads();
    sw.template faces<true, false>(0);
    __syncthreads();
    sw.owner_step(0, false, true);
    unsigned long long bits = dbits((double)sw.smax);
    int err = sw.err;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long b2 = __shfl_xor_sync(0xffffffffu, bits, o);
      bits = bits > b2 ? bits : b2;
    }
    if (__any_sync(0xffffffffu, err != 0)) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const int e2 = __shfl_xor_sync(0xffffffffu, err, o);
        err = err ? err : e2;
      }
    }
    if (lane == 0) {
      s_speed[wid] = bits;
      s_err[wid] = err;
    }
    __syncthreads();  // (also: every thread's stores of the step come before the release below)
    unsigned long long* const speed = sa.speed + (size_t)(done & 1) * ctas;
    const unsigned long long use = (done >> 1) & 1 ? 0ull : 1ull << 63;
    if (wid == 0) {
      if (lane == 0) {
        for (int w = 1; w < NT / 32; ++w) {
          bits = bits > s_speed[w] ? bits : s_speed[w];
          err = err ? err : s_err[w];
        }
        if (err) bits = FAILED;
        asm volatile("st.release.gpu.global.u64 [%0], %1;\n" ::"l"(speed + cta), "l"(bits | use) : "memory");
      }
      unsigned long long m = 0ull;
      bool late = false;
      for (unsigned int c = lane; c < ctas; c += 32) {
        unsigned long long b = ~use;
        for (int poll = 0; poll < sa.polls && ((b ^ use) >> 63) != 0ull; ++poll)
          asm volatile("ld.acquire.gpu.global.u64 %0, [%1];\n" : "=l"(b) : "l"(speed + c) : "memory");
        if (((b ^ use) >> 63) != 0ull) {  // the bounded wait expired
          b = FAILED;
          late = true;
        }
        b &= ~(1ull << 63);
        m = m > b ? m : b;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long b2 = __shfl_xor_sync(0xffffffffu, m, o);
        m = m > b2 ? m : b2;
      }
      // The status only now that every CTA has published: each has read it for
      // `idle` before that, and one that took this failure for an earlier one
      // would end without its word and leave the others to their whole wait.
      late = __any_sync(0xffffffffu, late);
      if (lane == 0 && (err != 0 || late)) {
        if (atomicCAS(&ctrl->status, 0, err ? err : ST_STEP_TIMEOUT) == 0) ctrl->err_step = step0 + done;
      }
      if (m < FAILED) smax = __longlong_as_double((long long)m);
      if (lane == 0) s_go = m < FAILED;
    }
    __syncthreads();
    if (!s_go) break;  // this step failed: the state before it stays
    t += dtd;
    last_dt = dtd;
    ++done;
  }
  // counters, and the commit of the steps done
  unsigned long long fb = sw.n_fallback, it = sw.n_iters;
  if (__any_sync(0xffffffffu, fb != 0 || it != 0)) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      fb += __shfl_xor_sync(0xffffffffu, fb, o);
      it += __shfl_xor_sync(0xffffffffu, it, o);
    }
    if (lane == 0) {
      if (fb) atomicAdd(&ctrl->fallbacks, fb);
      if (it) atomicAdd(&ctrl->iters, it);
    }
  }
  if (cta == 0 && threadIdx.x == 0 && done > 0) {
    volatile Ctrl* w = ctrl;
    w->smax_cur = smax;
    w->t = t;
    w->last_dt = last_dt;
    w->step = step0 + done;
    w->cur = cur0 ^ (done & 1);
  }
}

// Launch one instantiation and report the launch's shape.
template <typename T, int DIM, int NSX, int RS, int MODE, bool SMALL>
cudaError_t launch_tiled(const SweepArgs<T>& args, cudaStream_t s, LaunchShape* sh) {
  using S = SweepShape<T, DIM, NSX, SMALL>;
  SweepArgs<T> a = args;
  const void* fn = (const void*)sweep_kernel<T, DIM, NSX, RS, MODE, SMALL>;
  const size_t smem = a.tot_part ? S::tot_offset(MODE) + S::tot_bytes : S::smem_bytes_for(MODE);
  cudaError_t e = smem_attr_once(fn, (int)smem);
  if (e != cudaSuccess) return e;
  dim3 grid((a.n[0] + S::TX - 1) / S::TX, DIM >= 2 ? (a.n[1] + S::TY - 1) / S::TY : 1, 1);
  a.zchunk = 1;
  if (DIM == 3) {
    // (planned for the launch without totals, so that both take the same chunks)
    long long slots;
    if ((e = kernel_slots(fn, S::NT, S::smem_bytes_for(MODE), &slots)) != cudaSuccess) return e;
    a.zchunk = plan_zchunk((long long)grid.x * grid.y, a.n[2], slots, 1, 1.5, a.n[2]);
    grid.z = (a.n[2] + a.zchunk - 1) / a.zchunk;
  }
  sh->tx = S::TX;
  sh->ty = S::TY;
  sh->zchunk = a.zchunk;
  sh->threads = S::NT;
  sh->ctas = (long long)grid.x * grid.y * grid.z;
  sweep_kernel<T, DIM, NSX, RS, MODE, SMALL><<<grid, S::NT, smem, s>>>(a);
  return cudaGetLastError();
}

// Whether a 1D or 2D grid takes the small tiles: an SM's time goes with the
// threads of the CTAs it gets (FP64: with its warps, whatever their active
// lanes, from four warps on; fewer leave schedulers idle), so the shape whose
// busiest SM has fewer threads wins.  FP64 Sod, 1000 cells: 36 one-warp CTAs
// on 36 SMs instead of 4 of 8 warps on 4.
template <typename T, int DIM, int NSX>
bool small_tile(const int* n, int sms) {
  auto busiest = [&](long long tx, long long ty, long long threads) {
    const long long tiles = (n[0] + tx - 1) / tx * ((n[1] + ty - 1) / ty);
    return std::max(128ll, (tiles + sms - 1) / sms * threads);
  };
  using L = SweepShape<T, DIM, NSX, false>;
  using M = SweepShape<T, DIM, NSX, true>;
  return busiest(M::TX, M::TY, M::NPT) < busiest(L::TX, L::TY, L::NPT);
}

// nsteps steps in one launch (sa set but for its step count): whether the
// grid takes this path (small tiles, at most two CTAs per SM, all resident),
// reported in *taken; with nsteps 0 nothing is launched.
template <typename T, int DIM, int NSX, int RS>
cudaError_t launch_steps(const SweepArgs<T>& args, const StepsArgs& sa, cudaStream_t s, LaunchShape* sh, bool* taken) {
  using S = SweepShape<T, DIM, NSX, true>;
  *taken = false;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  dim3 grid((args.n[0] + S::TX - 1) / S::TX, DIM >= 2 ? (args.n[1] + S::TY - 1) / S::TY : 1);
  const long long ctas = (long long)grid.x * grid.y;
  if (!small_tile<T, DIM, NSX>(args.n, sms) || ctas > 2 * sms) return cudaSuccess;
  const void* fn = (const void*)sweep_steps_kernel<T, DIM, NSX, RS>;
  const size_t smem = S::smem_bytes_for(0);
  if ((e = smem_attr_once(fn, (int)smem)) != cudaSuccess) return e;
  long long slots;
  if ((e = kernel_slots(fn, S::NT, smem, &slots)) != cudaSuccess) return e;
  if (ctas > slots) return cudaSuccess;
  *taken = true;
  if (sa.nsteps < 1) return cudaSuccess;
  *sh = LaunchShape{S::TX, S::TY, 1, S::NT, ctas};
  SweepArgs<T> a = args;
  StepsArgs b = sa;
  void* params[] = {&a, &b};
  return cudaLaunchCooperativeKernel(fn, grid, dim3(S::NT), params, smem, s);
}

template <typename T, int DIM, int NSX, int RS, int MODE = 0>
cudaError_t launch_sweep(const SweepArgs<T>& a, cudaStream_t s, LaunchShape* sh) {
  if constexpr (DIM < 3 && MODE == 0) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (small_tile<T, DIM, NSX>(a.n, sms)) return launch_tiled<T, DIM, NSX, RS, MODE, true>(a, s, sh);
  }
  return launch_tiled<T, DIM, NSX, RS, MODE, false>(a, s, sh);
}

// Instantiate the dispatcher of one (precision, dimension) pair and MODE
// (ideal gas: 0, ideal gas + dual energy: 2).
#define HYDRO_SWEEP_DISPATCH_MODE(NAME, T, DIM, MODE)                                         \
  template <>                                                                                 \
  cudaError_t NAME<T, DIM>(const SweepArgs<T>& a, int nsx, int rs, cudaStream_t s,            \
                           LaunchShape* sh) {                                                 \
    switch (nsx * 4 + rs) {                                                                   \
      case 0: return launch_sweep<T, DIM, 0, RS_HLL, MODE>(a, s, sh);                  \
      case 1: return launch_sweep<T, DIM, 0, RS_HLLC, MODE>(a, s, sh);                 \
      case 2: return launch_sweep<T, DIM, 0, RS_EXACT, MODE>(a, s, sh);                \
      case 4: return launch_sweep<T, DIM, 1, RS_HLL, MODE>(a, s, sh);                  \
      case 5: return launch_sweep<T, DIM, 1, RS_HLLC, MODE>(a, s, sh);                 \
      case 6: return launch_sweep<T, DIM, 1, RS_EXACT, MODE>(a, s, sh);                \
      case 12: return launch_sweep<T, DIM, 3, RS_HLL, MODE>(a, s, sh);                 \
      case 13: return launch_sweep<T, DIM, 3, RS_HLLC, MODE>(a, s, sh);                \
      case 14: return launch_sweep<T, DIM, 3, RS_EXACT, MODE>(a, s, sh);               \
      default: return cudaErrorInvalidValue;                                                  \
    }                                                                                         \
  }
// Several steps in one launch: all solvers, or the exact one alone (FP32 2D).
#define HYDRO_STEPS_CASES(T, DIM, NSX, HYDRO_RS_CASES)                                        \
  switch (rs) {                                                                               \
    HYDRO_RS_CASES(T, DIM, NSX)                                                               \
    default: return cudaSuccess;                                                              \
  }
#define HYDRO_RS_ALL(T, DIM, NSX)                                                             \
  case RS_HLL: return launch_steps<T, DIM, NSX, RS_HLL>(a, sa, s, sh, taken);                 \
  case RS_HLLC: return launch_steps<T, DIM, NSX, RS_HLLC>(a, sa, s, sh, taken);               \
  case RS_EXACT: return launch_steps<T, DIM, NSX, RS_EXACT>(a, sa, s, sh, taken);
#define HYDRO_RS_EXACT_ONLY(T, DIM, NSX)                                                      \
  case RS_EXACT: return launch_steps<T, DIM, NSX, RS_EXACT>(a, sa, s, sh, taken);
#define HYDRO_STEPS_DISPATCH(T, DIM, HYDRO_RS_CASES)                                          \
  template <>                                                                                 \
  cudaError_t steps_dispatch<T, DIM>(const SweepArgs<T>& a, const StepsArgs& sa, int nsx,     \
                                     int rs, cudaStream_t s, LaunchShape* sh, bool* taken) {  \
    *taken = false;                                                                           \
    switch (nsx) {                                                                            \
      case 0: HYDRO_STEPS_CASES(T, DIM, 0, HYDRO_RS_CASES)                                    \
      case 1: HYDRO_STEPS_CASES(T, DIM, 1, HYDRO_RS_CASES)                                    \
      default: HYDRO_STEPS_CASES(T, DIM, 3, HYDRO_RS_CASES)                                   \
    }                                                                                         \
  }

// The exact solver alone (the FP32 2D forms, whose HLL and HLLC steps march).
#define HYDRO_SWEEP_DISPATCH_EXACT(T, DIM)                                                    \
  template <>                                                                                 \
  cudaError_t sweep_dispatch<T, DIM>(const SweepArgs<T>& a, int nsx, int rs, cudaStream_t s,  \
                                     LaunchShape* sh) {                                       \
    if (rs != RS_EXACT) return cudaErrorInvalidValue;                                         \
    switch (nsx) {                                                                            \
      case 0: return launch_sweep<T, DIM, 0, RS_EXACT, 0>(a, s, sh);                   \
      case 1: return launch_sweep<T, DIM, 1, RS_EXACT, 0>(a, s, sh);                   \
      default: return launch_sweep<T, DIM, 3, RS_EXACT, 0>(a, s, sh);                  \
    }                                                                                         \
  }
#define HYDRO_SWEEP_DISPATCH(T, DIM) HYDRO_SWEEP_DISPATCH_MODE(sweep_dispatch, T, DIM, 0)
#define HYDRO_SWEEP_DISPATCH_DUAL(T, DIM) HYDRO_SWEEP_DISPATCH_MODE(sweep_dispatch_dual, T, DIM, 2)
#define HYDRO_SWEEP_DISPATCH_XM(T, DIM) HYDRO_SWEEP_DISPATCH_MODE(sweep_dispatch_xm, T, DIM, 4)

// The gas + radiation dispatcher (HLL, HLLC) of one (precision, dimension)
// pair, without (MODE 1) and with (MODE 3) the dual-energy correction.
#define HYDRO_SWEEP_DISPATCH_RAD(T, DIM)                                                      \
  template <>                                                                                 \
  cudaError_t sweep_dispatch_rad<T, DIM>(const SweepArgs<T>& a, int nsx, int rs, int dual,    \
                                         cudaStream_t s, LaunchShape* sh) {                   \
    switch ((nsx * 4 + rs) * 2 + (dual ? 1 : 0)) {                                            \
      case 0: return launch_sweep<T, DIM, 0, RS_HLL, 1>(a, s, sh);                     \
      case 1: return launch_sweep<T, DIM, 0, RS_HLL, 3>(a, s, sh);                     \
      case 2: return launch_sweep<T, DIM, 0, RS_HLLC, 1>(a, s, sh);                    \
      case 3: return launch_sweep<T, DIM, 0, RS_HLLC, 3>(a, s, sh);                    \
      case 8: return launch_sweep<T, DIM, 1, RS_HLL, 1>(a, s, sh);                     \
      case 9: return launch_sweep<T, DIM, 1, RS_HLL, 3>(a, s, sh);                     \
      case 10: return launch_sweep<T, DIM, 1, RS_HLLC, 1>(a, s, sh);                   \
      case 11: return launch_sweep<T, DIM, 1, RS_HLLC, 3>(a, s, sh);                   \
      case 24: return launch_sweep<T, DIM, 3, RS_HLL, 1>(a, s, sh);                    \
      case 25: return launch_sweep<T, DIM, 3, RS_HLL, 3>(a, s, sh);                    \
      case 26: return launch_sweep<T, DIM, 3, RS_HLLC, 1>(a, s, sh);                   \
      case 27: return launch_sweep<T, DIM, 3, RS_HLLC, 3>(a, s, sh);                   \
      default: return cudaErrorInvalidValue;                                                  \
    }                                                                                         \
  }

}  // namespace hydro
