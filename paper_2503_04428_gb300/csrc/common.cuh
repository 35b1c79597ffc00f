// common.cuh -- argument blocks shared by the host runtime and the kernels.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>
#include <map>
#include <set>
#include <tuple>
#include <utility>

#include "physics.cuh"

namespace hydro {

// BC_EXCHANGED: a side whose ghosts are a neighbouring subdomain's cells,
// supplied by the caller (domain decomposition, Sect. 3.3.1).
enum { BC_PERIODIC = 0, BC_TRANSMISSIVE = 1, BC_REFLECTIVE = 2, BC_EXCHANGED = 3 };
enum { GRAV_NONE = 0, GRAV_UNIFORM = 1, GRAV_POINT = 2, GRAV_MONO = 3 };
enum { HEAT_NONE = 0, HEAT_CONST = 1, HEAT_NI56 = 2 };

// Device-resident control block of one handle.  Every step kernel reads it at
// start; the last CTA of a launch (ticket counter `done`) commits the step:
// it flips `cur`, advances t and step, and moves the next-state signal speed
// into smax_cur.  A failing launch never commits, so the input buffer of the
// failing step stays the current state.
struct Ctrl {
  double smax_cur;                  // max_cells sum_d (|u_d|+c)/h_d of the current state
  unsigned long long smax_next;     // same for the state being written (bits of a double >= 0)
  double t;                         // simulation time of the current state
  double last_dt;
  long long step;                   // committed steps
  long long err_step;               // step index of the first failure (-1 none)
  int status;                       // 0 or a hydro_status code
  int cur;                          // index of the buffer holding the current state
  unsigned int done;                // CTA tickets of the running launch
  unsigned int pad;
  unsigned long long iters;         // Newton iterations (exact solver)
  unsigned long long fallbacks;     // first-order face-state fallbacks
  unsigned long long mlp;           // faces whose guess came from the MLP
};

// Per-axis geometry, precomputed on the host in FP64 and stored as T.
// "ext" arrays are indexed by cell index + 2 for cells -2..n+1 (ghosts use
// the mirrored or wrapped interior widths); the others by interior cell
// (n entries) or interior face (n+1 entries).
template <typename T>
struct Geom {
  const T* sq[3];       // ext: (x_i - x_{i-1})/(x_{i+1} - x_i), the slopes' ratio of spacings
  const T* sf[3];       // ext: half coordinate width / (x_i - x_{i-1})
  const T* inv_w[3];    // ext: 1/coordinate width
  const T* inv_r;       // ext axis 0: 1/r_i (spherical)
  const T* inv_s;       // ext axis 1: 1/s_j, s_j = (sin th_- + sin th_+)/2 (spherical)
  const T* Af;          // axis-0 faces: r_f^2 (spherical) or 1
  const T* inva;        // axis 0: 1/a_i, a = (r+^3 - r-^3)/3 or dx
  const T* ga;          // axis 0: a2_i/a_i, a2 = (r+^2 - r-^2)/2 or dx
  const T* qr;          // axis 0: (r+ - r-)/((r+ + r-) a_i)
  const T* gr;          // axis 0: (Af_{i+1} - Af_i)/a_i
  const T* gpt;         // axis 0: point-mass acceleration -G Mc/r_i^2
  const T* Bf;          // axis-1 faces: sin th_f (spherical) or 1
  const T* invb;        // axis 1: 1/b_j, b = cos th_- - cos th_+ or dy
  const T* zc;          // axis 1: b3_j/b_j, b3 = dth or dy
  const T* gt;          // axis 1: (Bf_{j+1} - Bf_j)/b_j
  const T* qt;          // axis 1: (s+ - s-)/((s+ + s-) b_j)
  const T* invc;        // axis 2: 1/c_k, c = dphi or dz
};

template <typename T>
struct SweepArgs {
  const T* A;             // state buffer 0
  T* B;                   // state buffer 1 (in/out chosen by ctrl->cur)
  T* Aw;                  // writable alias of A
  Ctrl* mirror;           // host memory that receives the control block at the end of the launch, or null
  int n[3];
  long long ncell;
  int bc[3][2];
  int ns;                 // passive scalars in use (<= the kernel's NSX)
  int limiter;
  int spherical;
  int gravity;
  T g0[3];
  const T* gmono;         // monopole acceleration per radial cell (device)
  int heating;
  int ni_index;
  T heat_q;               // CONST: volumetric rate
  double ni_lambda, ni_a, ni_qco, ni_tni, ni_tco;  // Eq. 8 constants (CGS)
  Gas<T> gas;
  GasRad<T> grad;         // gas + radiation constants (kernels instantiated for Eq. 6-7)
  T eps_dual;             // dual-energy criterion epsilon (Sect. 2.5); 0 = off
  double dt_host;         // > 0: use this dt; otherwise CFL on the device
  double cfl;
  double t_end;           // > 0: clip dt so t does not pass t_end
  int zchunk;             // planes per CTA along axis 2 (3D general sweep)
  Ctrl* ctrl;
  Geom<T> geo;
  // domain decomposition: the axis whose sides may be BC_EXCHANGED (-1 none)
  // and their ghost layers [v][layer][cross section] (layer l = the ghost at
  // distance l+1 from the side; the cross section runs over the two other
  // axes, the lower one fastest)
  int xaxis;
  const T* halo[2];
  // moving grid (Sect. 3.1.1): the faces of axis maxis (-1 none) move with
  // velocity wg; vr (spherical radial motion, else null) = a_old/a_new per
  // radial cell, the volume ratio that spreads a cell's content over its
  // new volume
  int maxis;
  T wg;
  const T* vr;
  const T* ir_new;  // moving radial grid: 1/r of every radial cell after the step (its CFL widths)
  // conserved totals of the new state, accumulated in the step (a10): per
  // CTA and variable, sum over the CTA's cells of U dV in FP64, stored
  // [v][cta] (cta = blockIdx.x + gridDim.x (blockIdx.y + gridDim.y
  // blockIdx.z)); null: not accumulated
  double* tot_part;
  const double* dvol[3];  // dV of cell (i, j, k) = dvol[0][i] dvol[1][j] dvol[2][k] (FP64)
  const float2* dvz32;    // dvol[2][k] as an FP32 pair (hi, lo) with hi + lo = dvol[2][k] to ~2^-48
};

// The shape a step was launched with.
struct LaunchShape {
  int tx = 0, ty = 0;    // owned cells of a CTA's tile
  int zchunk = 0;        // planes of axis 2 per CTA (persistent CTAs: their share, rounded up)
  int threads = 0;
  long long ctas = 0;
};

// Planes per CTA of a march along axis 2 over `tiles` columns of n2 planes
// with room for `slots` CTAs at a time: the length (at most zmax) whose
// makespan is least, a CTA that takes z planes `per` at a time costing z/per
// steps (rounded up) plus `extra` for its partial planes and its start.  (Every
// length up to 256 is tried: where the general sweep of 32 x 32 x 2048 in FP32
// takes 18, multiples of 8 gave 24, 203 us per step against 157.)
// Measured: FP64 Sedov 128^3 (64 tiles, 152 slots, per 1, extra 1.5) 2.98 ms
// at 56 planes (128 CTAs of 56 and 64 of 16 on the free slots: 57.5), 3.13 at
// 19 = 3 waves of 20.5, 3.28 at 8 = 7 of 9.5, 3.39 at 64 = 1 of 65.5, 3.53 at
// 16 = 4 of 17.5.  The other sweeps (radiation, dual energy, moving grids, the
// exact solver; 64^3 to 128^3 and 96 x 40 x 200, both precisions) took 1.0 to 2.7
// times as long with chunks chosen by timed trials, in the code of those trials.
// A rule rather than a timed trial, so that equal handles take equal chunks and
// the sums of the totals, grouped by CTA, are the same bits.
struct ChunkPlan {
  int z = 0;         // planes per CTA
  double end = 0.0;  // its makespan
};
inline ChunkPlan plan_chunks(long long tiles, int n2, long long slots, int per, double extra, int zmax) {
  struct Plan {
    long long tiles = 0, slots = 0;
    int n2 = 0, per = 0;
    double extra = 0.0;
    int zmax = 0;
    ChunkPlan plan;
  };
  // (a step may ask for the march's plan and the general sweep's; a few handles in turn)
  static thread_local Plan kept[8];
  static thread_local unsigned next = 0;
  for (const Plan& p : kept)
    if (p.tiles == tiles && p.n2 == n2 && p.slots == slots && p.per == per && p.extra == extra && p.zmax == zmax)
      return p.plan;
  double least = 1e300;
  const int top = n2 < zmax ? n2 : zmax, stride = (top + 255) / 256;
  int best = top;
  for (int z = top; z >= 1; z -= z > 256 ? stride : 1) {
    const int chunks = (n2 + z - 1) / z, rest = n2 - (chunks - 1) * z;
    const double full = (z + per - 1) / per + extra, part = (rest + per - 1) / per + extra;
    // the full chunks run in waves; the last, shorter ones fill the slots that come free
    const long long nfull = tiles * (chunks - 1), waves = nfull / slots, busy = nfull % slots;
    double end = (waves + (busy ? 1 : 0)) * full;
    long long left = tiles;
    for (double t = waves * full; left > 0; t += part) {
      left -= slots - busy;
      if (t >= (waves + 1) * full - 1e-9) left -= busy;
      end = t + part > end ? t + part : end;
    }
    if (end < least * 0.999) {
      least = end;
      best = z;
    }
  }
  kept[next++ % 8] = {tiles, slots, n2, per, extra, zmax, {best, least}};
  return {best, least};
}
inline int plan_zchunk(long long tiles, int n2, long long slots, int per, double extra, int zmax) {
  return plan_chunks(tiles, n2, slots, per, extra, zmax).z;
}

template <typename T, int DIM>
cudaError_t sweep_dispatch(const SweepArgs<T>& a, int nsx, int rs, cudaStream_t s, LaunchShape* sh);
// Several steps in one launch (sweep_steps_kernel).
struct StepsArgs {
  unsigned long long* speed;  // 2 x CTAs words, zeroed before the launch: by step parity, the CTAs' speed maxima
  int nsteps;
  int polls;  // bound of the wait for another CTA's word
};
template <typename T, int DIM>
cudaError_t steps_dispatch(const SweepArgs<T>& a, const StepsArgs& sa, int nsx, int rs, cudaStream_t s,
                           LaunchShape* sh, bool* taken);
// The FP32 3D step of the plain ideal gas with HLL or HLLC (march3.cuh), and
// whether it is the faster form for a grid of these sizes (else the general sweep is).
bool march3_pays(const int* n, int nsx, int sms);
cudaError_t march3_dispatch(const SweepArgs<float>& a, int nsx, int rs, cudaStream_t s, LaunchShape* sh);
// The FP32 2D step of the plain ideal gas with HLL or HLLC (march2.cuh).
cudaError_t march2_dispatch(const SweepArgs<float>& a, int nsx, int rs, cudaStream_t s, LaunchShape* sh);
// The same with the dual-energy correction (Sect. 2.5).
template <typename T, int DIM>
cudaError_t sweep_dispatch_dual(const SweepArgs<T>& a, int nsx, int rs, cudaStream_t s, LaunchShape* sh);
// A slab of a decomposed grid or a moving grid (ideal gas, no dual energy).
template <typename T, int DIM>
cudaError_t sweep_dispatch_xm(const SweepArgs<T>& a, int nsx, int rs, cudaStream_t s, LaunchShape* sh);
// The gas + radiation EoS (HLL and HLLC only), with or without dual energy.
template <typename T, int DIM>
cudaError_t sweep_dispatch_rad(const SweepArgs<T>& a, int nsx, int rs, int dual, cudaStream_t s,
                               LaunchShape* sh);

// Raise the dynamic shared-memory limit of kernel `fn` to at least `bytes`
// on the current device.  The attribute is a property of the kernel on one
// device, so it is set per (device, kernel) pair when a launch needs more
// than was set before, under a lock (host threads may make their first calls
// at the same time).
inline cudaError_t smem_attr_once(const void* fn, int bytes) {
  static std::mutex mu;
  static std::map<std::pair<int, const void*>, int> done;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  auto it = done.find({dev, fn});
  if (it != done.end() && it->second >= bytes) return cudaSuccess;
  e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) done[{dev, fn}] = bytes;
  return e;
}

// CTAs of kernel `fn` that the current device holds at a time, looked up once
// per (device, kernel, shared memory).
inline cudaError_t kernel_slots(const void* fn, int threads, size_t smem, long long* slots) {
  static std::mutex mu;
  static std::map<std::tuple<int, const void*, size_t>, long long> known;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  auto it = known.find({dev, fn, smem});
  if (it == known.end()) {
    int sms = 0, occ = 0;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, threads, smem)) != cudaSuccess) return e;
    it = known.insert({{dev, fn, smem}, (long long)sms * (occ > 0 ? occ : 1)}).first;
  }
  *slots = it->second;
  return cudaSuccess;
}

// Bits of a non-negative double, for an ordered atomicMax.
__device__ __forceinline__ unsigned long long dbits(double x) {
  return (unsigned long long)__double_as_longlong(x);
}

}  // namespace hydro
