// mlp.cuh -- training of the star-pressure guess network on the GPU.
//
// Network: x (6) -> SiLU(W1 x + b1) (64) -> SiLU(W2 h1 + b2) (64) -> w3.h2 + b3,
// FP32 weights, loss = mean (y - t)^2 with t = ln(p_star / p_ref),
// p_ref = sqrt(P_L P_R).  Only faces that pass mlp_gate (the only faces where
// the network is used) are trained on.
// One CTA handles 64 samples: the three layers and their reverse-mode
// derivatives are small dense products on operands in shared memory; each CTA
// writes its partial gradient, and a second kernel sums the partials in a
// fixed order (deterministic), then Adam (Kingma & Ba 2015) updates the
// weights.
#pragma once
#include "common.cuh"

namespace hydro {

constexpr int MLP_SB = 64;  // samples per CTA

// Shared memory of the gradient kernel.  The three 64 x 64 x 64 products read
// both operands in rows of the summed index, four neighbours at a time, so the
// operands are kept in the orders they are read in; an array whose last
// reader is done takes its successor.  The transposed ones are written across
// their rows: there the four-element groups of row k are permuted by k / 4
// (swz), or those stores would all meet in one bank group.
struct __align__(16) MlpSmem {
  float w2[MLP_H * MLP_H];       // [o][i]
  float w2t_g1[MLP_H * MLP_H];   // [i][o] (swz), then G1 = dL/dz1 [sample][i]
  float h1[MLP_SB * MLP_H];      // [sample][i]
  float h1t_g2t[MLP_SB * MLP_H]; // [i][sample] (swz), then G2 = dL/dz2 [o][sample] (swz)
  float g2[MLP_SB * MLP_H];      // [sample][o]
  float h2[MLP_SB][MLP_H + 1];   // (read along both indices)
  float w1[MLP_H * MLP_IN], b1[MLP_H], b2[MLP_H], w3[MLP_H], b3;
  float x[MLP_SB][MLP_IN];
  float gy[MLP_SB];
  float loss[MLP_SB];
};

// Features, targets and the "network is used here" flag (Toro's rule picks
// the two-shock estimate) from face states (double) -- once per training set.
__global__ void mlp_features_kernel(const double* faces6, const double* log_pstar, long long n,
                                    Gas<double> gas, float* X, float* Y, unsigned char* use) {
  const double gamma = gas.g;
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double* f = faces6 + 6 * i;
  const double rref = sqrt(f[0] * f[3]);
  const double pref = sqrt(f[2] * f[5]);
  const double icref = 1.0 / sqrt(gamma * pref / rref);
  X[6 * i + 0] = (float)log(f[0] / rref);
  X[6 * i + 1] = (float)log(f[3] / rref);
  X[6 * i + 2] = (float)log(f[2] / pref);
  X[6 * i + 3] = (float)log(f[5] / pref);
  X[6 * i + 4] = (float)(f[1] * icref);
  X[6 * i + 5] = (float)(f[4] * icref);
  if (Y) Y[i] = (float)(log_pstar[i] - log(pref));
  if (use) {
    const double cL = sqrt(gamma * f[2] / f[0]), cR = sqrt(gamma * f[5] / f[3]);
    int kind;
    toro_guess<double>(f[0], f[1], f[2], cL, f[3], f[4], f[5], cR, gas, kind);
    use[i] = mlp_gate<double>(kind, f[2], f[5]);
  }
}

__device__ __forceinline__ int swz(int k, int group) { return k * 64 + 4 * (group ^ (k >> 2)); }

// acc[a][b] += sum_k A[k][4 r + a] B[k][4 c + b], k ascending, with fused
// multiply-adds: thread (r, c) of 16 x 16 holds a 4 x 4 tile of a 64 x 64
// product.  SA, SB: the operand is stored permuted (swz).
template <bool SA, bool SB>
__device__ __forceinline__ void tile_product(const float* __restrict__ A, const float* __restrict__ B, int r, int c,
                                             float acc[4][4]) {
#pragma unroll 8
  for (int k = 0; k < 64; ++k) {
    const float4 x = *reinterpret_cast<const float4*>(A + (SA ? swz(k, r) : k * 64 + 4 * r));
    const float4 y = *reinterpret_cast<const float4*>(B + (SB ? swz(k, c) : k * 64 + 4 * c));
    const float xa[4] = {x.x, x.y, x.z, x.w}, yb[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) acc[a][b] = fmaf(xa[a], yb[b], acc[a][b]);
  }
}
// A thread's 4 x 4 tile t[a][b] into M[4 r + a][4 c + b] and its transpose.
__device__ __forceinline__ void store_rows(float* M, int r, int c, const float t[4][4]) {
#pragma unroll
  for (int a = 0; a < 4; ++a)
    *reinterpret_cast<float4*>(M + (4 * r + a) * 64 + 4 * c) = make_float4(t[a][0], t[a][1], t[a][2], t[a][3]);
}
__device__ __forceinline__ void store_transposed(float* M, int r, int c, const float t[4][4]) {
#pragma unroll
  for (int b = 0; b < 4; ++b)
    *reinterpret_cast<float4*>(M + swz(4 * c + b, r)) = make_float4(t[0][b], t[1][b], t[2][b], t[3][b]);
}

// Forward + backward of 64 samples per CTA.  Samples are X[idx[first + s]]
// (idx may be null: identity); `count` samples in total, gradient scaled by
// inv_n.  Writes partial[blockIdx.x][p] and loss_partial[blockIdx.x].
//
// Bound by FP32 multiply-adds and the latency of its chain of phases: 0.8
// million multiply-adds in three products per CTA, held in 4 x 4 register
// tiles (two 16-byte shared loads per 16 of them; one scalar load or more per
// multiply-add, with bank conflicts, cost 113 us at 16384 samples; now 26).  Every sum
// runs over the same terms in the same order as a plain loop per output, so
// the tiles change no bit of it.
__global__ void __launch_bounds__(256, 2)
    mlp_grad_kernel(const float* __restrict__ W, const float* __restrict__ X,
                    const float* __restrict__ Y, const int* __restrict__ idx, long long first,
                    long long count, float inv_n, float* partial, double* loss_partial) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  MlpSmem& s = *reinterpret_cast<MlpSmem*>(smem_raw);
  const int tid = threadIdx.x;
  const int r = tid / 16, c = tid % 16;  // this thread's 4 x 4 tiles: samples (or units) 4r.., units 4c..
  float t[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) t[a][b] = W[MW2 + (4 * r + a) * MLP_H + 4 * c + b];
  store_rows(s.w2, r, c, t);
  store_transposed(s.w2t_g1, r, c, t);
  for (int p = tid; p < MLP_H * MLP_IN; p += 256) s.w1[p] = W[MW1 + p];
  if (tid < MLP_H) {
    s.b1[tid] = W[MB1 + tid];
    s.b2[tid] = W[MB2 + tid];
    s.w3[tid] = W[MW3 + tid];
    if (tid == 0) s.b3 = W[MB3];
  }
  const long long s0 = (long long)blockIdx.x * MLP_SB;
  for (int q = tid; q < MLP_SB * MLP_IN; q += 256) {
    const int sm = q / MLP_IN, i = q % MLP_IN;
    const long long g = s0 + sm;
    float v = 0.f;
    if (g < count) {
      const long long row = idx ? idx[first + g] : first + g;
      v = X[row * MLP_IN + i];
    }
    s.x[sm][i] = v;
  }
  __syncthreads();
  // layer 1 (z1 and, below, z2 stay with the thread that needs them back)
  float z1[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int sm = 4 * r + a, o = 4 * c + b;
      float z = s.b1[o];
#pragma unroll
      for (int i = 0; i < MLP_IN; ++i) z = fmaf(s.w1[o * MLP_IN + i], s.x[sm][i], z);
      z1[a][b] = z;
      t[a][b] = silu_f(z);
    }
  store_rows(s.h1, r, c, t);
  store_transposed(s.h1t_g2t, r, c, t);
  __syncthreads();
  // layer 2: z2[sm][o] = b2[o] + sum_i h1[sm][i] W2[o][i]
  float z2[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) z2[a][b] = s.b2[4 * c + b];
  tile_product<true, true>(s.h1t_g2t, s.w2t_g1, r, c, z2);
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      // h2 = silu(z2); the sigmoid is kept for its derivative
      const float d = 1.0f + expf(-z2[a][b]);
      s.h2[4 * r + a][4 * c + b] = z2[a][b] / d;
      t[a][b] = 1.0f / d;
    }
  __syncthreads();
  // output, loss and dL/dy
  if (tid < MLP_SB) {
    const long long g = s0 + tid;
    float y = s.b3;
#pragma unroll 16
    for (int i = 0; i < MLP_H; ++i) y = fmaf(s.w3[i], s.h2[tid][i], y);
    float e = 0.f;
    if (g < count) {
      const long long row = idx ? idx[first + g] : first + g;
      e = y - Y[row];
    }
    s.loss[tid] = e * e;
    s.gy[tid] = 2.0f * e * inv_n;
  }
  __syncthreads();
  float* P = partial + (long long)blockIdx.x * MLP_NPARAM;
  // G2 = dL/dz2, in both orders
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const float sg = t[a][b];
      t[a][b] = s.gy[4 * r + a] * s.w3[4 * c + b] * (sg * (1.0f + z2[a][b] * (1.0f - sg)));
    }
  store_rows(s.g2, r, c, t);
  store_transposed(s.h1t_g2t, r, c, t);
  // output layer gradients and the loss
  if (tid < MLP_H) {
    float a = 0.f;
#pragma unroll 16
    for (int sm = 0; sm < MLP_SB; ++sm) a = fmaf(s.gy[sm], s.h2[sm][tid], a);
    P[MW3 + tid] = a;
  } else if (tid < MLP_H + 32) {
    const int l = tid - MLP_H;
    double v = (double)s.loss[l] + (double)s.loss[l + 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (l == 0) loss_partial[blockIdx.x] = v;
  } else if (tid == MLP_H + 32) {
    float a = 0.f;
#pragma unroll 16
    for (int sm = 0; sm < MLP_SB; ++sm) a += s.gy[sm];
    P[MB3] = a;
  }
  __syncthreads();
  // dW2[o][i] = sum_sm G2[sm][o] h1[sm][i], db2 = sum G2 (thread (r, c): o = 4r.., i = 4c..)
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) t[a][b] = 0.f;
  tile_product<false, false>(s.g2, s.h1, r, c, t);
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) P[MW2 + (4 * r + a) * MLP_H + 4 * c + b] = t[a][b];
  if (tid < MLP_H) {
    float a = 0.f;
#pragma unroll 16
    for (int sm = 0; sm < MLP_SB; ++sm) a += s.g2[sm * MLP_H + tid];
    P[MB2 + tid] = a;
  }
  // G1[sm][i] = (sum_o G2[sm][o] W2[o][i]) silu'(z1)
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) t[a][b] = 0.f;
  tile_product<true, false>(s.h1t_g2t, s.w2, r, c, t);
#pragma unroll
  for (int a = 0; a < 4; ++a) {
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const float sg = 1.0f / (1.0f + expf(-z1[a][b]));
      t[a][b] = t[a][b] * (sg * (1.0f + z1[a][b] * (1.0f - sg)));
    }
  }
  store_rows(s.w2t_g1, r, c, t);
  __syncthreads();
  // dW1 = G1^T x, db1 = sum G1
  for (int q = tid; q < MLP_H * MLP_IN + MLP_H; q += 256) {
    float a = 0.f;
    if (q < MLP_H * MLP_IN) {
      const int i = q / MLP_H, o = q % MLP_H;
#pragma unroll 16
      for (int sm = 0; sm < MLP_SB; ++sm) a = fmaf(s.w2t_g1[sm * MLP_H + o], s.x[sm][i], a);
      P[MW1 + o * MLP_IN + i] = a;
    } else {
      const int o = q - MLP_H * MLP_IN;
#pragma unroll 16
      for (int sm = 0; sm < MLP_SB; ++sm) a += s.w2t_g1[sm * MLP_H + o];
      P[MB1 + o] = a;
    }
  }
}

// Sums of the per-CTA partials in a fixed order (FP64): 32 parameters per CTA
// of 8 warps, warp w summing the partials w, w + 8, ... (an SM adds FP64 at 19
// cycles per warp instruction, so the sums are spread over all SMs: one thread
// per parameter on 19 CTAs cost 45 us for 256 partials).  Returns the sum of
// parameter 32 blockIdx.x + lane to the threads of warp 0.
constexpr int MLP_RED = 8;
constexpr int MLP_RED_GRID = (MLP_NPARAM + 31) / 32;
__device__ __forceinline__ double mlp_partial_sum(const float* partial, int nblocks) {
  __shared__ double red[MLP_RED][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, p = blockIdx.x * 32 + lane;
  double a = 0.0;
  if (p < MLP_NPARAM)
#pragma unroll 8
    for (int b = w; b < nblocks; b += MLP_RED) a += (double)partial[(long long)b * MLP_NPARAM + p];
  red[w][lane] = a;
  __syncthreads();
  if (w == 0)
#pragma unroll
    for (int k = 1; k < MLP_RED; ++k) a += red[k][lane];
  return a;
}
// The sum of the loss partials, by one warp (returned to all of its lanes).
__device__ __forceinline__ double mlp_loss_sum(const double* loss_partial, int nblocks) {
  double l = 0.0;
  for (int b = threadIdx.x & 31; b < nblocks; b += 32) l += loss_partial[b];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
  return l;
}

// The gradient, and the loss sum times `scale` (added to *loss_out or, with
// `set`, stored there).
__global__ void __launch_bounds__(32 * MLP_RED)
    mlp_reduce_kernel(const float* partial, int nblocks, double* grad, const double* loss_partial, double* loss_out,
                      long n, int set) {
  const int p = blockIdx.x * 32 + threadIdx.x;
  const double g = mlp_partial_sum(partial, nblocks);
  if (threadIdx.x < 32 && p < MLP_NPARAM) grad[p] = g;
  if (blockIdx.x == 0 && threadIdx.x >= 32 && threadIdx.x < 64) {
    const double l = mlp_loss_sum(loss_partial, nblocks);
    if (threadIdx.x == 32) {
      if (set) *loss_out = l / (double)n;
      else *loss_out += l;
    }
  }
}

// The gradient sums followed by the Adam update of that parameter; the loss
// partials go to loss_acc.
__global__ void __launch_bounds__(32 * MLP_RED)
    mlp_reduce_adam_kernel(const float* partial, int nblocks, const double* loss_partial,
                           double* loss_acc, float* W, float* m, float* v, int step,
                           double lr, double b1, double b2, double eps) {
  const double g = mlp_partial_sum(partial, nblocks);
  if (blockIdx.x == 0 && threadIdx.x >= 32 && threadIdx.x < 64) {
    const double l = mlp_loss_sum(loss_partial, nblocks);
    if (threadIdx.x == 32) *loss_acc += l;
  }
  const int p = blockIdx.x * 32 + threadIdx.x;
  if (threadIdx.x >= 32 || p >= MLP_NPARAM) return;
  const double c1 = 1.0 - pow(b1, (double)step), c2 = 1.0 - pow(b2, (double)step);
  const double mm = b1 * m[p] + (1.0 - b1) * g;
  const double vv = b2 * v[p] + (1.0 - b2) * g * g;
  m[p] = (float)mm;
  v[p] = (float)vv;
  W[p] = (float)(W[p] - lr * (mm / c1) / (sqrt(vv / c2) + eps));
}

}  // namespace hydro
