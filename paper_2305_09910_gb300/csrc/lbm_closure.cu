// lbm_closure.cu -- learned closure: training samples from a fine lattice (box filter of
// width 2), the 7 -> 32 -> 32 -> 1 GELU network's forward and backward passes, the
// eddy-viscosity loss, and the Adam optimiser, all as CUDA kernels behind C entry points.
//
// The network gives the Smagorinsky coefficient of each cell, C_s^2 = softplus(y) C_s0^2 /
// ln 2, from the cell's non-equilibrium stress and density; its inference runs inside the
// collide kernel (lbm_kernels.cuh, mlp_cs2).  Training pairs come from the solver itself:
// a fine lattice is filtered onto the coarse grid (half resolution), and the target is the
// eddy viscosity that best reproduces the filtered subgrid stress (least-squares
// projection on the coarse strain rate).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <mutex>

#include "../../include/lbm.h"
#include "lbm_launch.cuh"

void lbm_internal_set_error(const char* msg);

namespace lbm {

// ---- training samples -------------------------------------------------------------------
struct SampleArgs {
  float* x;        // nc * 7
  float* target;   // nc
  float* smag;     // nc, |S_c|
  float* weight;   // nc, |S_c|^2
  int ncx, ncy, ncz;
  float tau0_c, cs0sq, scale_pi, scale_rho;
  int smag_fine;   // the fine lattice uses the Smagorinsky closure
};

// W fine cells at x, their populations and classes.  Natural layout (PAR 0): the cells (x, x + 1), one
// access per direction for both (x even and rows of a multiple of 32 elements: aligned),
// issued before the classes arrive; a cell that is not fluid is dropped by its class.  Other
// layouts: one cell, in FP32 the gather of a cell off the faces beside its class load (half
// storage spills with that: samples of D3Q27 20 % slower, the filter of D3Q19 11 %).
// Bound by memory latency: before, each cell's class load stood before its populations, one per
// access.  Samples and filter of a 384x192x192 lattice (us): D3Q19 FP32 natural 227 + 183 -> 206 + 172,
// gathered 258 + 203 -> 232 + 185; FP16 181 + 129 -> 162 + 102 and 225 + 149 -> 219 + 146; D3Q27 FP32
// natural 312 + 264 -> 273 + 236.  512x256x256 D3Q19 FP32, both calls: 885 -> 814.
// FIRST (the filter): a skipped cell returns before its load; the samples load it as zeros.
template <int Q, class S, int PAR, bool FIRST>
struct FineCells {
  static constexpr int W = PAR == 0 ? 2 : 1;
  float f[W][Q];
  int cls[W];

  __device__ __forceinline__ void load(const KParams& p, int cell) {
    if constexpr (PAR == 0) {
#pragma unroll
      for (int i = 0; i < Q; i++) {
        const S* a = plane_ptr<S>(p, i) + cell;
        float2 v = make_float2(0.f, 0.f);
        if (chk(p, a, 2 * (int)sizeof(S), CHK_POP)) {
          if constexpr (sizeof(S) == 4) v = *reinterpret_cast<const float2*>(a);
          else v = unpack2<S>(*reinterpret_cast<const uint32_t*>(a));
        }
        f[0][i] = v.x;
        f[W - 1][i] = v.y;
      }
#pragma unroll
      for (int k = 0; k < W; k++) cls[k] = cls_at(p, cell + k);
    }
  }

  // Cell k of the W; false if it is not fluid.  (x, y, z), c: the first.
  __device__ __forceinline__ bool cell(const KParams& p, int k, int x, int y, int z, int c) {
    if constexpr (PAR != 0) {
      const bool early = sizeof(S) == 4 && off_faces(p, x, y, z);
      if (early) gather_interior<Q, S, PAR>(p, c, f[0]);
      cls[k] = cls_at(p, c);
      if (FIRST && cls[k] == CLS_SKIP) return false;
      unsigned outmask;
      if (!early || cls[k] != CLS_INTERIOR) load_state<Q, S, PAR, sizeof(S) == 4>(p, x, y, z, c, cls[k], f[0], outmask);
    }
    return cls[k] != CLS_SKIP;
  }
};

template <int Q, class S, int PAR>
__global__ void __launch_bounds__(128) k_closure_samples(const __grid_constant__ KParams p, SampleArgs a) {
  constexpr int W = FineCells<Q, S, PAR, false>::W;
  const long long nc = (long long)a.ncx * a.ncy * a.ncz;
  const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nc) return;
  const int X = (int)(k % a.ncx), Y = (int)((k / a.ncx) % a.ncy), Z = (int)(k / ((long long)a.ncx * a.ncy));
  __shared__ float sh[8][4][128];  // rho, u of the thread's fine cells; as a local array 842 us (see FineCells)
  const int t = threadIdx.x;
  float rho_s = 0.f, m_s[3] = {0.f, 0.f, 0.f}, S_s[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  float nS_s[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  bool all_fluid = true;
#pragma unroll 1
  for (int n0 = 0; n0 < 8; n0 += W) {
    const int x = 2 * X + (n0 & 1), y = 2 * Y + ((n0 >> 1) & 1), z = 2 * Z + (n0 >> 2), c0 = cidx(p, x, y, z);
    FineCells<Q, S, PAR, false> fine;
    fine.load(p, c0);
#pragma unroll
    for (int k = 0; k < W; k++) {
      const int n = n0 + k;
      if (!fine.cell(p, k, x, y, z, c0)) {
        all_fluid = false;
        sh[n][0][t] = sh[n][1][t] = sh[n][2][t] = sh[n][3][t] = 0.f;
        continue;
      }
      const float(&f)[Q] = fine.f[k];
      const Mom<Q> m = moments<Q>(p, f);
      // non-equilibrium stress (shifted form), as in the collision
      float sxx = 0.f, syy = 0.f, szz = 0.f, sxy = 0.f, sxz = 0.f, syz = 0.f;
#pragma unroll
      for (int i = 0; i < Q; i++) {
        if (cx(i)) sxx += f[i];
        if (cy(i)) syy += f[i];
        if (cz(i)) szz += f[i];
        if (cx(i) * cy(i)) sxy += cx(i) * cy(i) > 0 ? f[i] : -f[i];
        if (cx(i) * cz(i)) sxz += cx(i) * cz(i) > 0 ? f[i] : -f[i];
        if (cy(i) * cz(i)) syz += cy(i) * cz(i) > 0 ? f[i] : -f[i];
      }
      const float d3 = m.drho * (1.f / 3.f);
      const float pi[6] = {sxx - d3 - m.jx * m.ux, syy - d3 - m.jy * m.uy, szz - d3 - m.jz * m.uz,
                           sxy - m.jx * m.uy, sxz - m.jx * m.uz, syz - m.jy * m.uz};
      const float qn = pi[0] * pi[0] + pi[1] * pi[1] + pi[2] * pi[2] +
                       2.f * (pi[3] * pi[3] + pi[4] * pi[4] + pi[5] * pi[5]);
      float tau = p.tau0;
      if (a.smag_fine)
        tau = 0.5f * (p.tau0 + sqrtf(p.tau0 * p.tau0 + 25.455844122715711f * p.cs2 * sqrtf(qn) / m.rho));
      const float nut = (tau - p.tau0) * (1.f / 3.f);
      const float sfac = -3.f / (2.f * m.rho * tau);
      sh[n][0][t] = m.rho;
      sh[n][1][t] = m.ux;
      sh[n][2][t] = m.uy;
      sh[n][3][t] = m.uz;
      rho_s += m.rho;
      m_s[0] += m.jx;
      m_s[1] += m.jy;
      m_s[2] += m.jz;
#pragma unroll
      for (int j = 0; j < 6; j++) {
        S_s[j] += sfac * pi[j];
        nS_s[j] += nut * sfac * pi[j];
      }
    }
  }
  float* xo = a.x + k * 7;
  if (!all_fluid) {
    for (int j = 0; j < 7; j++) xo[j] = 0.f;
    a.target[k] = 0.f;
    a.smag[k] = 0.f;
    a.weight[k] = 0.f;
    return;
  }
  const float rb = rho_s * 0.125f;
  const float ub[3] = {m_s[0] / rho_s, m_s[1] / rho_s, m_s[2] / rho_s};
  // Favre variance from deviations (no cancellation): sum rho (u - u_bar)(u - u_bar) / sum rho
  float R[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int n = 0; n < 8; n++) {
    const float rk = sh[n][0][t], dx = sh[n][1][t] - ub[0], dy = sh[n][2][t] - ub[1], dz = sh[n][3][t] - ub[2];
    R[0] += rk * dx * dx;
    R[1] += rk * dy * dy;
    R[2] += rk * dz * dz;
    R[3] += rk * dx * dy;
    R[4] += rk * dx * dz;
    R[5] += rk * dy * dz;
  }
  float tsg[6], Sc[6];
#pragma unroll
  for (int j = 0; j < 6; j++) {
    tsg[j] = R[j] / rho_s - 2.f * nS_s[j] * 0.125f;
    Sc[j] = 2.f * S_s[j] * 0.125f;
  }
  const float tr = (tsg[0] + tsg[1] + tsg[2]) * (1.f / 3.f);
  float num = 0.f, den = 0.f;
#pragma unroll
  for (int j = 0; j < 6; j++) {
    const float mult = j < 3 ? 1.f : 2.f;
    const float td = j < 3 ? tsg[j] - tr : tsg[j];
    num += mult * td * Sc[j];
    den += mult * Sc[j] * Sc[j];
  }
  const float Smag = sqrtf(2.f * den);
  float nu = Smag > 1e-10f ? -num / (2.f * den) : 0.f;
  nu = fmaxf(nu, 0.f);
  const float tauc = a.tau0_c + 3.f * a.cs0sq * Smag;
#pragma unroll
  for (int j = 0; j < 6; j++)
    xo[j] = fminf(fmaxf(a.scale_pi * (-(2.f * rb / 3.f) * tauc * Sc[j]), -MLP_XCLAMP), MLP_XCLAMP);
  xo[6] = fminf(fmaxf(a.scale_rho * (rb - 1.f), -MLP_XCLAMP), MLP_XCLAMP);
  a.target[k] = nu;
  a.smag[k] = Smag;
  a.weight[k] = Smag * Smag;
}

// Box filter of width 2: mean density and Favre velocity of each coarse cell's 8 fine cells.
template <int Q, class S, int PAR>
__global__ void __launch_bounds__(128) k_filter2(const __grid_constant__ KParams p, int ncx, int ncy, int ncz,
                                                 float* rho_bar, float* u_bar) {
  constexpr int W = FineCells<Q, S, PAR, true>::W;
  const long long nc = (long long)ncx * ncy * ncz;
  const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nc) return;
  const int X = (int)(k % ncx), Y = (int)((k / ncx) % ncy), Z = (int)(k / ((long long)ncx * ncy));
  float rs = 0.f, ms[3] = {0.f, 0.f, 0.f};
#pragma unroll 1
  for (int n0 = 0; n0 < 8; n0 += W) {
    const int x = 2 * X + (n0 & 1), y = 2 * Y + ((n0 >> 1) & 1), z = 2 * Z + (n0 >> 2), c0 = cidx(p, x, y, z);
    FineCells<Q, S, PAR, true> fine;
    fine.load(p, c0);
#pragma unroll
    for (int k = 0; k < W; k++) {
      if (!fine.cell(p, k, x, y, z, c0)) continue;
      const Mom<Q> m = moments<Q>(p, fine.f[k]);
      rs += m.rho;
      ms[0] += m.jx;
      ms[1] += m.jy;
      ms[2] += m.jz;
    }
  }
  rho_bar[k] = rs * 0.125f;
  const float inv = rs > 0.f ? 1.f / rs : 0.f;
  u_bar[k] = ms[0] * inv;
  u_bar[nc + k] = ms[1] * inv;
  u_bar[2 * nc + k] = ms[2] * inv;
}

// ---- network -------------------------------------------------------------------------------
__device__ __forceinline__ float mlp_forward_one(const float* W, const float* x) {
  const float* W1 = W;
  const float* b1 = W1 + MLP_NH * MLP_NIN;
  const float* W2 = b1 + MLP_NH;
  const float* b2 = W2 + MLP_NH * MLP_NH;
  const float* W3 = b2 + MLP_NH;
  const float* b3 = W3 + MLP_NH;
  float h1[MLP_NH];
#pragma unroll 4
  for (int j = 0; j < MLP_NH; j++) {
    float s = b1[j];
#pragma unroll
    for (int k = 0; k < MLP_NIN; k++) s = fmaf(W1[j * MLP_NIN + k], x[k], s);
    h1[j] = gelu_erf(s);
  }
  float y = b3[0];
#pragma unroll 2
  for (int j = 0; j < MLP_NH; j++) {
    float s = b2[j];
#pragma unroll
    for (int k = 0; k < MLP_NH; k++) s = fmaf(W2[j * MLP_NH + k], h1[k], s);
    y = fmaf(W3[j], gelu_erf(s), y);
  }
  return y;
}

__global__ void __launch_bounds__(128) k_mlp_forward(const float* __restrict__ params, const float* __restrict__ x,
                                                     long long n, float* __restrict__ y) {
  __shared__ float W[MLP_NPARAM];
  for (int j = threadIdx.x; j < MLP_NPARAM; j += blockDim.x) W[j] = params[j];
  __syncthreads();
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  float xs[MLP_NIN];
#pragma unroll
  for (int k = 0; k < MLP_NIN; k++) xs[k] = x[s * MLP_NIN + k];
  y[s] = mlp_forward_one(W, xs);
}

// Mode of the backward kernel: given dy per sample, or the eddy-viscosity loss.
enum : int { BW_DY = 0, BW_LOSS = 1 };

struct BackArgs {
  const float* params;
  const float* x;
  const float* dy;       // BW_DY
  const float* target;   // BW_LOSS
  const float* smag;
  const float* weight;
  long long n;           // samples in the batch
  long long offset, stride;  // sample s of the batch is offset + s * stride
  float k;               // C_s0^2 / ln 2
  float* grad;           // MLP_NPARAM, zeroed before; added to (FP32 atomics)
  double* sums;          // BW_LOSS: [sum w, sum w r^2, loss, blocks done], the first two and the last zeroed
  int slot;              // (before and after); or null and the slot of call_scratch
};

// Scratch slots of lbm_closure_loss_grad (see CallScratch), zero between calls but for the loss.
constexpr int SCRATCH_SLOTS = 64, SCRATCH_DOUBLES = 4;
__device__ double call_scratch[SCRATCH_SLOTS * SCRATCH_DOUBLES];

constexpr int BW_MINB = 2;          // resident blocks per SM: 255 registers (3 blocks spill 0.6 KB and ran 20 % slower)
constexpr int BW_WARPS = 4;         // warps per block
constexpr int BW_PITCH = MLP_NH + 4;  // row pitch of the activation tiles: 128-bit accesses without bank conflicts

struct alignas(16) BackTile {       // one warp's 32 samples
  float H1[32 * BW_PITCH];          // gelu'(a1) during layer 2, then h1
  float E[32 * BW_PITCH];           // W3 gelu'(a2), then dA1
  float H2[32 * BW_PITCH];
  float X[32 * 8];                  // the 7 inputs and 1
};

struct BackSmem {
  float W1[8 * MLP_NH];             // [k][j], row 7 is b1
  float W2[MLP_NH * MLP_NH];        // [j][k]
  float b2[MLP_NH], W3[MLP_NH], b3;
  double red[2][BW_WARPS];
  bool last;
  BackTile tile[BW_WARPS];
};
static_assert(offsetof(BackSmem, W2) % 16 == 0 && offsetof(BackSmem, W3) % 8 == 0 && offsetof(BackSmem, tile) % 16 == 0,
              "128-bit and 64-bit shared accesses");
static_assert(sizeof(BackTile) >= MLP_NPARAM * sizeof(float), "a tile also holds a warp's gradient");

// GELU and its derivative Phi(a) + a phi(a) of two values, from one exponential: erf by the
// rational approximation of Abramowitz & Stegun, formula 7.1.26 (after Hastings), erf(z) =
// 1 - u (a1 + u (a2 + u (a3 + u (a4 + u a5)))) exp(-z^2), u = 1 / (1 + p z) for z >= 0; absolute
// error below 1.5e-7.  Its exponential is that of phi, which gelu_v's form would need besides its own.
__device__ __forceinline__ void gelu_both(float2 a, float2& h, float2& g) {
  float2 az, t, e, er;
  az.x = fabsf(a.x) * 0.70710678118654752f;
  az.y = fabsf(a.y) * 0.70710678118654752f;
  const float2 den = vfma(az, vset<float2>(0.3275911f), vset<float2>(1.f));
  t.x = rcp_approx(den.x);
  t.y = rcp_approx(den.y);
  float2 q = vfma(vset<float2>(1.061405429f), t, vset<float2>(-1.453152027f));
  q = vfma(q, t, vset<float2>(1.421413741f));
  q = vfma(q, t, vset<float2>(-0.284496736f));
  q = vfma(q, t, vset<float2>(0.254829592f));
  const float2 arg = vmul(az, vmul(az, vset<float2>(-1.4426950408889634f)));
  e.x = ex2_approx(arg.x);
  e.y = ex2_approx(arg.y);
  const float2 m = vfma(vmul(q, t), e, vset<float2>(-1.f));  // -erf|z|
  er.x = copysignf(m.x, a.x);
  er.y = copysignf(m.y, a.y);
  const float2 phi = vfma(er, vset<float2>(0.5f), vset<float2>(0.5f));  // Phi(a)
  h = vfma(vmul(az, vset<float2>(-0.70710678118654752f)), m, vmul(a, vset<float2>(0.5f)));
  g = vfma(vmul(a, vset<float2>(0.39894228040143268f)), e, phi);
}

// Parameter gradients of a batch.  A warp takes 32 samples at a time: each lane runs one sample
// forward and back through the network (weights by broadcast from shared memory, each row of W2
// read once for the layer and for its transpose), then the warp sums the outer products over its
// 32 samples, each lane holding a 4 x 8 tile of dW2, a row of dW1, and its entries of the rest in
// registers over all of its batches.  No barrier until the end, when the block's warps are added
// and the sums go out with one atomic per parameter and block.
// Bound by shared-memory reads of the weights (one 32-bit word per lane and clock: about 2,200
// cycles per 32 samples and SM, against 1,000 of FMA issue).  Measured with dense samples, launch
// and memset included: 122,880 samples 198 -> 43 us, 1,000,000 samples 1,399 -> 246 us (before: one
// block per 128 samples, two shared reads per FMA of the parameter sums, an atomic per parameter
// and 128 samples; with the loss also two double atomics on one address per sample).
template <int MODE>
__global__ void __launch_bounds__(32 * BW_WARPS, BW_MINB) k_mlp_backward(const __grid_constant__ BackArgs a) {
  extern __shared__ __align__(16) unsigned char back_smem_raw[];
  BackSmem& sm = *reinterpret_cast<BackSmem*>(back_smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int P = BW_PITCH;
  for (int j = tid; j < MLP_NPARAM; j += 32 * BW_WARPS) {
    const float v = a.params[j];
    int e = j;
    if (e < MLP_NH * MLP_NIN) sm.W1[(e % MLP_NIN) * MLP_NH + e / MLP_NIN] = v;
    else if ((e -= MLP_NH * MLP_NIN) < MLP_NH) sm.W1[7 * MLP_NH + e] = v;
    else if ((e -= MLP_NH) < MLP_NH * MLP_NH) sm.W2[e] = v;
    else if ((e -= MLP_NH * MLP_NH) < MLP_NH) sm.b2[e] = v;
    else if ((e -= MLP_NH) < MLP_NH) sm.W3[e] = v;
    else sm.b3 = v;
  }
  __syncthreads();
  BackTile& T = sm.tile[warp];
  float* const h1row = T.H1 + lane * P;
  float* const erow = T.E + lane * P;
  float* const h2row = T.H2 + lane * P;
  const int r4 = (lane >> 2) * 4, c8 = (lane & 3) * 8;  // this lane's tile of dW2: rows r4.., columns c8..
  float2 gW2[4][4], gW1[4];
  float gb2 = 0.f, gW3 = 0.f, gb3 = 0.f;
  double sw = 0.0, swr = 0.0;
#pragma unroll
  for (int i = 0; i < 4; i++) {
    gW1[i] = vset<float2>(0.f);
#pragma unroll
    for (int j = 0; j < 4; j++) gW2[i][j] = vset<float2>(0.f);
  }
  const long long step = 32ll * BW_WARPS * gridDim.x;
  for (long long s0 = 32ll * ((long long)warp * gridDim.x + blockIdx.x); s0 < a.n; s0 += step) {
    const long long s = s0 + lane;
    const bool valid = s < a.n;
    const long long gs = a.offset + s * a.stride;
    float xs[8], dy = 0.f, tg = 0.f, S = 0.f, w = 0.f;
#pragma unroll
    for (int k = 0; k < MLP_NIN; k++) xs[k] = valid ? a.x[gs * MLP_NIN + k] : 0.f;
    xs[7] = 1.f;
    if (valid) {
      if (MODE == BW_DY) {
        dy = a.dy[s];
      } else {
        tg = a.target[gs];
        S = a.smag[gs];
        w = a.weight[gs];
      }
    }
    *reinterpret_cast<float4*>(T.X + lane * 8) = make_float4(xs[0], xs[1], xs[2], xs[3]);
    *reinterpret_cast<float4*>(T.X + lane * 8 + 4) = make_float4(xs[4], xs[5], xs[6], xs[7]);
    // layer 1: h1 stays in registers, gelu'(a1) waits in the tile
    float2 h1[MLP_NH / 2];
#pragma unroll
    for (int j = 0; j < MLP_NH; j += 4) {
      float2 u = vset<float2>(0.f), v = vset<float2>(0.f);
#pragma unroll
      for (int k = 0; k < 8; k++) {
        const float4 wv = *reinterpret_cast<const float4*>(sm.W1 + k * MLP_NH + j);
        u = vfma(make_float2(wv.x, wv.y), vset<float2>(xs[k]), u);
        v = vfma(make_float2(wv.z, wv.w), vset<float2>(xs[k]), v);
      }
      float2 gu, gv;
      gelu_both(u, h1[j / 2], gu);
      gelu_both(v, h1[j / 2 + 1], gv);
      *reinterpret_cast<float4*>(h1row + j) = make_float4(gu.x, gu.y, gv.x, gv.y);
    }
    // layer 2 and the output; d = W2^T (W3 gelu'(a2)), the derivative of y by h1
    float2 d[MLP_NH / 2], y2 = vset<float2>(0.f);
#pragma unroll
    for (int k = 0; k < MLP_NH / 2; k++) d[k] = vset<float2>(0.f);
#pragma unroll 1
    for (int j = 0; j < MLP_NH; j += 2) {
      float2 row[2][MLP_NH / 2], a2;
#pragma unroll
      for (int i = 0; i < 2; i++) {
        float2 u = vset<float2>(0.f), v = vset<float2>(0.f);
#pragma unroll
        for (int k = 0; k < MLP_NH; k += 4) {
          const float4 wv = *reinterpret_cast<const float4*>(sm.W2 + (j + i) * MLP_NH + k);
          row[i][k / 2] = make_float2(wv.x, wv.y);
          row[i][k / 2 + 1] = make_float2(wv.z, wv.w);
          u = vfma(row[i][k / 2], h1[k / 2], u);
          v = vfma(row[i][k / 2 + 1], h1[k / 2 + 1], v);
        }
        const float2 uv = vadd(u, v);
        (i ? a2.y : a2.x) = sm.b2[j + i] + (uv.x + uv.y);
      }
      float2 h2, g2;
      gelu_both(a2, h2, g2);
      const float2 w3 = *reinterpret_cast<const float2*>(sm.W3 + j);
      y2 = vfma(w3, h2, y2);
      const float2 e = vmul(w3, g2);
      *reinterpret_cast<float2*>(h2row + j) = h2;
      *reinterpret_cast<float2*>(erow + j) = e;
#pragma unroll
      for (int k = 0; k < MLP_NH / 2; k++)
        d[k] = vfma(row[1][k], vset<float2>(e.y), vfma(row[0][k], vset<float2>(e.x), d[k]));
    }
    if (MODE == BW_LOSS) {
      const float y = sm.b3 + (y2.x + y2.y);
      const float sp = fmaxf(y, 0.f) + log1pf(expf(-fabsf(y)));
      const float sg = 1.f / (1.f + expf(-y));
      const float r = sp * a.k * S - tg;
      dy = valid ? 2.f * w * r * a.k * S * sg : 0.f;  // unnormalised; scaled by 1 / sum w at the end
      if (valid) {
        sw += (double)w;
        swr += (double)w * (double)r * (double)r;
      }
    }
    // dA1 in d; h1 to its tile
#pragma unroll
    for (int k = 0; k < MLP_NH; k += 4) {
      const float4 g1 = *reinterpret_cast<const float4*>(h1row + k);
      d[k / 2] = vmul(d[k / 2], vmul(make_float2(g1.x, g1.y), vset<float2>(dy)));
      d[k / 2 + 1] = vmul(d[k / 2 + 1], vmul(make_float2(g1.z, g1.w), vset<float2>(dy)));
      *reinterpret_cast<float4*>(h1row + k) = make_float4(h1[k / 2].x, h1[k / 2].y, h1[k / 2 + 1].x, h1[k / 2 + 1].y);
    }
    gb3 += dy;
    __syncwarp();
    // dW2 += dy e h1^T, db2 += dy e, dW3 += dy h2
#pragma unroll 2
    for (int q = 0; q < 32; q++) {
      const float dq = __shfl_sync(0xffffffffu, dy, q);
      const float4 e4 = *reinterpret_cast<const float4*>(T.E + q * P + r4);
      const float4 ha = *reinterpret_cast<const float4*>(T.H1 + q * P + c8);
      const float4 hb = *reinterpret_cast<const float4*>(T.H1 + q * P + c8 + 4);
      const float ev[4] = {e4.x * dq, e4.y * dq, e4.z * dq, e4.w * dq};
#pragma unroll
      for (int i = 0; i < 4; i++) {
        const float2 ee = vset<float2>(ev[i]);
        gW2[i][0] = vfma(ee, make_float2(ha.x, ha.y), gW2[i][0]);
        gW2[i][1] = vfma(ee, make_float2(ha.z, ha.w), gW2[i][1]);
        gW2[i][2] = vfma(ee, make_float2(hb.x, hb.y), gW2[i][2]);
        gW2[i][3] = vfma(ee, make_float2(hb.z, hb.w), gW2[i][3]);
      }
      gb2 = fmaf(T.E[q * P + lane], dq, gb2);
      gW3 = fmaf(T.H2[q * P + lane], dq, gW3);
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < MLP_NH; k += 4)
      *reinterpret_cast<float4*>(erow + k) = make_float4(d[k / 2].x, d[k / 2].y, d[k / 2 + 1].x, d[k / 2 + 1].y);
    __syncwarp();
    // dW1 += dA1 x^T, db1 += dA1 (the eighth input is 1)
#pragma unroll 4
    for (int q = 0; q < 32; q++) {
      const float2 dq = vset<float2>(T.E[q * P + lane]);
      const float4 xa = *reinterpret_cast<const float4*>(T.X + q * 8);
      const float4 xb = *reinterpret_cast<const float4*>(T.X + q * 8 + 4);
      gW1[0] = vfma(dq, make_float2(xa.x, xa.y), gW1[0]);
      gW1[1] = vfma(dq, make_float2(xa.z, xa.w), gW1[1]);
      gW1[2] = vfma(dq, make_float2(xb.x, xb.y), gW1[2]);
      gW1[3] = vfma(dq, make_float2(xb.z, xb.w), gW1[3]);
    }
    __syncwarp();
  }
  // this warp's gradient in parameter order, over its tile
  {
    float* G = reinterpret_cast<float*>(&T);
    __syncwarp();
    const float w1[8] = {gW1[0].x, gW1[0].y, gW1[1].x, gW1[1].y, gW1[2].x, gW1[2].y, gW1[3].x, gW1[3].y};
#pragma unroll
    for (int k = 0; k < MLP_NIN; k++) G[lane * MLP_NIN + k] = w1[k];
    G += MLP_NH * MLP_NIN;
    G[lane] = w1[7];
    G += MLP_NH;
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
      for (int j = 0; j < 4; j++) {
        G[(r4 + i) * MLP_NH + c8 + 2 * j] = gW2[i][j].x;
        G[(r4 + i) * MLP_NH + c8 + 2 * j + 1] = gW2[i][j].y;
      }
    G += MLP_NH * MLP_NH;
    G[lane] = gb2;
    G[MLP_NH + lane] = gW3;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) gb3 += __shfl_xor_sync(0xffffffffu, gb3, o);
    if (lane == 0) G[2 * MLP_NH] = gb3;
    if (MODE == BW_LOSS) {
      sw = warp_sum(sw);
      swr = warp_sum(swr);
      if (lane == 0) {
        sm.red[0][warp] = sw;
        sm.red[1][warp] = swr;
      }
    }
  }
  __syncthreads();
  for (int e = tid; e < MLP_NPARAM; e += 32 * BW_WARPS) {
    float g = 0.f;
#pragma unroll
    for (int w = 0; w < BW_WARPS; w++) g += reinterpret_cast<const float*>(&sm.tile[w])[e];
    atomicAdd(a.grad + e, g);
  }
  if (MODE != BW_LOSS) return;
  double* const sums = a.sums ? a.sums : call_scratch + a.slot * SCRATCH_DOUBLES;
  if (tid < 2) {
    double v = 0.0;
    for (int w = 0; w < BW_WARPS; w++) v += sm.red[tid][w];
    atomicAdd(sums + tid, v);
  }
  // the last block to finish divides by the sum of the weights
  __threadfence();
  __syncthreads();
  if (tid == 0) sm.last = atomicAdd(reinterpret_cast<unsigned*>(sums + 3), 1u) == gridDim.x - 1;
  __syncthreads();
  if (!sm.last) return;
  __threadfence();
  const double wsum = __ldcg(sums), wrr = __ldcg(sums + 1);
  const float inv = wsum > 0.0 ? (float)(1.0 / wsum) : 0.f;
  for (int e = tid; e < MLP_NPARAM; e += 32 * BW_WARPS) a.grad[e] = __ldcg(a.grad + e) * inv;
  __syncthreads();  // all threads have read the sums
  if (tid == 0) {
    sums[0] = sums[1] = sums[3] = 0.0;
    sums[2] = wsum > 0.0 ? wrr / wsum : 0.0;
  }
}

__global__ void k_adam(float* p, const float* g, float* m, float* v, int n, float lr, float b1,
                       float b2, float eps, float c1, float c2) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const float gj = g[j];
  const float mj = b1 * m[j] + (1.f - b1) * gj;
  const float vj = b2 * v[j] + (1.f - b2) * gj * gj;
  m[j] = mj;
  v[j] = vj;
  p[j] -= lr * (mj / c1) / (sqrtf(vj / c2) + eps);
}

}  // namespace lbm

using namespace lbm;

// ---- host side --------------------------------------------------------------------------------

struct lbm_s;
// accessors into the handle (defined with the rest of the ABI)
KParams lbm_internal_kparams(lbm_handle h);
int lbm_internal_info(lbm_handle h, int* q, int* precision, int* parity, int* closure, int* nx, int* ny,
                      int* nz, void** stream);
lbm_status lbm_internal_fail(lbm_handle h, lbm_status s, const char* msg);

template <int Q, class S>
static void launch_samples(const KParams& p, int parity, const SampleArgs& a, long long nc, cudaStream_t st) {
  const unsigned blocks = (unsigned)((nc + 127) / 128);
  if (parity == 0) k_closure_samples<Q, S, 0><<<blocks, 128, 0, st>>>(p, a);
  else if (parity == 1) k_closure_samples<Q, S, 1><<<blocks, 128, 0, st>>>(p, a);
  else k_closure_samples<Q, S, 2><<<blocks, 128, 0, st>>>(p, a);
}

template <int Q, class S>
static void launch_filter(const KParams& p, int parity, int ncx, int ncy, int ncz, float* rb, float* ub,
                          cudaStream_t st) {
  const long long nc = (long long)ncx * ncy * ncz;
  const unsigned blocks = (unsigned)((nc + 127) / 128);
  if (parity == 0) k_filter2<Q, S, 0><<<blocks, 128, 0, st>>>(p, ncx, ncy, ncz, rb, ub);
  else if (parity == 1) k_filter2<Q, S, 1><<<blocks, 128, 0, st>>>(p, ncx, ncy, ncz, rb, ub);
  else k_filter2<Q, S, 2><<<blocks, 128, 0, st>>>(p, ncx, ncy, ncz, rb, ub);
}

extern "C" {

lbm_status lbm_filter2(lbm_handle fine, float* rho_bar, float* u_bar) {
  if (!fine) return LBM_EINVAL;
  if (!rho_bar || !u_bar) return lbm_internal_fail(fine, LBM_EINVAL, "lbm_filter2: NULL output");
  int q, prec, parity, closure, nx, ny, nz;
  void* stream;
  lbm_internal_info(fine, &q, &prec, &parity, &closure, &nx, &ny, &nz, &stream);
  KParams p = lbm_internal_kparams(fine);
  if (p.outflow) return lbm_internal_fail(fine, LBM_EUNSUPPORTED, "lbm_filter2: lattices with an outflow face");
  if (nx % 2 || ny % 2 || nz % 2) return lbm_internal_fail(fine, LBM_EINVAL, "lbm_filter2: sizes must be even");
  const cudaStream_t st = (cudaStream_t)stream;
  if (q == 19) {
    if (prec == LBM_F32) launch_filter<19, float>(p, parity, nx / 2, ny / 2, nz / 2, rho_bar, u_bar, st);
    else if (prec == LBM_F16_SHIFTED) launch_filter<19, __half>(p, parity, nx / 2, ny / 2, nz / 2, rho_bar, u_bar, st);
    else launch_filter<19, __nv_bfloat16>(p, parity, nx / 2, ny / 2, nz / 2, rho_bar, u_bar, st);
  } else {
    if (prec == LBM_F32) launch_filter<27, float>(p, parity, nx / 2, ny / 2, nz / 2, rho_bar, u_bar, st);
    else if (prec == LBM_F16_SHIFTED) launch_filter<27, __half>(p, parity, nx / 2, ny / 2, nz / 2, rho_bar, u_bar, st);
    else launch_filter<27, __nv_bfloat16>(p, parity, nx / 2, ny / 2, nz / 2, rho_bar, u_bar, st);
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return lbm_internal_fail(fine, LBM_ECUDA, cudaGetErrorString(e));
  return LBM_OK;
}

lbm_status lbm_closure_samples(lbm_handle fine, double tau0_c, double cs0, const double scale[2], float* x,
                               float* target, float* smag, float* weight) {
  if (!fine) return LBM_EINVAL;
  if (!x || !target || !smag || !weight || !scale)
    return lbm_internal_fail(fine, LBM_EINVAL, "lbm_closure_samples: NULL output");
  int q, prec, parity, closure, nx, ny, nz;
  void* stream;
  lbm_internal_info(fine, &q, &prec, &parity, &closure, &nx, &ny, &nz, &stream);
  KParams p = lbm_internal_kparams(fine);
  if (p.outflow)
    return lbm_internal_fail(fine, LBM_EUNSUPPORTED, "lbm_closure_samples: lattices with an outflow face");
  if (nx % 2 || ny % 2 || nz % 2)
    return lbm_internal_fail(fine, LBM_EINVAL, "lbm_closure_samples: fine sizes must be even");
  SampleArgs a;
  a.x = x;
  a.target = target;
  a.smag = smag;
  a.weight = weight;
  a.ncx = nx / 2;
  a.ncy = ny / 2;
  a.ncz = nz / 2;
  a.tau0_c = (float)tau0_c;
  a.cs0sq = (float)(cs0 * cs0);
  a.scale_pi = (float)scale[0];
  a.scale_rho = (float)scale[1];
  a.smag_fine = closure == LBM_CLOSURE_SMAG;
  const long long nc = (long long)a.ncx * a.ncy * a.ncz;
  const cudaStream_t st = (cudaStream_t)stream;
  if (q == 19) {
    if (prec == LBM_F32) launch_samples<19, float>(p, parity, a, nc, st);
    else if (prec == LBM_F16_SHIFTED) launch_samples<19, __half>(p, parity, a, nc, st);
    else launch_samples<19, __nv_bfloat16>(p, parity, a, nc, st);
  } else {
    if (prec == LBM_F32) launch_samples<27, float>(p, parity, a, nc, st);
    else if (prec == LBM_F16_SHIFTED) launch_samples<27, __half>(p, parity, a, nc, st);
    else launch_samples<27, __nv_bfloat16>(p, parity, a, nc, st);
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return lbm_internal_fail(fine, LBM_ECUDA, cudaGetErrorString(e));
  return LBM_OK;
}

// Scratch of a call that synchronises before it returns: one of SCRATCH_SLOTS small blocks in the
// module's own device storage, taken for the duration of the call by any thread and stream, or
// stream-ordered memory where all are taken.  An allocation per call cost 0.1 ms: the default pool gives
// its memory back at every synchronisation and maps 32 MB again.  The storage lives and dies with the
// module in its context and the host keeps no address of it (after a device reset that would be stale);
// the kernel finds the slot itself and leaves it zeroed, so a call asks for no address and zeroes nothing.
class CallScratch {
 public:
  cudaError_t take(cudaStream_t st) {
    cudaError_t e = cudaGetDevice(&dev_);
    if (e != cudaSuccess) return e;
    if (dev_ < DEVICES) {
      std::lock_guard<std::mutex> hold(lock());
      for (int i = 0; slot < 0 && i < SCRATCH_SLOTS; i++)
        if (!(used()[dev_] >> i & 1)) {
          used()[dev_] |= 1ull << i;
          slot = i;
        }
    }
    if (slot >= 0) return cudaSuccess;
    e = cudaMallocAsync((void**)&p, SCRATCH_DOUBLES * sizeof(double), st);
    return e == cudaSuccess ? cudaMemsetAsync(p, 0, SCRATCH_DOUBLES * sizeof(double), st) : e;
  }
  // after the call's work is queued; idle: the stream has been waited for
  void give(cudaStream_t st, bool idle) {
    if (slot < 0) {
      if (p) cudaFreeAsync(p, st);
    } else if (idle) {  // after an error the slot stays taken: its work may still be running
      std::lock_guard<std::mutex> hold(lock());
      used()[dev_] &= ~(1ull << slot);
    }
    p = nullptr;
  }
  double* p = nullptr;
  int slot = -1;

 private:
  static constexpr int DEVICES = 64;
  static std::mutex& lock() {
    static std::mutex m;
    return m;
  }
  static uint64_t* used() {  // a bit per slot and device
    static uint64_t u[DEVICES];
    return u;
  }
  int dev_ = 0;
};

lbm_status lbm_mlp_forward(const float* params, const float* x, int64_t n, float* y, void* stream) {
  if (!params || !x || !y || n < 0) {
    lbm_internal_set_error("lbm_mlp_forward: bad argument");
    return LBM_EINVAL;
  }
  if (n == 0) return LBM_OK;
  k_mlp_forward<<<(unsigned)((n + 127) / 128), 128, 0, (cudaStream_t)stream>>>(params, x, n, y);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    lbm_internal_set_error(cudaGetErrorString(e));
    return LBM_ECUDA;
  }
  return LBM_OK;
}

// Grid of the backward kernel for n samples: what is resident at once, or a block per 32 samples.
// (lbm_closure_loss_grad, 122,880 samples with stride 64, and an Adam step: 752 -> 116 us a call pair.)
static cudaError_t backward_grid(int64_t n, unsigned* grid) {
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  *grid = (unsigned)std::min<int64_t>((n + 31) / 32, (int64_t)BW_MINB * std::max(nsm, 1));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_mlp_backward<BW_DY>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BackSmem));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_mlp_backward<BW_LOSS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BackSmem));
  return e;
}

lbm_status lbm_mlp_backward(const float* params, const float* x, const float* dy, int64_t n, float* grad,
                            void* stream) {
  if (!params || !x || !dy || !grad || n < 0) {
    lbm_internal_set_error("lbm_mlp_backward: bad argument");
    return LBM_EINVAL;
  }
  const cudaStream_t st = (cudaStream_t)stream;
  unsigned grid = 0;
  cudaError_t e = backward_grid(n, &grid);
  if (e == cudaSuccess) e = cudaMemsetAsync(grad, 0, MLP_NPARAM * sizeof(float), st);
  if (e == cudaSuccess && n > 0) {
    BackArgs a{};
    a.params = params;
    a.x = x;
    a.dy = dy;
    a.n = n;
    a.offset = 0;
    a.stride = 1;
    a.grad = grad;
    k_mlp_backward<BW_DY><<<grid, 32 * BW_WARPS, sizeof(BackSmem), st>>>(a);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) {
    lbm_internal_set_error(cudaGetErrorString(e));
    return LBM_ECUDA;
  }
  return LBM_OK;
}

lbm_status lbm_closure_loss_grad(const float* params, const float* x, const float* target, const float* smag,
                                 const float* weight, int64_t n, int64_t offset, int64_t stride, double cs0,
                                 float* grad, double* loss, void* stream) {
  if (!params || !x || !target || !smag || !weight || !grad || !loss || n < 0 || offset < 0 || stride < 1) {
    lbm_internal_set_error("lbm_closure_loss_grad: bad argument");
    return LBM_EINVAL;
  }
  const cudaStream_t st = (cudaStream_t)stream;
  CallScratch scratch;
  unsigned grid = 0;
  cudaError_t e = backward_grid(n, &grid);
  if (e == cudaSuccess) e = scratch.take(st);
  if (e == cudaSuccess) e = cudaMemsetAsync(grad, 0, MLP_NPARAM * sizeof(float), st);
  if (e == cudaSuccess && n > 0) {
    BackArgs a{};
    a.params = params;
    a.x = x;
    a.target = target;
    a.smag = smag;
    a.weight = weight;
    a.n = n;
    a.offset = offset;
    a.stride = stride;
    a.k = (float)(cs0 * cs0 / std::log(2.0));
    a.grad = grad;
    a.sums = scratch.p;
    a.slot = scratch.slot;
    k_mlp_backward<BW_LOSS><<<grid, 32 * BW_WARPS, sizeof(BackSmem), st>>>(a);
    e = cudaGetLastError();
  }
  static const double zero = 0.0;
  if (e == cudaSuccess && n == 0) e = cudaMemcpyAsync(loss, &zero, sizeof(double), cudaMemcpyDefault, st);
  else if (e == cudaSuccess && scratch.p) e = cudaMemcpyAsync(loss, scratch.p + 2, sizeof(double), cudaMemcpyDefault, st);
  else if (e == cudaSuccess)
    e = cudaMemcpyFromSymbolAsync(loss, call_scratch, sizeof(double), (scratch.slot * SCRATCH_DOUBLES + 2) * sizeof(double),
                                  cudaMemcpyDefault, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  scratch.give(st, e == cudaSuccess);
  if (e != cudaSuccess) {
    lbm_internal_set_error(cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA;
  }
  return LBM_OK;
}

lbm_status lbm_adam_step(float* params, const float* grad, float* m, float* v, int n, double lr, double beta1,
                         double beta2, double eps, int64_t t, void* stream) {
  if (!params || !grad || !m || !v || n < 0 || t < 1) {
    lbm_internal_set_error("lbm_adam_step: bad argument");
    return LBM_EINVAL;
  }
  if (n == 0) return LBM_OK;
  const float c1 = (float)(1.0 - std::pow(beta1, (double)t));
  const float c2 = (float)(1.0 - std::pow(beta2, (double)t));
  k_adam<<<(n + 255) / 256, 256, 0, (cudaStream_t)stream>>>(params, grad, m, v, n, (float)lr, (float)beta1,
                                                           (float)beta2, (float)eps, c1, c2);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    lbm_internal_set_error(cudaGetErrorString(e));
    return LBM_ECUDA;
  }
  return LBM_OK;
}

}  // extern "C"
