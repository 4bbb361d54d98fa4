// lbm_h2.cuh -- the step for half-precision storage with two x-adjacent cells per thread.
//
// A lane owns cells (x, x+1), x even, so every slot the pair owns in a direction with
// c_x = 0 (and every own-cell slot) is one aligned 32-bit word holding both cells' 16-bit
// values: one load and one store move two populations.  Slots shifted in x by the odd AA
// gather (c_x != 0) straddle two words and move as two 16-bit accesses.  The loaded words
// stay packed (one register per direction for both cells) until the collision, which runs on
// both cells at once in the packed FP32x2 pipe (float2 operands: FFMA2/FADD2/FMUL2); the two
// results are rounded and packed into one word each.  This halves the memory instructions,
// the address arithmetic and the arithmetic instructions per cell and doubles the bytes a
// thread keeps in flight.
//
// In the pull step a lane with a cell that needs boundary rules, a periodic y/z wrap or no update
// loads its two cells by the one-cell code, out of line; in the odd AA step a warp with such a lane
// runs the one-cell code for its cells.  The zero-gradient outflow passes what cell x-1 receives
// from the lane that owns it (nx % 32 != 1 keeps x = nx-1 off lane 0).
// Block (32, 4) covers 64 x 4 cells of one z plane; grid (ceil(nxp/64), ceil(ny/4), nz).
#pragma once

#include "lbm_kernels.cuh"

namespace lbm {

// 16-bit pattern of v rounded to the storage precision (round to nearest even)
template <class S> __device__ __forceinline__ uint32_t bits16(float v);
template <> __device__ __forceinline__ uint32_t bits16<__half>(float v) { return __half_as_ushort(__float2half_rn(v)); }
template <> __device__ __forceinline__ uint32_t bits16<__nv_bfloat16>(float v) {
  return __bfloat16_as_ushort(__float2bfloat16_rn(v));
}

// Checked 32-bit (two cells) and 16-bit (one cell) population accesses.
__device__ __forceinline__ uint32_t ld32(const KParams& p, const void* a) {
  return chk(p, a, 4, CHK_POP) ? *static_cast<const uint32_t*>(a) : 0u;
}
__device__ __forceinline__ void st32(const KParams& p, void* a, uint32_t v) {
  if (chk(p, a, 4, CHK_POP)) *static_cast<uint32_t*>(a) = v;
}
__device__ __forceinline__ uint32_t ld16(const KParams& p, const void* a) {
  return chk(p, a, 2, CHK_POP) ? *static_cast<const unsigned short*>(a) : 0u;
}
__device__ __forceinline__ void st16(const KParams& p, void* a, uint32_t v) {
  if (chk(p, a, 2, CHK_POP)) *static_cast<unsigned short*>(a) = (unsigned short)v;
}

// Zero-gradient outflow for x-pairs: cell x-1 of lane t's first cell is lane t-1's second.
template <int Q>
__device__ __forceinline__ void outflow_fix2(const KParams& p, int x0, float (&fa)[Q], float (&fb)[Q],
                                             unsigned oa, unsigned ob) {
  if (!p.outflow) return;
  if (!(x0 <= p.nx - 1 && p.nx - 1 < x0 + 64)) return;  // warp-uniform
#pragma unroll
  for (int i = 0; i < Q; i++) {
    if (cx(i) != -1) continue;
    const float v = __shfl_up_sync(0xffffffffu, fb[i], 1);
    if (ob & (1u << i)) fb[i] = fa[i];  // x-1 is this lane's first cell (never itself an outflow cell)
    if (oa & (1u << i)) fa[i] = v;
  }
}

// Slot offsets of the two cells' sources in a direction with c_x != 0 (periodic x wrap).  LAST: the
// row's last cell may be the first of its pair (odd nx, see k_step_h2), else it is always the second.
template <bool LAST = false>
__device__ __forceinline__ void xsrc(int c, const KParams& p, int x, int cell, int& ca, int& cb) {
  if (c > 0) {  // sources x-1, x
    ca = cell + (x == 0 ? p.nx : 0);
    cb = cell + 1;
  } else {       // sources x+1, x+2
    ca = cell - (LAST && x == p.nx - 1 ? p.nx : 0);
    cb = cell + 1 - (x + 1 == p.nx - 1 ? p.nx : 0);
  }
}

// One-cell code for both cells of a lane (warps with a non-interior cell).  Kept out of
// line so that the rare path does not take registers from the fast one.
template <int Q, class S, int CL, int LOAD, int STORE, bool STATS>
__device__ __noinline__ void pair_fallback(const KParams& p, int x, int y, int z, int cell, int clsA, int clsB,
                                           float (&v)[NSTAT]) {
  float fa[Q], fb[Q];
  unsigned oa, ob;
  load_state<Q, S, LOAD>(p, x, y, z, cell, clsA, fa, oa);
  load_state<Q, S, LOAD>(p, x + 1, y, z, cell + 1, clsB, fb, ob);
  outflow_fix2<Q>(p, 64 * blockIdx.x, fa, fb, oa, ob);
  if (clsA != CLS_SKIP) {
    Macro<float> M;
    const float r = collide<Q, CL, float, false>(p, fa, STATS ? &M : nullptr);
    if (!(r > 0.f && r < 3.0e38f)) flag_unstable(p);
    store_state<Q, S, STORE>(p, x, y, z, cell, clsA, fa);
    if (STATS) stat_values(M, v);
  }
  if (clsB != CLS_SKIP) {
    Macro<float> M;
    const float r = collide<Q, CL, float, false>(p, fb, STATS ? &M : nullptr);
    if (!(r > 0.f && r < 3.0e38f)) flag_unstable(p);
    store_state<Q, S, STORE>(p, x + 1, y, z, cell + 1, clsB, fb);
    if (STATS) {
      float w[NSTAT];
      stat_values(M, w);
#pragma unroll
      for (int k = 0; k < NSTAT; k++) v[k] += w[k];
    }
  }
}

// ---- two-grid pull: every warp takes the pair path ---------------------------------------
// A lane whose cells are not both interior loads them with the boundary rules of the one-cell
// step (out of line, below); the collision and the own-cell stores are common to all lanes, a
// lane with a skipped (solid or padding) cell storing only its other cell's half.

// Both cells of a boundary lane with the one-cell loads, packed into hs (the loaded values are
// exact in the storage precision); ca, cb: class bytes.  Out of line: the rule-by-rule loads are
// long, run for few lanes, and inlined they would crowd the instruction cache of every warp.
template <int Q, class S, int PAR>
__device__ __noinline__ void load_pair_rules(const KParams& p, int x, int y, int z, int cell, int ca, int cb,
                                             uint32_t* hs, unsigned* oa, unsigned* ob) {
  float f[Q];
  auto one = [&](int xc, int cc, int cbyte, unsigned& om) {
    if (PAR != 0 && (cbyte & CLS_XFACE)) gather_xface<Q, S, PAR == 0 ? 1 : PAR>(p, xc, cc, f, om);
    else load_state<Q, S, PAR, true>(p, xc, y, z, cc, cbyte & CLS_MASK, f, om);
  };
  unsigned om = 0;
  one(x, cell, ca, om);
  *oa = om;
#pragma unroll
  for (int i = 0; i < Q; i++) hs[i] = bits16<S>(f[i]);
  om = 0;
  one(x + 1, cell + 1, cb, om);
  *ob = om;
#pragma unroll
  for (int i = 0; i < Q; i++) hs[i] |= bits16<S>(f[i]) << 16;
}

// Zero-gradient outflow on packed words: x = nx-1 takes what x-1 receives (the lane's own
// first cell, or the previous lane's second).  Warp-uniform condition, full-mask shuffles.
template <int Q>
__device__ __forceinline__ void outflow_fix_packed(const KParams& p, int x0, uint32_t (&h)[Q], unsigned oa,
                                                   unsigned ob) {
  if (!p.outflow) return;
  if (!(x0 <= p.nx - 1 && p.nx - 1 < x0 + 64)) return;
#pragma unroll
  for (int i = 0; i < Q; i++) {
    if (cx(i) != -1) continue;
    const uint32_t prev = __shfl_up_sync(0xffffffffu, h[i], 1);
    if (ob & (1u << i)) h[i] = (h[i] & 0xffffu) | (h[i] << 16);
    if (oa & (1u << i)) h[i] = (h[i] & 0xffff0000u) | (prev >> 16);
  }
}

#ifndef LBM_H2_PACKED19
#define LBM_H2_PACKED19 0
#endif
#ifndef LBM_H2_PACKED27
#define LBM_H2_PACKED27 1
#endif
#ifndef LBM_H2_MINB27
#define LBM_H2_MINB27 5
#endif

// The collision of both cells (float2 lanes).  PACKED: the populations stay packed and are
// unpacked at each use (fewer live registers); else they are unpacked once into float2 values.
template <int Q, class S, int CL, bool PACKED>
__device__ __forceinline__ float2 collide_pair(const KParams& p, uint32_t (&h)[Q], Macro<float2>* mout) {
  if constexpr (PACKED) {
    PackedPops<Q, S> a{h};
    const Macro<float2> M = macro_acc<Q, CL != CL_NONE, float2>(p, a);
    if (mout) *mout = M;
    float2 wp = vset<float2>(p.omega_p), wm = vset<float2>(p.omega_m);
    if (CL != CL_NONE) {
      les_rates(p, M.qn.x, M.inv.x, p.cs2, wp.x, wm.x);
      les_rates(p, M.qn.y, M.inv.y, p.cs2, wp.y, wm.y);
    }
    relax_lean<Q, float2>(p, a, M, wp, wm);
    return M.rho;
  } else {
    float2 f[Q];
#pragma unroll
    for (int i = 0; i < Q; i++) f[i] = unpack2<S>(h[i]);
    const float2 rho = collide<Q, CL, float2, false>(p, f, mout);
#pragma unroll
    for (int i = 0; i < Q; i++) h[i] = pack2rn<S>(f[i]);
    return rho;
  }
}

// Natural layout after a streaming step: the copied slots of the outflow face were not written;
// their directions in the cell at x = nx - 1 (oa: the lane's first cell, ob: its second).
template <int Q>
__device__ __forceinline__ void own_outflow_masks(const KParams& p, int x, int cell, int clsA, int clsB, unsigned& oa,
                                                  unsigned& ob) {
  if (!p.outflow || p.nat_valid) return;
  const bool endA = x == p.nx - 1 && clsA == CLS_BOUNDARY, endB = x + 1 == p.nx - 1 && clsB == CLS_BOUNDARY;
  if (!endA && !endB) return;
  const unsigned long long r = rule_at(p, cell + (endB ? 1 : 0));
  unsigned m = 0;
#pragma unroll
  for (int i = 0; i < Q; i++)
    if (cx(i) == -1 && ((r >> (2 * i)) & 3) == R_SPECIAL) m |= 1u << i;
  (endB ? ob : oa) = m;
}

// SPLIT (gather step of a handle with a cell list, no statistics): only the interior cells and
// the simple inflow/outflow face cells are updated here, the listed ones by k_step_list.  A lane with one interior cell loads both cells'
// words (the other cell's sources, one x further, stay inside the arrays) and stores one half.
// The packed loads of a lane whose two cells take the fast path.
template <int Q, class S, int LOAD, bool LAST = false>
__device__ __forceinline__ void pair_loads(const KParams& p, int x, int cell, uint32_t (&h)[Q]) {
#pragma unroll
  for (int i = 0; i < Q; i++) {
    if (LOAD == 0) {
      h[i] = ld32(p, plane_ptr<S>(p, i) + cell);
    } else {
      const S* base = static_cast<const S*>(LOAD == 1 ? p.ga[i] : p.gb[i]);
      if (cx(i) == 0) {
        h[i] = chk(p, base + cell, 4, CHK_POP) ? ldh_u32(base + cell) : 0u;
      } else {
        int a, b;
        xsrc<LAST>(cx(i), p, x, cell, a, b);
        const uint32_t lo = chk(p, base + a, 2, CHK_POP) ? ldh_u16(base + a) : 0u;
        const uint32_t hi = chk(p, base + b, 2, CHK_POP) ? ldh_u16(base + b) : 0u;
        h[i] = lo | (hi << 16);
      }
    }
  }
}

// Statistics of the live cells of a pair.
__device__ __forceinline__ void pair_stats(const Macro<float2>& M2, bool liveA, bool liveB, float (&v)[NSTAT]) {
  float va[NSTAT], vb[NSTAT];
  Macro<float> Ma, Mb;
  Ma.ux = M2.ux.x; Ma.uy = M2.uy.x; Ma.uz = M2.uz.x;
  Mb.ux = M2.ux.y; Mb.uy = M2.uy.y; Mb.uz = M2.uz.y;
  stat_values(Ma, va);
  stat_values(Mb, vb);
#pragma unroll
  for (int k = 0; k < NSTAT; k++) v[k] = (liveA ? va[k] : 0.f) + (liveB ? vb[k] : 0.f);
}

// The split step's inflow/outflow face cells (CLS_XFACE; their other sources are plain fluid
// neighbours, so the fast loads hold them): the directions crossing the face take the
// moving-wall value of the own cell (inflow, x = 0: always the lane's first cell) or what the
// upstream cell x - 1 receives (outflow; x - 1 is the lane's first cell or, for a first cell
// at x = nx - 1, a plain gather one cell back).
template <int Q, class S>
__device__ __forceinline__ void xface_fix(const KParams& p, int x, int cell, bool xfA, bool xfB, uint32_t (&h)[Q]) {
  if (xfA && x == 0) {
#pragma unroll
    for (int i = 0; i < Q; i++) {
      if (cx(i) != 1) continue;
      const float v = rnd<S>(ldp<S>(p, plane_ptr<S>(p, opp(i)) + cell) + p.inflow_term[i]);
      h[i] = (h[i] & 0xffff0000u) | bits16<S>(v);
    }
  } else if (xfA) {  // x = nx - 1
#pragma unroll
    for (int i = 0; i < Q; i++)
      if (cx(i) == -1) h[i] = (h[i] & 0xffff0000u) | ld16(p, static_cast<const S*>(p.gb[i]) + cell - 1);
  }
  if (xfB) {  // x + 1 = nx - 1
#pragma unroll
    for (int i = 0; i < Q; i++)
      if (cx(i) == -1) h[i] = (h[i] & 0xffffu) | (h[i] << 16);
  }
}

template <int Q, class S, int CL, int LOAD, bool STATS, bool SPLIT, bool LAST>
__device__ __forceinline__ void pair_pull(const KParams& p, int x, int y, int z, int cell, int clsA, int clsB,
                                          bool fast, float (&v)[NSTAT], bool xfA, bool xfB) {
  constexpr bool PACKED = Q == 27 ? LBM_H2_PACKED27 : LBM_H2_PACKED19;
  static_assert(!SPLIT || (LOAD == 2 && !STATS), "the split runs the gather step without statistics");
  uint32_t h[Q];
  unsigned oa = 0, ob = 0;
  if (SPLIT) {
    if (clsA != CLS_INTERIOR && clsB != CLS_INTERIOR && !xfA && !xfB) return;
    fast = true;
  }
  if (fast) {
    pair_loads<Q, S, LOAD, LAST>(p, x, cell, h);
  } else {
    uint32_t hs[Q];
    load_pair_rules<Q, S, LOAD>(p, x, y, z, cell, clsA | (xfA ? CLS_XFACE : 0), clsB | (xfB ? CLS_XFACE : 0), hs, &oa, &ob);
#pragma unroll
    for (int i = 0; i < Q; i++) h[i] = hs[i];
  }
  if (!SPLIT) outflow_fix_packed<Q>(p, 64 * blockIdx.x, h, oa, ob);
  else if (xfA || xfB) xface_fix<Q, S>(p, x, cell, xfA, xfB, h);
  Macro<float2> M2;
  const float2 rho = collide_pair<Q, S, CL, PACKED>(p, h, STATS ? &M2 : nullptr);
  const bool liveA = SPLIT ? (clsA == CLS_INTERIOR || xfA) : clsA != CLS_SKIP;
  const bool liveB = SPLIT ? (clsB == CLS_INTERIOR || xfB) : clsB != CLS_SKIP;
  if ((liveA && !(rho.x > 0.f && rho.x < 3.0e38f)) || (liveB && !(rho.y > 0.f && rho.y < 3.0e38f)))
    flag_unstable(p);
  if (STATS) pair_stats(M2, liveA, liveB, v);
  if (liveA && liveB) {
#pragma unroll
    for (int i = 0; i < Q; i++) st32(p, static_cast<S*>(p.fq[i]) + cell, h[i]);
  } else if (liveA) {
#pragma unroll
    for (int i = 0; i < Q; i++) st16(p, static_cast<S*>(p.fq[i]) + cell, h[i] & 0xffffu);
  } else if (liveB) {
#pragma unroll
    for (int i = 0; i < Q; i++) st16(p, static_cast<S*>(p.fq[i]) + cell + 1, h[i] >> 16);
  }
}

// ---- AA even: every warp takes the pair path ----------------------------------------------
// The even step reads and writes own slots whatever a cell's class: only the copied slots of the
// outflow face (x = nx - 1) are taken from the upstream cell, and a lane with one cell that is not
// updated stores its other half.  Before, one such lane (the odd end of a row, a wall, a seam)
// sent its whole warp through the one-cell code twice: 251x130x121 FP16 D3Q19 channel 75 -> 66 us,
// 375x190x187 tunnel 243 -> 206 us, 512x256x128 261 -> 244 us; D3Q27 (one-cell kernel before)
// 102 -> 98, 342 -> 309 and 412 -> 367 us.
template <int Q, class S, int CL, bool STATS>
__device__ __forceinline__ void pair_even(const KParams& p, int x, int cell, int clsA, int clsB, float (&v)[NSTAT]) {
  constexpr bool PACKED = Q == 27 ? LBM_H2_PACKED27 : LBM_H2_PACKED19;
  const bool liveA = clsA != CLS_SKIP, liveB = clsB != CLS_SKIP;
  uint32_t h[Q];
  unsigned oa = 0, ob = 0;
  if (liveA || liveB) {
#pragma unroll
    for (int i = 0; i < Q; i++) h[i] = ld32(p, plane_ptr<S>(p, i) + cell);
    own_outflow_masks<Q>(p, x, cell, clsA, clsB, oa, ob);
  } else {
#pragma unroll
    for (int i = 0; i < Q; i++) h[i] = 0;
  }
  outflow_fix_packed<Q>(p, 64 * blockIdx.x, h, oa, ob);
  if (!liveA && !liveB) return;
  Macro<float2> M2;
  const float2 rho = collide_pair<Q, S, CL, PACKED>(p, h, STATS ? &M2 : nullptr);
  if ((liveA && !(rho.x > 0.f && rho.x < 3.0e38f)) || (liveB && !(rho.y > 0.f && rho.y < 3.0e38f))) flag_unstable(p);
  if (STATS) pair_stats(M2, liveA, liveB, v);
  if (liveA && liveB) {
#pragma unroll
    for (int i = 0; i < Q; i++) st32(p, plane_ptr<S>(p, opp(i)) + cell, h[i]);
  } else {
#pragma unroll
    for (int i = 0; i < Q; i++)
      st16(p, plane_ptr<S>(p, opp(i)) + cell + (liveB ? 1 : 0), liveB ? h[i] >> 16 : h[i] & 0xffffu);
  }
}

template <int Q, class S, int CL>
__device__ __noinline__ void list_cell(const KParams& p, long long t);

#ifndef LBM_H2_MINB
#define LBM_H2_MINB 7
#endif
// STATS: also write the plane statistics of the state this step starts from (warp slot
// blockIdx.x of each row, ceil(nxp/64) slots per row).
// LAST (split step of odd rows with a periodic x seam): the row's last cell is an interior cell and
// the first of its pair, and its sources with c_x = -1 wrap.  A form of its own, as the two selects cost
// the even rows 1 % (1024x512x512 D3Q19 FP16, ten steps and moments 41.55 -> 41.97 ms).
template <int Q, class S, int CL, int LOAD, int STORE, bool STATS = false, bool SPLIT = false, bool LAST = false>
__global__ void __launch_bounds__(128, Q == 27 ? LBM_H2_MINB27 : LBM_H2_MINB) k_step_h2(const __grid_constant__ KParams p) {
  static_assert(sizeof(S) == 2, "two 16-bit populations per word");
  chain_begin();
  if constexpr (SPLIT) {
    // blocks past the last z plane take the listed cells, 128 per block: they follow the pair
    // blocks in launch order and fill the SMs the pair grid's tail leaves idle
    if (blockIdx.z >= (unsigned)p.nz) {
      const long long b = ((long long)(blockIdx.z - p.nz) * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
      list_cell<Q, S, CL>(p, b * 128 + threadIdx.y * 32 + threadIdx.x);
      return;
    }
  }
  const int x = 2 * (blockIdx.x * 32 + threadIdx.x);
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z;
  if (y >= p.ny) return;  // whole warp
  const int cell = cidx(p, x, y, z);
  // (the gather issued with the class load instead of after it: D3Q19 FP16 channel 501 -> 506 us,
  // D3Q27 FP16 tunnel 2466 -> 2488 us)
  int ca_ = CLS_SKIP, cb_ = CLS_SKIP;
  if (x < p.nx) {
    const unsigned c2 = chk(p, p.cls + cell, 2, CHK_CLS) ? *reinterpret_cast<const unsigned short*>(p.cls + cell) : 0x0202u;
    ca_ = c2 & 0xff;
    cb_ = x + 1 < p.nx ? (int)(c2 >> 8) : CLS_SKIP;
  }
  const int clsA = ca_ & CLS_MASK, clsB = cb_ & CLS_MASK;
  const bool xfA = ca_ & CLS_XFACE, xfB = cb_ & CLS_XFACE;
  const bool fast = LOAD == 0 ? ((clsA == CLS_INTERIOR || clsA == CLS_WRAP) && (clsB == CLS_INTERIOR || clsB == CLS_WRAP))
                              : (clsA == CLS_INTERIOR && clsB == CLS_INTERIOR);
  float v[NSTAT];
#pragma unroll
  for (int k = 0; k < NSTAT; k++) v[k] = 0.f;
  if constexpr (STORE == 2) {
    pair_pull<Q, S, CL, LOAD, STATS, SPLIT, LAST>(p, x, y, z, cell, clsA, clsB, fast, v, xfA, xfB);
  } else if constexpr (LOAD == 0) {
    pair_even<Q, S, CL, STATS>(p, x, cell, clsA, clsB, v);
  } else if (__all_sync(0xffffffffu, fast)) {
    // AA odd, all lanes interior: gather, and store back into the slots the gather read
    uint32_t h[Q];
#pragma unroll
    for (int i = 0; i < Q; i++) {
      const S* base = static_cast<const S*>(p.ga[i]);
      if (cx(i) == 0) {
        h[i] = ld32(p, base + cell);
      } else {
        int a, b;
        xsrc(cx(i), p, x, cell, a, b);
        const uint32_t lo = ld16(p, base + a);
        const uint32_t hi = ld16(p, base + b);
        h[i] = lo | (hi << 16);
      }
    }
    Macro<float2> M2;
    const float2 rho = collide_pair<Q, S, CL, false>(p, h, STATS ? &M2 : nullptr);
    if (STATS) pair_stats(M2, true, true, v);
    if (!(rho.x > 0.f && rho.x < 3.0e38f) || !(rho.y > 0.f && rho.y < 3.0e38f)) flag_unstable(p);
#pragma unroll
    for (int i = 0; i < Q; i++) {  // the slots of direction i take f*_opp(i)
      S* base = static_cast<S*>(p.ga[i]);
      const uint32_t w = h[opp(i)];
      if (cx(i) == 0) {
        st32(p, base + cell, w);
      } else {
        int a, b;
        xsrc(cx(i), p, x, cell, a, b);
        st16(p, base + a, w & 0xffffu);
        st16(p, base + b, w >> 16);
      }
    }
  } else {
    pair_fallback<Q, S, CL, LOAD, STORE, STATS>(p, x, y, z, cell, clsA, clsB, v);
  }
  if (STATS) stat_warp_store(p, y, z, blockIdx.x, (p.nxp + 63) / 64, v);
}

// ---- fields of the current state, half storage -----------------------------------------------
// rho and u of two x-adjacent cells per thread (the one-cell export's values): packed loads, both
// cells' sums in the FP32x2 pipe, 64-bit stores where the arrays and rows allow them (vec).
// Bound by HBM and latency; one cell per thread moved 64 bytes per load
// and warp.  1024x512x512 D3Q19 FP16 pull 3513 -> 2660 us, 375x190x187 FP16 AA tunnel 157 -> 121 us.
template <int Q, class S, int PAR>
__global__ void __launch_bounds__(128, Q == 27 ? 6 : 8) k_moments_h2(const __grid_constant__ KParams p, ExportArgs a, int vec) {
  const int x = 2 * (blockIdx.x * 32 + threadIdx.x);
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z;
  if (y >= p.ny) return;  // whole warp
  const int cell = cidx(p, x, y, z);
  uint32_t h[Q];
#pragma unroll
  for (int i = 0; i < Q; i++) h[i] = 0;
  // own slots of any cell, or the gather of a pair off the faces: in bounds whatever the classes, so
  // in flight with the class load below
  const bool early = PAR == 0 ? x < p.nx
                              : x >= 1 && x + 1 < p.nx - 1 && y >= 1 && y < p.ny - 1 && z >= 1 && z < p.nz - 1;
  if (early) pair_loads<Q, S, PAR>(p, x, cell, h);
  int ca = CLS_SKIP, cb = CLS_SKIP;
  if (x < p.nx) {
    const unsigned c2 = chk(p, p.cls + cell, 2, CHK_CLS) ? *reinterpret_cast<const unsigned short*>(p.cls + cell) : 0x0202u;
    ca = c2 & 0xff;
    cb = x + 1 < p.nx ? (int)(c2 >> 8) : CLS_SKIP;
  }
  const bool liveA = (ca & CLS_MASK) != CLS_SKIP, liveB = (cb & CLS_MASK) != CLS_SKIP;
  unsigned oa = 0, ob = 0;
  if (PAR == 0) {
    own_outflow_masks<Q>(p, x, cell, ca & CLS_MASK, cb & CLS_MASK, oa, ob);
  } else if ((ca & CLS_MASK) == CLS_INTERIOR && (cb & CLS_MASK) == CLS_INTERIOR) {
    if (!early) pair_loads<Q, S, PAR>(p, x, cell, h);
  } else if (liveA || liveB) {
    uint32_t hs[Q];
    load_pair_rules<Q, S, PAR>(p, x, y, z, cell, ca, cb, hs, &oa, &ob);
#pragma unroll
    for (int i = 0; i < Q; i++) h[i] = hs[i];
  }
  outflow_fix_packed<Q>(p, 64 * blockIdx.x, h, oa, ob);
  if (x >= p.nx) return;
  PackedPops<Q, S> pops{h};
  const Macro<float2> M = macro_acc<Q, false, float2>(p, pops);
  const long long dense = ((long long)z * p.ny + y) * p.nx + x;
  const long long N = (long long)p.nx * p.ny * p.nz;
  auto put = [&](float* out, float2 v) {
    v.x = liveA ? v.x : 0.f;
    v.y = liveB ? v.y : 0.f;
    if (vec) {
      *reinterpret_cast<float2*>(out + dense) = v;
    } else {
      out[dense] = v.x;
      if (x + 1 < p.nx) out[dense + 1] = v.y;
    }
  };
  if (a.rho) put(a.rho, M.rho);
  if (a.u) {
    put(a.u, M.ux);
    put(a.u + N, M.uy);
    put(a.u + 2 * N, M.uz);
  }
}

// ---- the listed cells of a split pull step ---------------------------------------------------
// A listed cell reads each incoming population through a table built with the list: for
// direction i, the cell the value is read from and a code byte holding the plane (bits 0-4),
// LT_INFLOW (the moving-wall term is added and the sum rounded to the storage precision, as
// for a bounce-back from a moving wall) or LT_ZERO (the value is 0).  The entry is what
// load_state of the gather step and its zero-gradient outflow copy read.
constexpr int LT_INFLOW = 0x40, LT_ZERO = 0x80;

// The table entry of direction i of the cell at `cell` with class cls and rule word r; false
// (and no entry) for a zero-gradient outflow copy, which reads what the upstream cell receives.
__device__ inline bool list_source_at(const KParams& p, int x, int y, int z, int cell, int cls, unsigned long long r,
                                      int i, int& src, int& code) {
  src = cell;
  code = LT_ZERO;
  if (cls == CLS_SKIP) return true;  // the upstream cell of an outflow copy is not fluid: 0
  Nbr nb;
  nb.init(p, x, y, z);
  src = nb.src(p, i);
  code = i;
  if (cls == CLS_INTERIOR || cls == CLS_WRAP) return true;
  const int k = (int)((r >> (2 * i)) & 3);
  if (k == R_STREAM) return true;
  if (k == R_SPECIAL) {
    int pl, ce;
    if (resolve_special(p, x, y, z, i, pl, ce) == K_OUTCOPY) return false;
    src = ce;
    code = opp(pl);
    return true;
  }
  src = cell;  // bounce-back from the own cell (moving wall: plus the inflow term)
  code = opp(i) | (k == R_INFLOW ? LT_INFLOW : 0);
  return true;
}

// The table entry of direction i of a listed cell (set-up): an outflow copy takes the entry of
// the upstream cell x - 1, which is never an outflow cell itself.
__device__ inline void list_source(const KParams& p, int x, int y, int z, int cell, int cls, unsigned long long r,
                                   int i, int& src, int& code) {
  if (list_source_at(p, x, y, z, cell, cls, r, i, src, code)) return;
  const int cu = cidx(p, x - 1, y, z);
  const int cl = cls_at(p, cu);
  if (!list_source_at(p, x - 1, y, z, cu, cl, cl == CLS_BOUNDARY ? rule_at(p, cu) : 0ull, i, src, code)) {
    src = cell;  // not reached (x - 1 is off the outflow face)
    code = LT_ZERO;
  }
}

// Listed cell t: loads through the table, the collision of the storage precision's form,
// own-cell store (the one-cell gather step's bits).
template <int Q, class S, int CL>
__device__ __noinline__ void list_cell(const KParams& p, long long t) {
  if (t >= p.nblist) return;
  const int cell = p.blist[t];
  const S* base = plane_ptr<S>(p, 0);
  float f[Q];
#pragma unroll
  for (int i = 0; i < Q; i++) {
    const long long e = i * p.nblist + t;
    const int src = p.bltab[e];
    const int code = p.blcode[e];
    float v = 0.f;
    if (!(code & LT_ZERO)) v = ldp<S>(p, base + (code & 31) * p.pstride + src);
    if (code & LT_INFLOW) v = rnd<S>(v + p.inflow_term[i]);
    f[i] = v;
  }
  const float rho = collide<Q, CL, float, acc_form<S>>(p, f, nullptr);
  if (!(rho > 0.f && rho < 3.0e38f)) flag_unstable(p);
  store_state<Q, S, 2>(p, 0, 0, 0, cell, CLS_BOUNDARY, f);
}

// The listed cells as a launch of their own (one per thread), for a long list: above 2^18 cells
// (it then runs at the list code's own occupancy rather than the x-pair kernel's), or too many
// blocks to follow the x-pair grid in its z dimension.
template <int Q, class S, int CL>
__global__ void __launch_bounds__(128) k_step_list(const __grid_constant__ KParams p) {
  chain_begin();
  list_cell<Q, S, CL>(p, blockIdx.x * 128ll + threadIdx.x);
}

}  // namespace lbm
