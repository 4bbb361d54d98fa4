// kern_inst.cu -- instantiates the kernels and launchers for one (stencil, precision) pair.
// Compiled once per pair with -DLBM_Q=19|27 and -DLBM_S=float|__half|__nv_bfloat16.
#include <algorithm>
#include <type_traits>

#include "lbm_launch.cuh"

#ifndef LBM_Q
#error "LBM_Q must be defined"
#endif
#ifndef LBM_S
#error "LBM_S must be defined"
#endif

namespace lbm {

// stats: also write the warp-slot plane statistics of the starting state (p.stats_w); *nws
// receives the number of warp slots per row.  coll: 0 TRT, 1 MRT (D3Q19, one cell per thread),
// 2 regularised (one cell per thread).
// listed cells up to which a split step runs them in its x-pair grid
#ifndef LBM_LIST_FUSE_MAX
#define LBM_LIST_FUSE_MAX (1ll << 18)
#endif

// The odd AA step of half storage, D3Q19: x-pairs or one cell per thread.  A pair warp with a lane
// at an odd row end runs 3.4 times as long as a clean one, with an inflow, outflow or wall lane 6
// times, and one cell per thread costs 1.22 times the clean pairs: pairs for rows of at least 11
// pair warps per odd end and 23 per face.  FP16, us, pairs / one cell: 512x256x128 channel 282 /
// 346, 256x130x121 91 / 98, 251x130x121 106 / 100, 375x190x187 tunnel 597 / 297.
static bool odd_pairs(const KParams& p) {
  const int faces = (p.face[0] != FACE_PERIODIC) + (p.face[1] != FACE_PERIODIC);
  return (p.nxp + 63) / 64 >= 11 * (p.nx & 1) + 23 * faces;
}

// Step launches are chained (programmatic stream serialisation), in graph replays only where the grid
// takes about a wave of blocks or more, 8 per SM of the one-cell kernel, 6 of the pairs (D3Q27: 3).  Below, the
// blocks of a chained step find free places on every SM beside those of the step before, and its last
// ones go where these end first, so that SMs end up with uneven shares; launched one by one such steps
// wait for the host anyhow (2:1 refined box 64x32x32 FP16 with nine launches 31.7 us chained, 33-35
// not).  Replays, us a step, chained / not: D3Q19 FP32 AA box 64x50x46 (1196 blocks) 5.4 / 4.9, channel
// 32x80x90 (1800) 9.8 / 9.9; D3Q27 FP32 32x50x60 (780) AA box 6.1 / 5.0, pull channel 13.0 / 10.8; FP16
// pull pairs 64x50x46 (598) 6.2 / 5.9, 128x48x48 (1152) 8.5 / 8.7, D3Q27 64x40x38 (380) 7.9 / 7.7,
// 100x40x30 (600) 8.5 / 9.0.
static void launch_step_grid(void (*kern)(KParams), dim3 g, const Launch& L, int wave, const KParams& p) {
  const bool chain = !L.replay || (long long)g.x * g.y * g.z > (long long)wave * L.nsm;
  launch_chained(chain, kern, g, L.block, L.stream, p);
}
constexpr int WAVE_CELLS = 8, WAVE_PAIRS = LBM_Q == 27 ? 3 : 6;

template <int Q, class S, int LOAD, int STORE, bool STATS>
static void step_mode_s(const KParams& p, int closure, const Launch& L, int coll, int* nws) {
  if constexpr (Q == 19) {
    if (coll == 1) {
      if (nws) *nws = p.nxp / 32;
      if (closure == CL_NONE) launch_step_grid(k_step<Q, S, CL_NONE, LOAD, STORE, STATS, 1>, L.grid, L, WAVE_CELLS, p);
      else launch_step_grid(k_step<Q, S, CL_SMAG, LOAD, STORE, STATS, 1>, L.grid, L, WAVE_CELLS, p);
      return;
    }
  }
  if (coll == 2) {  // regularised collision: one cell per thread, every stencil and storage
    if (nws) *nws = p.nxp / 32;
    if (closure == CL_NONE) launch_step_grid(k_step<Q, S, CL_NONE, LOAD, STORE, STATS, 2>, L.grid, L, WAVE_CELLS, p);
    else launch_step_grid(k_step<Q, S, CL_SMAG, LOAD, STORE, STATS, 2>, L.grid, L, WAVE_CELLS, p);
    return;
  }
  // half storage, gather step of two-grid pull without statistics (both stencils; D3Q19 unless
  // built with LBM_SPLIT19=0): the x-pair step over the interior cells (populations packed in
  // registers through the collision for D3Q27) and the cells the handle listed (rules, wraps):
  // a short list in extra z slices of the pair grid (no launch of its own: the 2:1 refined box's
  // small FP16 lattices 69.5 -> 71.9 % of the copy bandwidth), a long one as k_step_list at its
  // own occupancy (the D3Q27 bluff body's 1.5 M listed cells: 74.6 % against 73.0 % in the pair
  // grid, whose 95 registers leave fewer warps for the latency-bound list).  The other D3Q27
  // pull steps (first after an import, statistics samples) take the one-cell kernel.
  if constexpr (sizeof(S) == 2 && (Q == 27 || LBM_SPLIT19) && LOAD == 2 && STORE == 2 && !STATS) {
    if (p.split && coll == 0) {
      dim3 g = L.grid;
      g.x = (p.nxp + 63) / 64;
      const long long per = 128ll * g.x * g.y;  // listed cells per extra z slice
      const long long extra = (p.nblist + per - 1) / per;
      const bool fused = p.nblist <= LBM_LIST_FUSE_MAX && g.z + extra <= 65535;
      if (fused) g.z += (unsigned)extra;
      if (p.nx % 2 && p.face[1] == FACE_PERIODIC) {
        if (closure == CL_NONE) launch_step_grid(k_step_h2<Q, S, CL_NONE, 2, 2, false, true, true>, g, L, WAVE_PAIRS, p);
        else launch_step_grid(k_step_h2<Q, S, CL_SMAG, 2, 2, false, true, true>, g, L, WAVE_PAIRS, p);
      } else {
        if (closure == CL_NONE) launch_step_grid(k_step_h2<Q, S, CL_NONE, 2, 2, false, true>, g, L, WAVE_PAIRS, p);
        else launch_step_grid(k_step_h2<Q, S, CL_SMAG, 2, 2, false, true>, g, L, WAVE_PAIRS, p);
      }
      if (!fused) {
        const unsigned nb = (unsigned)((p.nblist + 127) / 128);
        if (closure == CL_NONE) launch_chained(true, k_step_list<Q, S, CL_NONE>, nb, 128, L.stream, p);
        else launch_chained(true, k_step_list<Q, S, CL_SMAG>, nb, 128, L.stream, p);
      }
      return;
    }
  }
  // half storage: x-pairs, 64 x per warp; D3Q27 (the AA even step only, see above) for rows of more
  // than 32 cells and lattices of more than a wave of one-cell blocks: below, half the lanes idle or the
  // longer chain of a pair shows (graph replays of AA, us a step, pairs / one cell: channel 32x80x90
  // 12.9 / 12.1, 64x50x46 10.3 / 9.8, box 32x64x72 6.4 / 5.7, 17x60x60 5.7 / 4.9).
  const bool pairs27 = p.nxp > 32 && (long long)L.grid.x * L.grid.y * L.grid.z > (long long)WAVE_CELLS * L.nsm;
  if (sizeof(S) == 2 && (Q == 19 ? STORE != 1 || odd_pairs(p) : STORE == 0 && pairs27)) {
    if constexpr (sizeof(S) == 2 && (Q == 19 || STORE == 0)) {
      dim3 g = L.grid;
      g.x = (p.nxp + 63) / 64;
      if (nws) *nws = (int)g.x;
      if (closure == CL_NONE) launch_step_grid(k_step_h2<Q, S, CL_NONE, LOAD, STORE, STATS>, g, L, WAVE_PAIRS, p);
      else launch_step_grid(k_step_h2<Q, S, CL_SMAG, LOAD, STORE, STATS>, g, L, WAVE_PAIRS, p);
      return;
    }
  }
  if (nws) *nws = p.nxp / 32;
  if (closure == CL_NONE) launch_step_grid(k_step<Q, S, CL_NONE, LOAD, STORE, STATS>, L.grid, L, WAVE_CELLS, p);
  else launch_step_grid(k_step<Q, S, CL_SMAG, LOAD, STORE, STATS>, L.grid, L, WAVE_CELLS, p);
}

template <int Q, class S, int LOAD, int STORE>
static void step_mode(const KParams& p, int closure, const Launch& L, bool stats, int coll, int* nws) {
  if (stats) step_mode_s<Q, S, LOAD, STORE, true>(p, closure, L, coll, nws);
  else step_mode_s<Q, S, LOAD, STORE, false>(p, closure, L, coll, nws);
}

// mode: 0 AA even, 1 AA odd, 2 first pull step after an import, 3 pull step
template <int Q, class S>
cudaError_t launch_step(const KParams& p, int closure, int mode, const Launch& L, bool stats, int* nws, int coll) {
  switch (mode) {
    case 0: step_mode<Q, S, 0, 0>(p, closure, L, stats, coll, nws); break;
    case 1: step_mode<Q, S, 1, 1>(p, closure, L, stats, coll, nws); break;
    case 2: step_mode<Q, S, 0, 2>(p, closure, L, stats, coll, nws); break;
    default: step_mode<Q, S, 2, 2>(p, closure, L, stats, coll, nws); break;
  }
  return cudaGetLastError();
}

// nsteps plain steps in one cooperative launch (k_step_multi): pull alternates p0 and p1, AA
// alternates the even and odd forms on p0 starting with `odd0`.  The fewest blocks per SM that give
// every SM the same share of the row segments in as few passes as the resident warps allow (blocks of
// 16 warps throughout left 36 of 152 SMs two blocks and the others one for 3,000 segments: 32x50x60
// D3Q19 FP32 pull channel 5.9 -> 4.7 us a step, AA box 5.2 -> 3.9, 64x64x64 pull channel 10.8 -> 9.1); the
// grid is at most what fits on the device at once (a cooperative launch refuses more, it never waits).
template <int Q, class S, int CL, int COLL, bool AA>
static cudaError_t multi_one(const KParams2& pp, int nsteps, int odd0, unsigned* count, int* alarm, cudaStream_t stream, int nsm) {
  auto kern = k_step_multi<Q, S, CL, COLL, AA>;
  const KParams& p = pp.p[0];
  const long long nseg = (long long)(p.nxp / 32) * p.ny * p.nz;
  const long long passes = (nseg + multi_cap<Q>(nsm) - 1) / multi_cap<Q>(nsm);
  const int share = (int)((nseg + passes * nsm - 1) / (passes * nsm));  // warps per SM
  const int per = (share + MULTI_WARPS<Q> - 1) / MULTI_WARPS<Q>;        // blocks per SM
  const int warps = (share + per - 1) / per;
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * warps, 0);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorCooperativeLaunchTooLarge;
  const int blocks = (int)std::min<long long>((nseg + warps - 1) / warps, (long long)std::min(per, per_sm) * nsm);
  e = cudaMemsetAsync(count, 0, sizeof(unsigned), stream);
  if (e != cudaSuccess) return e;
  void* args[] = {(void*)&pp, (void*)&nsteps, (void*)&odd0, (void*)&count, (void*)&alarm};
  return cudaLaunchCooperativeKernel((const void*)kern, dim3(blocks), dim3(32, warps), args, 0, stream);
}

template <int Q, class S, int COLL, bool AA>
static cudaError_t multi_cl(const KParams2& pp, int closure, int nsteps, int odd0, unsigned* count, int* alarm, cudaStream_t st,
                            int nsm) {
  return closure == CL_NONE ? multi_one<Q, S, CL_NONE, COLL, AA>(pp, nsteps, odd0, count, alarm, st, nsm)
                            : multi_one<Q, S, CL_SMAG, COLL, AA>(pp, nsteps, odd0, count, alarm, st, nsm);
}

template <int Q, class S, bool AA>
static cudaError_t multi_coll(const KParams2& pp, int closure, int coll, int nsteps, int odd0, unsigned* count,
                              int* alarm, cudaStream_t st, int nsm) {
  if constexpr (Q == 19) {
    if (coll == 1) return multi_cl<Q, S, 1, AA>(pp, closure, nsteps, odd0, count, alarm, st, nsm);
  }
  if (coll == 2) return multi_cl<Q, S, 2, AA>(pp, closure, nsteps, odd0, count, alarm, st, nsm);
  return multi_cl<Q, S, 0, AA>(pp, closure, nsteps, odd0, count, alarm, st, nsm);
}

template <int Q, class S>
cudaError_t launch_step_multi(const KParams& p0, const KParams& p1, int closure, int coll, bool aa, int odd0,
                              int nsteps, unsigned* count, int* alarm, cudaStream_t stream, int nsm) {
  KParams2 pp;
  pp.p[0] = p0;
  pp.p[1] = p1;
  return aa ? multi_coll<Q, S, true>(pp, closure, coll, nsteps, odd0, count, alarm, stream, nsm)
            : multi_coll<Q, S, false>(pp, closure, coll, nsteps, odd0, count, alarm, stream, nsm);
}

template <int Q, class S, int LOAD, int STORE>
static cudaError_t mlp_one(const KParams& p, cudaStream_t stream, int nsm) {
  constexpr int smem = (int)sizeof(MlpSmem);
  auto kern = k_step_mlp<Q, S, LOAD, STORE>;
  static int blocks_per_sm = 0;  // per instantiation, found once (one: the kernel allocates TMEM)
  if (blocks_per_sm == 0) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks_per_sm, kern, 128 * MLP_NG, smem);
    if (e != cudaSuccess) return e;
    if (blocks_per_sm < 1) blocks_per_sm = 1;
  }
  const long long ntiles = (long long)(p.nxp / 32) * ((p.ny + 3) / 4) * p.nz;
  if (ntiles >= (1ll << 31)) return cudaErrorInvalidValue;  // tile indices are 32-bit in the kernel
  const long long groups = (ntiles + MLP_NG - 1) / MLP_NG;
  const long long grid = std::min<long long>(groups, (long long)nsm * blocks_per_sm);
  kern<<<(unsigned)grid, dim3(32, 4 * MLP_NG, 1), smem, stream>>>(p, ntiles);
  return cudaGetLastError();
}

// The step with the learned closure (tensor-core hidden layer); mode as in launch_step.
template <int Q, class S>
cudaError_t launch_step_mlp(const KParams& p, int mode, cudaStream_t stream, int nsm) {
  switch (mode) {
    case 0: return mlp_one<Q, S, 0, 0>(p, stream, nsm);
    case 1: return mlp_one<Q, S, 1, 1>(p, stream, nsm);
    case 2: return mlp_one<Q, S, 0, 2>(p, stream, nsm);
    default: return mlp_one<Q, S, 2, 2>(p, stream, nsm);
  }
}

// Blocks of k_row_sums.  EX_SUM: one wave of what is resident (8 per SM), in gathered layouts of more
// rows two (768x192x192 FP16 D3Q27 tunnel 830 -> 743 us; 96x64x48 channel 36 -> 43 us).  EX_STATS: at least four
// times as many, in gathered layouts of at most ROWS_MAX rows, since a block's rows are all of one plane
// and those of a wall plane take several times as long (256x128x130 channel: 111 us with one wave; four take 25 us
// off a pass of two steps, sums, statistics and exports).
constexpr int ROW_BLOCKS_SM = 8, ROWS_MAX = 4;

template <int Q, class S, int PAR>
static void export_par(const KParams& p, int mode, const ExportArgs& a, const Launch& L) {
  switch (mode) {
    case EX_POP: k_export<Q, S, PAR, EX_POP><<<L.grid, L.block, 0, L.stream>>>(p, a); break;
    case EX_MOM:
      // half storage: two cells per thread (64-bit stores need even rows and 8-byte aligned arrays),
      // D3Q27 in natural layout only: gathered, its 80 registers cost more than the pairs give
      // (FP16 512x256x128 AA after an even step 253 -> 179 us, pull 283 us against 303); gathered D3Q19
      // above a hundred one-cell blocks per SM: below, the lanes with boundary cells, loaded out of line,
      // make the launch (pull channel, pairs / one cell: 64x32x32 12.9 / 8.5, 128x128x100 (12,800 blocks)
      // 32-33 / 32, 192x128x100 (19,200) 44.4 / 45.9, 256x200x200 126 / 145)
      if constexpr (sizeof(S) == 2 && (Q == 19 || PAR == 0)) {
        if (PAR == 0 || (long long)L.grid.x * L.grid.y * L.grid.z > 100ll * L.nsm) {
          const int vec = p.nx % 2 == 0 && (uintptr_t)a.rho % 8 == 0 && (uintptr_t)a.u % 8 == 0;
          k_moments_h2<Q, S, PAR><<<dim3((p.nxp + 63) / 64, L.grid.y, L.grid.z), L.block, 0, L.stream>>>(p, a, vec);
          break;
        }
      }
      k_export<Q, S, PAR, EX_MOM><<<L.grid, L.block, 0, L.stream>>>(p, a);
      break;
    case EX_SUM: {
      const int rows = p.ny * p.nz, wave = ROW_BLOCKS_SM * L.nsm;
      const int want = PAR != 0 && rows >= 4 * wave ? 2 * wave : wave, cnt = (rows + want - 1) / want;
      const int nblk = (rows + cnt - 1) / cnt;
      k_row_sums<Q, S, PAR, EX_SUM><<<(unsigned)nblk, ROW_THREADS, 0, L.stream>>>(p, cnt, a.partial);
      k_row_total<EX_SUM><<<1, 256, 0, L.stream>>>(a.partial, p.ny, nblk, a.sums);
      break;
    }
    default: {
      const int least = PAR == 0 ? 1 : (p.nz + ROWS_MAX - 1) / ROWS_MAX;
      const int per = std::max(least, 4 * ROW_BLOCKS_SM * L.nsm / p.ny);  // blocks per plane
      const int cnt = (p.nz + per - 1) / per, nblk = (p.nz + cnt - 1) / cnt * p.ny;
      k_row_sums<Q, S, PAR, EX_STATS><<<(unsigned)nblk, ROW_THREADS, 0, L.stream>>>(p, cnt, a.partial);
      k_row_total<EX_STATS><<<(unsigned)p.ny, 256, 0, L.stream>>>(a.partial, p.ny, nblk, a.sums);
      break;
    }
  }
}

template <int Q, class S>
cudaError_t launch_export(const KParams& p, int parity, int mode, const ExportArgs& a, const Launch& L) {
  if (parity == 0) export_par<Q, S, 0>(p, mode, a, L);
  else if (parity == 1) export_par<Q, S, 1>(p, mode, a, L);
  else export_par<Q, S, 2>(p, mode, a, L);
  return cudaGetLastError();
}

template <int Q, class S>
cudaError_t launch_init_eq(const KParams& p, const float* rho, const float* u, const Launch& L) {
  k_init_eq<Q, S><<<L.grid, L.block, 0, L.stream>>>(p, rho, u);
  return cudaGetLastError();
}

template <int Q, class S>
cudaError_t launch_set_pop(const KParams& p, const float* df, const Launch& L) {
  k_set_pop<Q, S><<<L.grid, L.block, 0, L.stream>>>(p, df);
  return cudaGetLastError();
}

template cudaError_t launch_step<LBM_Q, LBM_S>(const KParams&, int, int, const Launch&, bool, int*, int);
template cudaError_t launch_step_mlp<LBM_Q, LBM_S>(const KParams&, int, cudaStream_t, int);
template cudaError_t launch_export<LBM_Q, LBM_S>(const KParams&, int, int, const ExportArgs&, const Launch&);
template cudaError_t launch_init_eq<LBM_Q, LBM_S>(const KParams&, const float*, const float*, const Launch&);
template cudaError_t launch_set_pop<LBM_Q, LBM_S>(const KParams&, const float*, const Launch&);
template cudaError_t launch_step_multi<LBM_Q, LBM_S>(const KParams&, const KParams&, int, int, bool, int, int,
                                                     unsigned*, int*, cudaStream_t, int);

}  // namespace lbm
