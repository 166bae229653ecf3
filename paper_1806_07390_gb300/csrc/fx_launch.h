// Launch entry points of the stage kernel instantiations (one translation unit per precision and
// dimension, compiled in parallel).
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "fx_couple.cuh"
#include "fx_couple64.cuh"
#include "fx_stage.cuh"
#include "fx_vterms.cuh"
#include "fx_ye.cuh"

namespace fx {

constexpr int STAGE_SMEM_MAX = 200 * 1024;  // most dynamic shared memory of a stage kernel block

// Tile and march chunk of the stage kernel for a grid, fitted to the device.  A model of its time
// over every tile that the kernel's capacities allow and every chunk length picks the least:
//   waves x ((chunk + 2) x (time of one plane) + start), two planes being the prologue's share,
// where a fractional number of waves x costs x + 0.9 (ceil x - x) / ceil x (fitted to measured
// chunks: multiprocessors that finish early idle, the others run faster with fewer blocks).
// A plane's time on a multiprocessor with r resident blocks joins (root of squares) what one block
// alone takes (in FP32 a warp issues about every sixth cycle; in FP64 its chain of 16-cycle operations,
// nearly as long for one block as for two) and the issue of the r blocks' instructions.  The
// instruction counts are per warp and plane, from the kernel's operation counts: they only rank
// tiles against each other.  So small grids get small tiles and short chunks that spread over the
// device, and large ones the tiles with the least halo share and the fewest idle lanes.  Measured
// against a sweep of tiles and chunks (stage kernel, microseconds, chosen / best of the sweep):
// 1024^2 x 16 FP32 253 / 245, 640 x 128 x 20 spherical FP32 70 / 70, 96 x 80 x 8 FP32 10.9 / 10.5,
// 512^2 x 16 FP64 1862 / 1862; with blocks of up to 192 threads in 3-d 256^3 x 12 FP32 7140 / 7140,
// 75 x 61 x 50 x 20 FP32 250 / 243 (blocks of 256: 6235 and 166, see StageCap).
template <class R, int D>
inline void fit_tile(const int* n, int G, int nsm, int regs, RadTile& best, int& chunk) {
  using C = StageCap<R, D>;
  constexpr int W = LaneOf<R>::W;
  constexpr int NRV = 1 + D;
  const int gl = (G + W - 1) / W;
  const double recon = 12.0 * NRV + 3.0, flux = 64.0 + 5.0 * NRV, own = D * (recon + flux) + NRV * 30.0 + 60.0;
  const double alone = sizeof(R) == 8 ? own * 155.0 : own / 0.16 + 800.0, IPC = sizeof(R) == 8 ? 0.097 : 2.6;
  double least = 1e300;
  best = RadTile{};
  const int nm = D >= 2 ? n[D - 1] : 1;
  for (int ty = D == 3 ? 16 : 1; ty >= 1; --ty) {
    for (int tx = 1; tx * ty * gl <= C::NT; ++tx) {
      if (ty * gl > C::XP || (D == 3 && tx * gl > C::XP) || tx > n[0] + 3) continue;
      RadTile t{};
      t.tx = tx; t.ty = ty; t.gl = gl;
      t.nth = (tx * ty * gl + 31) / 32 * 32;
      t.ntx = (n[0] + tx - 1) / tx;
      t.nty = D == 3 ? (n[1] + ty - 1) / ty : 1;
      // upper faces: at most one per thread; in 1-d and 2-d also one halo reconstruction, one halo
      // copy and two records
      const int nt = (ty + (D == 3 ? tx : 0)) * gl;
      if (nt > t.nth || (D < 3 && (4 * gl > t.nth || 8 * gl > C::NT || tile_recs<D>(t) > 2 * t.nth))) continue;
      // copies past the ones whose offsets a thread keeps
      const int late = std::max(0, tile_halo<D>(t) * gl - (D == 3 ? 2 : 1) * t.nth) + std::max(0, tile_recs<D>(t) - 2 * t.nth);
      const size_t smem = stage_smem_bytes<R, D>(t);
      if (smem > STAGE_SMEM_MAX) continue;
      const int rmax = std::max(1, std::min({65536 / (regs * t.nth), (int)(227 * 1024 / (smem + 1024)), 2048 / t.nth, 32}));
      const double instr = t.nth / 32 * own + (2 * nt + 31) / 32 * (recon + 30.0) + (nt + 31) / 32 * (flux + 30.0) + (late + 31) / 32 * 60.0;
      const double tiles = (double)t.ntx * t.nty;
      // the shortest chunk of every count of chunks
      for (int c = std::min(nm, 160), m; c >= 1; --c) {
        m = (nm + c - 1) / c;
        c = (nm + m - 1) / m;
        const double blocks = tiles * m;
        const double r = std::min((double)rmax, std::ceil(blocks / nsm));
        const double issue = r * instr / IPC, plane = std::sqrt(alone * alone + issue * issue);
        const double x = blocks / (r * nsm), xc = std::ceil(x), w = x <= 1.0 ? 1.0 : x + 0.9 * (xc - x) / xc;
        const double cost = w * ((c + (D >= 2 ? 2.0 : 0.0)) * plane + 1500.0);
        if (cost <= least) {
          least = cost;
          best = t;
          chunk = c;
        }
      }
    }
  }
  // gas cells per thread: one on small grids, up to four where the gas blocks fill the device anyway
  double cells = 1.0;
  for (int d = 0; d < D; ++d) cells *= n[d];
  best.gpt = std::min(4, std::max(1, (int)(cells / (2048.0 * nsm))));
  best.mgl = (unsigned)(((1ull << 32) + gl - 1) / gl);
}

// Enqueue one stage (state type R, D dimensions, Newton/bookkeeping type NT; SPH: the 2-d
// spherical grid) on stream s: the gas face kernel, the radiation/update kernel, with the
// velocity-dependent terms on the velocity-term kernel, and with the interaction on the
// interaction kernel.  When non-null, `mid` is recorded after the face kernel and `mid2` after the
// radiation/update kernel (per-kernel timing).  Returns the CUDA error of the launches.
template <class R, int D, class NT, bool SPH>
cudaError_t launch_stage(const StageArgs<R>& a, cudaStream_t s, cudaEvent_t mid,
                         cudaEvent_t mid2);

// Registers per thread of the stage kernel (radiation reconstruction order ro), for fit_tile.
template <class R, int D, class NT, bool SPH>
cudaError_t stage_regs(int ro, int* regs);

#ifdef FX_LAUNCH_DEFINE
// Definition, included only by the per-instantiation translation units.  The group arithmetic
// type of the stage kernel is the state type R.
template <class R, int D, class NT, bool SPH>
cudaError_t launch_stage(const StageArgs<R>& a0, cudaStream_t s, cudaEvent_t mid, cudaEvent_t mid2) {
  if ((a0.g.geom != 0) != SPH) return cudaErrorInvalidValue;  // the grid's geometry decides SPH
  StageArgs<R> a = a0;
  // lanes copy and store pairs with 8-byte accesses where every pair is complete and aligned
  auto al8 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 7) == 0; };
  a.rt.vec = a.g.G % 2 == 0 && ((2 + D) * a.g.ncell) % 2 == 0 && al8(a.in) && al8(a.base) && al8(a.out);
  // (the boundary budgets are compiled into the kernel for grids with a non-periodic boundary;
  // the second-order radiation reconstruction always carries them)
  constexpr bool PV = sizeof(R) == 4 && D < 3;  // an instance for whole pairs
  auto kern = a.g.rad_order == 2 ? (a.rt.vec ? stage_kernel<R, D, SPH, 2, true, PV> : stage_kernel<R, D, SPH, 2, true, false>)
              : a.budget_bnd     ? (a.rt.vec ? stage_kernel<R, D, SPH, 1, true, PV> : stage_kernel<R, D, SPH, 1, true, false>)
                                 : (a.rt.vec ? stage_kernel<R, D, SPH, 1, false, PV> : stage_kernel<R, D, SPH, 1, false, false>);
  const size_t smem = stage_smem_bytes<R, D>(a.rt);
  // (a function's limit is the process's: it is set to the same value by every handle, the most that any
  // needs, so that handles of other threads cannot lower it between this call and the launch)
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, STAGE_SMEM_MAX);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                           cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return e;
  // gas faces first (same stream): fluxes and contact speeds of every face of every direction,
  // one block per tile of faces, one grid row per direction
  constexpr int FT = D == 3 ? FACE_THREADS_3D : FACE_THREADS;
  const bool small = face_small(a.g.n, D);
  unsigned ntmax = 0;
  for (int d = 0; d < D; ++d)
    ntmax = std::max(ntmax, small ? face_tiles<FACE_THREADS_SMALL>(a.g.n, D, d) : face_tiles<FT>(a.g.n, D, d));
  dim3 gg(ntmax, D, 1);
  if (a.sflag != nullptr) {  // carbuncle guard: shock flags of the stage input first
    shock_flag_kernel<R, D><<<(unsigned)((a.g.ncell + 255) / 256), 256, 0, s>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (small) gas_face_kernel<R, D, SPH, FACE_THREADS_SMALL><<<gg, FACE_THREADS_SMALL, 0, s>>>(a);
  else gas_face_kernel<R, D, SPH, FT><<<gg, FT, 0, s>>>(a);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (mid) {
    e = cudaEventRecord(mid, s);
    if (e != cudaSuccess) return e;
  }
  // radiation blocks (tiles across the fast axes, chunks of the slowest) and gas blocks
  a.rt.nrad = a.rt.ntx * a.rt.nty * (D >= 2 ? (a.g.n[D - 1] + a.chunk - 1) / a.chunk : 1);
  const int64_t ngas = (a.g.ncell + a.rt.gpt * a.rt.nth - 1) / (a.rt.gpt * a.rt.nth);
  kern<<<(unsigned)(a.rt.nrad + ngas), (unsigned)a.rt.nth, smem, s>>>(a);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (mid2) {
    e = cudaEventRecord(mid2, s);
    if (e != cudaSuccess) return e;
  }
  // the velocity-dependent radiation terms of the stage input, added to the explicit update
  // before the interaction
  if (a.g.vterms) {
    constexpr int W = LaneOf<R>::W;
    const int cells = VT_THREADS / 32 * (32 / ((a.g.G + W - 1) / W));  // cells of one x row per block
    const dim3 vg((unsigned)((a.g.n[1] * a.g.n[2] + VT_ROWS - 1) / VT_ROWS), (unsigned)((a.g.n[0] + cells - 1) / cells), 1);
    vterm_kernel<R, D, SPH><<<vg, VT_THREADS, 0, s>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  // three species: the composition's update, then the two-equation interaction (FP64 arithmetic)
  if (a.g.species > 1) {
    comp_kernel<R, D, SPH><<<(unsigned)((a.g.ncell + 255) / 256), 256, 0, s>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess || !a.g.couple) return e;
    const bool f32 = std::is_same<R, float>::value;
    const size_t cs = f32 ? couple_ye32_smem_bytes<D>(a.g.G) : couple_ye_smem_bytes(a.g.G);
    if constexpr (f32) {
      e = cudaFuncSetAttribute(couple_ye32_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)couple_ye32_smem_bytes<D>(MAXG));
      if (e != cudaSuccess) return e;
      couple_ye32_kernel<D><<<(unsigned)((a.g.ncell + CPL_THREADS - 1) / CPL_THREADS), CPL_THREADS, cs, s>>>(a);
    } else {
      e = cudaFuncSetAttribute(couple_ye_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)couple_ye_smem_bytes(MAXG));
      if (e != cudaSuccess) return e;
      couple_ye_kernel<D><<<(unsigned)((a.g.ncell + CPLYE_THREADS - 1) / CPLYE_THREADS), CPLYE_THREADS, cs, s>>>(a);
    }
    return cudaGetLastError();
  }
  // the interaction (FP32 state: couple_kernel, one thread per cell; FP64 state: couple64_kernel, 1 to 16)
  if (a.g.couple) {
    if constexpr (std::is_same<R, float>::value) {
      auto ck = couple_kernel<D, NT>;
      const size_t cs = couple_smem_bytes<D>(a.g.G);
      e = cudaFuncSetAttribute(ck, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)couple_smem_bytes<D>(MAXG));
      if (e != cudaSuccess) return e;
      const unsigned nb = (unsigned)((a.g.ncell + CPL_THREADS - 1) / CPL_THREADS);
      ck<<<nb, CPL_THREADS, cs, s>>>(a);
    } else {
      const int lanes = couple64_lanes(a.g.ncell, a.g.G), cells = CPL64_THREADS / lanes;
      auto ck = lanes == 1   ? couple64_kernel<D, 1>
                : lanes == 2 ? couple64_kernel<D, 2>
                : lanes == 4 ? couple64_kernel<D, 4>
                : lanes == 8 ? couple64_kernel<D, 8>
                             : couple64_kernel<D, 16>;
      const size_t cs = couple64_smem_bytes<D>(a.g.G, cells);
      e = cudaFuncSetAttribute(ck, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)couple64_smem_bytes<D>(MAXG, CPL64_THREADS));
      if (e != cudaSuccess) return e;
      ck<<<(unsigned)((a.g.ncell + cells - 1) / cells), CPL64_THREADS, cs, s>>>(a);
    }
    e = cudaGetLastError();
  }
  return e;
}

template <class R, int D, class NT, bool SPH>
cudaError_t stage_regs(int ro, int* regs) {
  cudaFuncAttributes fa;
  const cudaError_t e = ro == 2 ? cudaFuncGetAttributes(&fa, stage_kernel<R, D, SPH, 2, true, false>)
                                : cudaFuncGetAttributes(&fa, stage_kernel<R, D, SPH, 1, false, false>);
  if (e == cudaSuccess) *regs = fa.numRegs;
  return e;
}

#endif

}  // namespace fx
