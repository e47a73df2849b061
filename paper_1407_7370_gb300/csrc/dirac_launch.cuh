// dirac_launch.cuh -- launchers of the pass kernels of dirac_kernels.cuh, shared
// by the units that instantiate them (FP32: dirac_capi.cu, FP64: dirac_step.cu).
#pragma once
#include "dirac_internal.h"
#include "dirac_kernels.cuh"

#include <algorithm>

namespace dirac {

// Persistent launch: as many CTAs as are resident at once (at most one per
// tile), each taking a contiguous chunk of the tile list whose size differs
// from the others' by at most one tile.
template <class S, int R, int TH, bool D, bool V, bool AY>
cudaError_t launch_pass_t(LaunchParams p, const LaunchShape& ls, cudaStream_t s) {
  static std::atomic<int> occ_dev[OCC_MAX_DEVICES];
  constexpr int NT = sub_workers<S>() * 32 * (TH / rows_per_thread<S, TH>());
  constexpr size_t smem = dyn_smem_bytes<S, R, TH, sub_workers<S>()>();
  int occ = 0;
  cudaError_t e = occupancy_on_device(occ_dev, lanczos_pass<S, R, TH, D, V, AY>, NT, smem, &occ);
  if (e != cudaSuccess) return e;
  if (occ < 1) occ = 1;
  const int per_sm = ls.cta_cap > 0 ? std::min(occ, ls.cta_cap) : occ;
  const int slots = std::max(1, ls.n_sm * per_sm);
  const int grid = std::max(1, std::min(p.total_tiles, slots));
  p.chunk_q = p.total_tiles / grid;
  p.chunk_r = p.total_tiles % grid;
  p.async_tiles = p.chunk_q >= ASYNC_MIN_TILES;
  return launch_pdl(lanczos_pass<S, R, TH, D, V, AY>, grid, NT, smem, s, p);
}

// Multiply-add FP64: a kernel without the c A_y terms (four FMAs per site of
// ~54) when no step of the launch has A_y != 0 (linear polarisation along x,
// static fields); the FP32 pass, bound by memory, keeps one kernel
template <class S, int R, int TH, bool D, bool V>
cudaError_t launch_pass_ay(const LaunchParams& p, const LaunchShape& ls, cudaStream_t s) {
  if constexpr (sizeof(S) == sizeof(double)) {
    if (!p.has_ay) return launch_pass_t<S, R, TH, D, V, false>(p, ls, s);
  }
  return launch_pass_t<S, R, TH, D, V, true>(p, ls, s);
}

template <class S, int TH>
cudaError_t launch_pass_s(int order, bool diri, bool hasv, const LaunchParams& p, const LaunchShape& ls,
                          cudaStream_t s) {
  if (order == 2) {
    if (diri) return hasv ? launch_pass_ay<S, 1, TH, true, true>(p, ls, s) : launch_pass_ay<S, 1, TH, true, false>(p, ls, s);
    return hasv ? launch_pass_ay<S, 1, TH, false, true>(p, ls, s) : launch_pass_ay<S, 1, TH, false, false>(p, ls, s);
  }
  if (diri) return hasv ? launch_pass_ay<S, 2, TH, true, true>(p, ls, s) : launch_pass_ay<S, 2, TH, true, false>(p, ls, s);
  return hasv ? launch_pass_ay<S, 2, TH, false, true>(p, ls, s) : launch_pass_ay<S, 2, TH, false, false>(p, ls, s);
}

}  // namespace dirac
