// dirac_step64.cu -- launcher of the fixed-point FP64 one-launch time step
// (`lanczos_step64`), in a unit of its own so that it compiles in parallel with
// the per-pass kernels.
#include "dirac.h"
#include "dirac_internal.h"
#include "dirac_pass64.cuh"

#include <cuda_runtime.h>

#include <algorithm>

namespace dirac {

namespace {

template <int R, int TH, bool D, bool V, bool ISO>
cudaError_t launch_t(LaunchParams p, int n_sm, CoopArgs ca, cudaStream_t s) {
  static std::atomic<int> occ_dev[OCC_MAX_DEVICES];
  constexpr size_t smem = fx_smem_bytes<R, TH>();
  int occ = 0;
  cudaError_t e = occupancy_on_device(occ_dev, lanczos_step64<R, TH, D, V, ISO>, fx_threads<TH>(), smem, &occ);
  if (e != cudaSuccess) return e;
  if (occ < 1) return cudaErrorCooperativeLaunchTooLarge;
  // every CTA resident (a cooperative launch checks it) and each with at
  // least one tile, so that every CTA writes its partial in every pass
  // (one CTA per SM; the packet buffer has a slot more than that)
  const int grid = std::max(1, std::min(p.total_tiles, std::min(n_sm, ca.cap - 1)));
  p.chunk_q = p.total_tiles / grid;
  p.chunk_r = p.total_tiles % grid;
  ca.bar_count = grid + ca.bar_count;   // ca.bar_count comes in as the extra arrivals to wait for
  ca.G = grid;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(fx_threads<TH>());
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, lanczos_step64<R, TH, D, V, ISO>, p, ca);
}

template <int R, int TH, bool D, bool V>
cudaError_t launch_iso(const LaunchParams& p, int n_sm, const CoopArgs& ca, cudaStream_t s) {
  return p.iso ? launch_t<R, TH, D, V, true>(p, n_sm, ca, s) : launch_t<R, TH, D, V, false>(p, n_sm, ca, s);
}

template <int R, int TH>
cudaError_t launch_r(bool diri, bool hasv, const LaunchParams& p, int n_sm, const CoopArgs& ca, cudaStream_t s) {
  if (diri) return hasv ? launch_iso<R, TH, true, true>(p, n_sm, ca, s) : launch_iso<R, TH, true, false>(p, n_sm, ca, s);
  return hasv ? launch_iso<R, TH, false, true>(p, n_sm, ca, s) : launch_iso<R, TH, false, false>(p, n_sm, ca, s);
}

}  // namespace

cudaError_t launch_step64(int th, int order, bool diri, bool hasv, const LaunchParams& p, int n_sm,
                          const CoopArgs& ca, cudaStream_t s) {
  if (th == 16) return order == 2 ? launch_r<1, 16>(diri, hasv, p, n_sm, ca, s) : launch_r<2, 16>(diri, hasv, p, n_sm, ca, s);
  return order == 2 ? launch_r<1, 8>(diri, hasv, p, n_sm, ca, s) : launch_r<2, 8>(diri, hasv, p, n_sm, ca, s);
}

}  // namespace dirac
