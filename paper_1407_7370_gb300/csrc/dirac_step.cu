// dirac_step.cu -- launcher of the FP64 one-launch time step (`lanczos_step`):
// all Lanczos passes of a step of one problem and its recombination in one
// cooperative launch, the passes separated by grid-wide barriers.  Kept in a
// translation unit of its own so that it compiles in parallel with the
// per-pass kernels.
#include "dirac.h"
#include "dirac_internal.h"
#include "dirac_kernels.cuh"

#include <cuda_runtime.h>

#include <algorithm>

namespace dirac {

namespace {

template <int R, int TH, bool D, bool V, bool ISO>
cudaError_t launch_step_t(LaunchParams p, int n_sm, CoopArgs ca, cudaStream_t s) {
  static std::atomic<int> occ_dev[OCC_MAX_DEVICES];
  constexpr int NT = pass_threads<double, TH>();
  constexpr size_t smem = dyn_smem_bytes<double, R, TH, sub_workers<double>()>();
  int occ = 0;
  cudaError_t e = occupancy_on_device(occ_dev, lanczos_step<R, TH, D, V, ISO>, NT, smem, &occ);
  if (e != cudaSuccess) return e;
  if (occ < 1) return cudaErrorCooperativeLaunchTooLarge;
  // every CTA resident (a cooperative launch checks it) and each with at
  // least one tile, so that every CTA writes its partial in every pass
  const int grid = std::max(1, std::min(std::min(p.total_tiles, n_sm * occ), ca.cap));
  p.chunk_q = p.total_tiles / grid;
  p.chunk_r = p.total_tiles % grid;
  ca.bar_count = grid + ca.bar_count;   // ca.bar_count comes in as the extra arrivals to wait for
  ca.G = grid;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, lanczos_step<R, TH, D, V, ISO>, p, ca);
}

template <int R, int TH, bool D, bool V>
cudaError_t launch_step_iso(const LaunchParams& p, int n_sm, const CoopArgs& ca, cudaStream_t s) {
  return p.iso ? launch_step_t<R, TH, D, V, true>(p, n_sm, ca, s) : launch_step_t<R, TH, D, V, false>(p, n_sm, ca, s);
}

template <int R, int TH>
cudaError_t launch_step_r(bool diri, bool hasv, const LaunchParams& p, int n_sm, const CoopArgs& ca, cudaStream_t s) {
  if (diri) return hasv ? launch_step_iso<R, TH, true, true>(p, n_sm, ca, s)
                        : launch_step_iso<R, TH, true, false>(p, n_sm, ca, s);
  return hasv ? launch_step_iso<R, TH, false, true>(p, n_sm, ca, s)
              : launch_step_iso<R, TH, false, false>(p, n_sm, ca, s);
}

template <int TH>
cudaError_t launch_step_s(int order, bool diri, bool hasv, const LaunchParams& p, int n_sm, const CoopArgs& ca,
                          cudaStream_t s) {
  return order == 2 ? launch_step_r<1, TH>(diri, hasv, p, n_sm, ca, s)
                    : launch_step_r<2, TH>(diri, hasv, p, n_sm, ca, s);
}

}  // namespace

cudaError_t launch_step(int precision, int th, int order, bool diri, bool hasv, const LaunchParams& p, int n_sm,
                        const CoopArgs& ca, cudaStream_t s) {
  // the mixed path has its own one-launch step (dirac_step32.cu)
  if (precision != DIRAC_FP64) return cudaErrorInvalidValue;
  if (th == 16) return launch_step_s<16>(order, diri, hasv, p, n_sm, ca, s);
  return launch_step_s<32>(order, diri, hasv, p, n_sm, ca, s);
}

}  // namespace dirac
