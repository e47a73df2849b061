// dirac_pass64.cu -- launchers of the fixed-point FP64 pass and recombination.
#include "dirac.h"
#include "dirac_internal.h"
#include "dirac_pass64.cuh"

#include <cuda_runtime.h>

#include <algorithm>

namespace dirac {

namespace {

// Persistent launch: one CTA per SM (at most one worker per tile), each taking
// a contiguous chunk of the tile list whose size differs from the others' by at
// most one tile.
template <int R, int TH, bool D, bool V, bool ISO>
cudaError_t launch_t(LaunchParams p, const LaunchShape& ls, cudaStream_t s) {
  static std::atomic<int> occ_dev[OCC_MAX_DEVICES];
  constexpr size_t smem = fx_smem_bytes<R, TH>();
  int occ = 0;
  cudaError_t e = occupancy_on_device(occ_dev, lanczos_pass64<R, TH, D, V, ISO>, fx_threads<TH>(), smem, &occ);
  if (e != cudaSuccess) return e;
  const int per_sm = ls.cta_cap > 0 ? std::min(std::max(occ, 1), ls.cta_cap) : std::max(occ, 1);
  const int grid = std::max(1, std::min(p.total_tiles, ls.n_sm * per_sm));
  p.chunk_q = p.total_tiles / grid;
  p.chunk_r = p.total_tiles % grid;
  return launch_pdl(lanczos_pass64<R, TH, D, V, ISO>, grid, fx_threads<TH>(), smem, s, p);
}

// kx = ky (dx = dy): the two differences of a row are added before their one product
template <int R, int TH, bool D, bool V>
cudaError_t launch_iso(const LaunchParams& p, const LaunchShape& ls, cudaStream_t s) {
  return p.iso ? launch_t<R, TH, D, V, true>(p, ls, s) : launch_t<R, TH, D, V, false>(p, ls, s);
}

template <int R, int TH>
cudaError_t launch_r(bool diri, bool hasv, const LaunchParams& p, const LaunchShape& ls, cudaStream_t s) {
  if (diri) return hasv ? launch_iso<R, TH, true, true>(p, ls, s) : launch_iso<R, TH, true, false>(p, ls, s);
  return hasv ? launch_iso<R, TH, false, true>(p, ls, s) : launch_iso<R, TH, false, false>(p, ls, s);
}

}  // namespace

cudaError_t launch_pass64(int order, bool diri, bool hasv, const LaunchParams& p, const LaunchShape& ls,
                          cudaStream_t s) {
  if (ls.th == 16) return order == 2 ? launch_r<1, 16>(diri, hasv, p, ls, s) : launch_r<2, 16>(diri, hasv, p, ls, s);
  return order == 2 ? launch_r<1, 8>(diri, hasv, p, ls, s) : launch_r<2, 8>(diri, hasv, p, ls, s);
}

cudaError_t launch_recombine64(const RecombParams& rp, int grid, cudaStream_t s) {
  return launch_pdl(recombine64, grid, 256, 0, s, rp);
}

}  // namespace dirac
