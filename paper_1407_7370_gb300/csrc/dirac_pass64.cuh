// dirac_pass64.cuh -- device code of the FP64 path: one Lanczos pass over
// complex128 fields with its products in 60-bit fixed point (dirac_fixed.cuh),
// the recombination likewise, and the one-launch step made of them.  Same
// recurrence, tile list and scalars as dirac_kernels.cuh.
#pragma once
#include <type_traits>

#include "dirac_kernels.cuh"

namespace dirac {

// Tiles of 32 x TH sites.  A tile worker has fx_warps warps with fx_rows rows a
// thread; a CTA (one per SM) holds fx_workers of them, so that one worker's loads
// and barriers overlap the others' arithmetic.  TH = 16: four workers of four
// warps, four rows a thread (128 registers): 2048^2, m = 20 in 4.6 ms against 4.83
// with two workers of eight warps on 32-row tiles and 5.05 with three of eight
// warps and two rows a thread (80 registers).  TH = 8: three workers of eight
// warps, one row a thread, for grids of few tiles, where the time of one tile
// counts (64^2, m = 10: 111 us a step; the tall tiles took 167).
template <int TH>
__host__ __device__ constexpr int fx_warps() { return TH == 16 ? 4 : 8; }
template <int TH>
__host__ __device__ constexpr int fx_rows() { return TH / fx_warps<TH>(); }
template <int TH>
__host__ __device__ constexpr int fx_workers() { return TH == 16 ? 4 : 3; }
template <int TH>
__host__ __device__ constexpr int fx_threads() { return fx_workers<TH>() * fx_warps<TH>() * 32; }

constexpr int COEF_SLOTS = 16;   // eight per half
template <int R, int TH>
__host__ __device__ constexpr int half_sites() { return (TH + 2 * R) * (TILE_W + 2 * R); }

// Shared memory of one tile worker.  q^_i on the tile and its halo, q^_{i-1} on
// the tile, in fixed point; the upper and the lower components in separate
// halves (16 bytes per site each, so that a warp's row is read without bank
// conflicts); a table of coefficients per warp; the exponents of two tiles.
template <int R, int TH>
struct FxTile {
  longlong2 q[2][half_sites<R, TH>()];
  longlong2 qp[2][TH * TILE_W];
  int2 coef[fx_warps<TH>()][COEF_SLOTS];
  unsigned emax[2][4];
};
template <int R, int TH>
__host__ __device__ constexpr size_t fx_smem_bytes() { return fx_workers<TH>() * sizeof(FxTile<R, TH>); }

// What a CTA needs of the problem it works on, in shared memory so that it
// occupies no registers between its uses.
struct FxSegment {
  const vec4* qsrc;        // q^_{i-1} (q^_1 if i = 1)
  const vec4* yprev;
  vec4* q_out;             // null: not stored
  vec4* y_out;
  const double* V;
  double gd;
  double coef[COEF_SLOTS]; // slots 0 diagonal, 1 kx, 2 ky, 3 c A_x, 4 c A_y, 5 coupling, of the upper and the lower row
  int nx, ny, tiles_x, tile_begin, i, yexp, vbe, has_ax, has_ay;
  // what the pointers of a pass are made from
  const vec4* psi;
  vec4 *basis, *ybuf0, *ybuf1;
};

// One of P, Y, X over the lanes of a warp
__device__ __forceinline__ double lane_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum over `n` slots of three doubles (P, Y, X), quantity j by warp j: an FP64
// addition occupies a sub-partition for 76 cycles, so the three sums run on
// three of them side by side.  Fixed order; result in tot[0..2] after the next
// barrier of the CTA.
constexpr int SLOTS_IN_FLIGHT = 5;   // loads in flight per lane: 160 slots, one per SM

__device__ __forceinline__ void sum_slots(const double* slots, int n, double* tot) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp >= 3) return;
  double t = 0.0;
  for (int c0 = lane; c0 < n; c0 += SLOTS_IN_FLIGHT * 32) {
    double v[SLOTS_IN_FLIGHT];
#pragma unroll
    for (int k = 0; k < SLOTS_IN_FLIGHT; ++k)
      v[k] = c0 + k * 32 < n ? __ldcg(slots + 3 * (c0 + k * 32) + warp) : 0.0;
#pragma unroll
    for (int k = 0; k < SLOTS_IN_FLIGHT; ++k) t += v[k];
  }
  t = lane_sum(t);
  if (lane == 0) tot[warp] = t;
}

// The grid barrier of the one-launch step is the exchange of the partials that
// every CTA needs anyway: a partial travels as two 64-bit words, each half of
// the number beside the pass's epoch, so that a reader that sees the epoch has
// the number too -- one L2 round trip instead of an arrival counter, a
// generation and the read of the slots (4 against 6.5 thousand cycles).  Slot
// of CTA c, quantity j: words 6 c + 2 j and 6 c + 2 j + 1.
__device__ __forceinline__ void post_partial(unsigned long long* slots, int j, double v, unsigned epoch) {
  __threadfence();   // the CTA's stores (ordered before by a barrier) before the words
  cuda::atomic_ref<unsigned long long, cuda::thread_scope_device> w0(slots[6 * blockIdx.x + 2 * j]);
  cuda::atomic_ref<unsigned long long, cuda::thread_scope_device> w1(slots[6 * blockIdx.x + 2 * j + 1]);
  w0.store((unsigned long long)epoch << 32 | (unsigned)__double2loint(v), cuda::memory_order_relaxed);
  w1.store((unsigned long long)epoch << 32 | (unsigned)__double2hiint(v), cuda::memory_order_relaxed);
}

// The sums over all CTAs' partials of this epoch, quantity j by warp j, in
// tot[0..2] after the next barrier of the CTA.  After a bounded number of polls,
// or once another CTA has given up, *failed is set and bar[2] tells the others.
constexpr unsigned SLOT_SPIN_MAX = 1u << 21;   // polls of an L2 round trip each: about a second

__device__ __forceinline__ void collect_partials(unsigned long long* slots, int n, double* tot, unsigned epoch,
                                                 unsigned* bar, int* failed) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp >= 3) return;
  cuda::atomic_ref<unsigned, cuda::thread_scope_device> timeout(bar[2]);
  double t = 0.0;
  bool good = true;
  for (int c0 = lane; c0 < n && good; c0 += SLOTS_IN_FLIGHT * 32) {
    unsigned long long w[SLOTS_IN_FLIGHT][2];
    unsigned missing = 0u, spins = 0;   // slots still awaited: only these are polled again
#pragma unroll
    for (int k = 0; k < SLOTS_IN_FLIGHT; ++k) {
      w[k][0] = w[k][1] = 0;
      if (c0 + k * 32 < n) missing |= 1u << k;
    }
    for (;;) {
#pragma unroll
      for (int k = 0; k < SLOTS_IN_FLIGHT; ++k) {
        if (missing >> k & 1u) {
          const int at = 6 * (c0 + k * 32) + 2 * warp;
          cuda::atomic_ref<unsigned long long, cuda::thread_scope_device> w0(slots[at]), w1(slots[at + 1]);
          w[k][0] = w0.load(cuda::memory_order_relaxed);
          w[k][1] = w1.load(cuda::memory_order_relaxed);
        }
      }
#pragma unroll
      for (int k = 0; k < SLOTS_IN_FLIGHT; ++k)
        if ((unsigned)(w[k][0] >> 32) == epoch && (unsigned)(w[k][1] >> 32) == epoch) missing &= ~(1u << k);
      if (!missing) break;
      if (++spins > SLOT_SPIN_MAX || ((spins & 63u) == 0u && timeout.load(cuda::memory_order_relaxed) != 0u)) {
        timeout.store(1u, cuda::memory_order_relaxed);
        *failed = 1;
        good = false;
        break;
      }
    }
#pragma unroll
    for (int k = 0; k < SLOTS_IN_FLIGHT; ++k) t += __hiloint2double((int)(unsigned)w[k][1], (int)(unsigned)w[k][0]);
  }
  __syncwarp();
  __threadfence();   // the other CTAs' fields after their words
  t = lane_sum(t);
  if (lane == 0) tot[warp] = t;
}

// This CTA's share of a problem, the warps' sums in red[], -> one partial per
// (problem, CTA) slot.  COOP = false: then the problem's ticket, and the CTA
// that completes the problem sums its slots and updates its scalars.  COOP =
// true (one-launch step): the partial is posted and the caller collects them.
template <bool COOP, int NW>
__device__ __forceinline__ void pass_sums64(const LaunchParams& lp, const Problem* pr, int i, int seg_tiles,
                                            double (*red)[3], double* tot, int* last_flag,
                                            unsigned long long* coop_slots, unsigned epoch) {
  const int cq = lp.chunk_q, cr = lp.chunk_r;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (warp < 3) {
    const double v = lane_sum(lane < NW ? red[lane][warp] : 0.0);
    if (lane == 0) {
      if constexpr (COOP) post_partial(coop_slots, warp, v, epoch);
      else pr->partials[3 * (blockIdx.x - cta_of_tile(pr->tile_begin, cq, cr)) + warp] = v;
    }
  }
  if constexpr (!COOP) {
    __syncthreads();
    if (threadIdx.x == 0) {
      // release the CTA's partial / acquire everybody else's
      cuda::atomic_ref<unsigned, cuda::thread_scope_device> ticket(pr->st->counter);
      *last_flag = (ticket.fetch_add((unsigned)seg_tiles, cuda::memory_order_acq_rel) + seg_tiles ==
                    (unsigned)pr->ntiles);
    }
    __syncthreads();
    if (*last_flag) {
      const int cta_lo = cta_of_tile(pr->tile_begin, cq, cr);
      sum_slots(pr->partials, cta_of_tile(pr->tile_begin + pr->ntiles - 1, cq, cr) - cta_lo + 1, tot);
      __syncthreads();
      if (warp == 0) {
        if (lane == 0) pr->st->counter = 0u;
        finish_fast(lp, pr, pr->st, i, tot[0], tot[1], tot[2], pr->shift);
      }
      __syncthreads();
    }
  }
}

// One FP64 pass over this CTA's chunk.  COOP = false: a launch of its own
// (lanczos_pass64).  COOP = true: inside the one-launch step: one problem, the
// state read from `coop_st`, and the CTA's partial sums written to coop_slots;
// the caller synchronises the grid and finishes.
//
// Per site and pass only the formation of q^_i (one FP64 multiply-add per
// number, the scale of y^ being a power of two) and the final conversion of
// y^_i use the FP64 pipe.  The stencil, the coupling to q^_{i-1} and the three
// sums are fixed point: a tile (with its halo) shares one exponent for the
// upper and one for the lower components of q^_i, another pair for q^_{i-1},
// taken from their largest numbers; every row of the operator is one sum of
// products, good to 2^-58 of the row's scale (ROW_BITS, dirac_fixed.cuh): a site's y^
// has the accuracy that FP64 gives it as long as its numbers are within about 2^-4
// of the largest of its tile, and 2^-58 of that largest below.  y^ enters the sums
// as 60 bits of the warp's largest number; each tile's sums are integers, the
// squares with their lowest partial products, P without them.
//
// Per tile: load and form (all loads of a thread in flight at once), exponents
// -> barrier -> fixed point into shared memory, coefficients at the tile's
// scale -> barrier -> the upper, then the lower components.
//
// The FP64 multiply-adds of this pass (40 a site) kept the FP64 pipe, 64 cycles
// a warp instruction, busy for 0.8 of the time.  Now the pipe is a third busy
// and the integer pipes 0.40 and 0.46; what bounds the pass is latency, four
// warps a sub-partition being what 128 registers allow (stall cycles an
// instruction: fixed latencies 1.9, loads 1.3, shared memory 1.2).  A step of
// m = 20 with V, A constant: 1024^2 2.50 -> 1.42 ms; 4096^2, m = 10: 17.3 ->
// 8.4 ms; 64^2, m = 10: 194 -> 111 us.  A pass of 2048^2: 206 us, 2.6 TB/s.
template <int R, int TH, bool DIRI, bool HAS_V, bool ISO, bool COOP>
__device__ __forceinline__ void pass_body64(const LaunchParams& lp, const DevState* coop_st,
                                            unsigned long long* coop_slots, int step, unsigned epoch,
                                            double* coop_shift) {
  constexpr int RPT = fx_rows<TH>();
  constexpr int NTS = 32 * fx_warps<TH>();  // threads of a worker
  constexpr int SUB = fx_workers<TH>();
  constexpr int NW = SUB * fx_warps<TH>();  // warps
  constexpr int W = TILE_W + 2 * R;
  constexpr int F = fx::ROW_BITS;           // bits of q^ and q^_{i-1}
  constexpr int NH_ROW = 2 * R * TILE_W, NH = NH_ROW + 2 * R * TH;
  constexpr int HPT = (NH + NTS - 1) / NTS; // halo sites per thread
  static_assert(2 * RPT <= 8, "bounds of the per-tile sums");
  extern __shared__ __align__(32) unsigned char dyn_smem[];
  __shared__ double red[NW][3], tot[3];
  __shared__ int last_flag;
  __shared__ FxSegment sg;

  const int cq = lp.chunk_q, cr = lp.chunk_r;
  const int t_begin = blockIdx.x * cq + min((int)blockIdx.x, cr);
  const int t_end = t_begin + cq + ((int)blockIdx.x < cr ? 1 : 0);
  const int sub = (int)threadIdx.x / NTS;   // this thread's worker
  const int ltid = (int)threadIdx.x - sub * NTS;
  const int tx = ltid & 31, tg = ltid >> 5;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r0 = tg * RPT;                  // this thread's rows of a tile
  FxTile<R, TH>& sm = reinterpret_cast<FxTile<R, TH>*>(dyn_smem)[sub];
  auto sub_sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + sub), "r"(NTS) : "memory"); };
  if (ltid < 8) sm.emax[ltid >> 2][ltid & 3] = 0u;
  int par = 0;                              // which exponents the tile uses

  // problem of the first tile (problems are sorted by tile_begin)
  int b = 0;
  if constexpr (!COOP) {
    int lo = 0, hi = lp.nprob - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (lp.probs[mid].tile_begin <= t_begin) lo = mid; else hi = mid - 1;
    }
    b = lo;
  }
  for (int t = t_begin; t < t_end; ++b) {
    const Problem* pr = lp.probs + b;
    const int seg_end = COOP ? t_end : min(t_end, pr->tile_begin + pr->ntiles);
    const int seg_tiles = seg_end - t;
    const DevState* st = COOP ? coop_st : lp.states + b;
    if (!COOP && st->stopped) { t = seg_end; continue; }
    if (threadIdx.x < COEF_SLOTS) {
      const int j = threadIdx.x;
      const int i = lp.probe ? 1 : max(1, st->cur_pass);
      const PassCoef& pc = lp.probe ? pr->probe_coef : st->pc_cur;
      if (!COOP || epoch == 1u) {   // what the passes of a step share
        const FieldStep* const fs = lp.fields + step * lp.fstride + b;
        double c = 0.0;
        if ((j & 7) == 1) c = R == 1 ? pr->kx : 8.0 * pr->kx;   // of the inner difference
        if ((j & 7) == 2) c = R == 1 ? pr->ky : 8.0 * pr->ky;
        if ((j & 7) == 3) c = fs->cAx;
        if ((j & 7) == 4) c = fs->cAy;
        sg.coef[j] = c;
        if (COOP && TH == 8 && j == 6) *coop_shift = pr->shift;
        if (j == 0) {
          sg.psi = pr->psi;
          sg.basis = static_cast<vec4*>(pr->basis);
          sg.ybuf0 = static_cast<vec4*>(pr->ybuf0);
          sg.ybuf1 = static_cast<vec4*>(pr->ybuf1);
          sg.V = HAS_V ? static_cast<const double*>(pr->V) : nullptr;   // NULL: V = 0 for this problem
          sg.nx = pr->nx;
          sg.ny = pr->ny;
          sg.tiles_x = pr->tiles_x;
          sg.tile_begin = pr->tile_begin;
          sg.vbe = pr->vbe;
          sg.has_ax = fs->cAx != 0.0;
          sg.has_ay = fs->cAy != 0.0;
        }
      }
      if ((j & 7) == 0) sg.coef[j] = j ? pc.ad0 : pc.au0;
      if ((j & 7) == 5) sg.coef[j] = i >= 2 ? pc.e : 0.0;
      if (j == 0) {
        const size_t n = (size_t)sg.nx * sg.ny;
        sg.qsrc = i <= 2 ? sg.psi : sg.basis + (size_t)(i - 3) * n;
        sg.yprev = (i & 1) ? sg.ybuf0 : sg.ybuf1;
        sg.q_out = (i >= 2 && !lp.probe) ? sg.basis + (size_t)(i - 2) * n : nullptr;
        sg.y_out = (i < lp.m && !lp.probe) ? ((i & 1) ? sg.ybuf1 : sg.ybuf0) : nullptr;
        sg.gd = pc.gd;
        sg.i = i;
        sg.yexp = (int)pc.yexp;
      }
    }
    __syncthreads();
    bool bad = __any_sync(0xffffffffu, fx::exp_field(sg.coef[lane & 15]) == 0x7ff);

    // index of grid point (gx, gy), wrapped; `in` false outside the grid (Dirichlet)
    auto site = [&](int gx, int gy, bool& in) {
      bool ox, oy;
      const int ix = wrap<DIRI>(gx, sg.nx, ox), iy = wrap<DIRI>(gy, sg.ny, oy);
      in = !(ox || oy);
      return (unsigned)iy * (unsigned)sg.nx + (unsigned)ix;
    };
    // q^_i from what was loaded, and q^_{i-1} (zero if i = 1)
    auto form = [&](const vec4& qv, const vec4& yv, bool first, double (&q)[4], double (&qp)[4]) {
      cvt4(qv, qp);
      if (first) {
#pragma unroll
        for (int c = 0; c < 4; ++c) { q[c] = qp[c]; qp[c] = 0.0; }
      } else {
        double y[4];
        cvt4(yv, y);
#pragma unroll
        for (int c = 0; c < 4; ++c) q[c] = fma(-sg.gd, qp[c], y[c]);
      }
    };
    auto mag = [](double x) { return (unsigned)__double2hiint(x) << 1; };   // orders by |x| (to 20 bits)

    // Sums of tiles waiting for their conversion to FP64: lane 6 c + 3 h + j holds
    // sum j (P, Y, X) of half h of the c-th of up to five tiles, so that the warp
    // converts 30 sums at once; lane l then accumulates in acc sums of kind l % 3
    double acc = 0.0;
    fx::WarpSum pend = {0, 0, 0};
    int pend_e = 0, pend_tiles = 0;
    for (int tt = t + sub; tt < seg_end; tt += SUB) {
      const int lt = tt - sg.tile_begin;
      const int ty = lt / sg.tiles_x;
      const int x0 = (lt - ty * sg.tiles_x) * TILE_W;
      const int y0 = ty * TH;
      const bool full = x0 + TILE_W <= sg.nx && y0 + TH <= sg.ny;
      const int rows_in = x0 + tx < sg.nx ? sg.ny - (y0 + r0) : 0;    // row k is in the grid if k < rows_in
      const unsigned idx0 = (unsigned)(y0 + r0) * (unsigned)sg.nx + (unsigned)(x0 + tx);   // used where in the grid
      const int at0 = (r0 + R) * W + tx + R;                          // this thread's first site in the tile
      {
        double q[RPT][4], qp[RPT][4], hq[HPT][4];
        int hat[HPT];                           // the halo sites' places in the tile
        {
          // all loads before their first use
          const bool first = sg.i == 1;
          const vec4* const qsrc = sg.qsrc;
          const vec4* const yprev = first ? qsrc : sg.yprev;
          vec4 zero;
          zero.x = zero.y = zero.z = zero.w = 0.0;
          vec4 qv[RPT], yv[RPT], hqv[HPT], hyv[HPT];
          if (full) {
#pragma unroll
            for (int k = 0; k < RPT; ++k) {
              const unsigned idx = idx0 + (unsigned)(k * sg.nx);
              qv[k] = ld4<COOP>(qsrc + idx);
              yv[k] = first ? zero : ld4<COOP>(yprev + idx);
            }
          } else {
#pragma unroll
            for (int k = 0; k < RPT; ++k) {
              bool in;
              const unsigned idx = site(x0 + tx, y0 + r0 + k, in);
              qv[k] = in ? ld4<COOP>(qsrc + idx) : zero;
              yv[k] = in && !first ? ld4<COOP>(yprev + idx) : zero;
            }
          }
#pragma unroll
          for (int p = 0; p < HPT; ++p) {
            const int h = ltid + p * NTS;
            hqv[p] = hyv[p] = zero;
            hat[p] = 0;
            if (h < NH) {
              int hrow, hcol;
              if (h < NH_ROW) {                 // rows above / below
                const int r = h / TILE_W;
                hrow = (r < R) ? r : TH + r;
                hcol = (h % TILE_W) + R;
              } else {                          // columns left / right
                const int h2 = h - NH_ROW;
                hrow = h2 / (2 * R) + R;
                const int c = h2 % (2 * R);
                hcol = (c < R) ? c : TILE_W + c;
              }
              hat[p] = hrow * W + hcol;
              bool in;
              const unsigned idx = site(x0 + hcol - R, y0 + hrow - R, in);
              if (in) {
                hqv[p] = ld4<COOP>(qsrc + idx);
                if (!first) hyv[p] = ld4<COOP>(yprev + idx);
              }
            }
          }
#pragma unroll
          for (int k = 0; k < RPT; ++k) form(qv[k], yv[k], first, q[k], qp[k]);
#pragma unroll
          for (int p = 0; p < HPT; ++p) {
            hq[p][0] = hq[p][1] = hq[p][2] = hq[p][3] = 0.0;
            double unused[4];
            if (ltid + p * NTS < NH) form(hqv[p], hyv[p], first, hq[p], unused);
          }
        }
        // the largest numbers of the tile
        unsigned m0 = 0u, m1 = 0u, m2 = 0u, m3 = 0u;
#pragma unroll
        for (int p = 0; p < HPT; ++p) {
          m0 = max(m0, max(mag(hq[p][0]), mag(hq[p][1])));
          m1 = max(m1, max(mag(hq[p][2]), mag(hq[p][3])));
        }
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
          m0 = max(m0, max(mag(q[k][0]), mag(q[k][1])));
          m1 = max(m1, max(mag(q[k][2]), mag(q[k][3])));
          m2 = max(m2, max(mag(qp[k][0]), mag(qp[k][1])));
          m3 = max(m3, max(mag(qp[k][2]), mag(qp[k][3])));
        }
        m0 = __reduce_max_sync(0xffffffffu, m0);
        m1 = __reduce_max_sync(0xffffffffu, m1);
        m2 = __reduce_max_sync(0xffffffffu, m2);
        m3 = __reduce_max_sync(0xffffffffu, m3);
        if (lane < 4) atomicMax(&sm.emax[par][lane], lane == 0 ? m0 : lane == 1 ? m1 : lane == 2 ? m2 : m3);
        if (vec4* const q_out = sg.q_out) {
#pragma unroll
          for (int k = 0; k < RPT; ++k) {
            if (k < rows_in) {
              vec4 o;
              o.x = q[k][0]; o.y = q[k][1]; o.z = q[k][2]; o.w = q[k][3];
              q_out[idx0 + (unsigned)(k * sg.nx)] = o;
            }
          }
        }
        sub_sync();   // the exponents are complete, and the previous tile has been read
        // exponents of 128 and below (numbers under 2^-894) count as zero
        const int be_u = max((int)(sm.emax[par][0] >> 21), 128), be_d = max((int)(sm.emax[par][1] >> 21), 128);
        const int be_pu = max((int)(sm.emax[par][2] >> 21), 128), be_pd = max((int)(sm.emax[par][3] >> 21), 128);
        if (ltid < 4) sm.emax[par ^ 1][ltid] = 0u;
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
          // sites beyond the grid's edge are halo of the sites inside, but not summed
          const int at = at0 + k * W, ap = (r0 + k) * TILE_W + tx;
          sm.q[0][at] = make_longlong2(fx::to_fixed<F>(q[k][0], be_u), fx::to_fixed<F>(q[k][1], be_u));
          sm.q[1][at] = make_longlong2(fx::to_fixed<F>(q[k][2], be_d), fx::to_fixed<F>(q[k][3], be_d));
          sm.qp[0][ap] = make_longlong2(-fx::to_fixed<F>(qp[k][0], be_pu), -fx::to_fixed<F>(qp[k][1], be_pu));
          sm.qp[1][ap] = make_longlong2(-fx::to_fixed<F>(qp[k][2], be_pd), -fx::to_fixed<F>(qp[k][3], be_pd));
        }
#pragma unroll
        for (int p = 0; p < HPT; ++p) {
          if (ltid + p * NTS < NH) {
            sm.q[0][hat[p]] = make_longlong2(fx::to_fixed<F>(hq[p][0], be_u), fx::to_fixed<F>(hq[p][1], be_u));
            sm.q[1][hat[p]] = make_longlong2(fx::to_fixed<F>(hq[p][2], be_d), fx::to_fixed<F>(hq[p][3], be_d));
          }
        }
        // this warp's coefficient table: row scale = the largest term's, the
        // coefficients of a row as 60-bit fractions of it.  Lanes 0-7: the upper
        // row, 8-15 the lower; slot 6 is V, of which the exponent alone counts
        // here, slot 7 takes the scale
        const int cj = lane & 7, ch = (lane >> 3) & 1;
        const double my_coef = sg.coef[lane & 15];
        const int my_xe = cj == 6 ? (HAS_V && sg.V ? sg.vbe : 0) : fx::exp_field(my_coef);
        const int be_own = ch ? be_d : be_u, be_oth = ch ? be_u : be_d, be_p = ch ? be_pd : be_pu;
        const int be_x = (cj == 0 || cj == 6) ? be_own : (cj == 5 ? be_p : be_oth);
        int sc = my_xe ? my_xe + be_x : 0;
        sc = max(sc, __shfl_xor_sync(0xffffffffu, sc, 1));
        sc = max(sc, __shfl_xor_sync(0xffffffffu, sc, 2));
        sc = max(sc, __shfl_xor_sync(0xffffffffu, sc, 4));
        if (lane < COEF_SLOTS) {
          const fx::Limbs l = fx::split(fx::to_fixed<60>(my_coef, max(sc - be_x, 63)));
          sm.coef[tg][lane] = cj == 7 ? make_int2(sc, 0) : make_int2(l.hi, l.lo);
        }
      }
      sub_sync();   // tile and coefficients are in shared memory

      auto half = [&](auto half_c) {
        constexpr int HALF = decltype(half_c)::value;
        const longlong2* const own = sm.q[HALF] + at0;
        const longlong2* const oth = sm.q[1 - HALF] + at0;
        const longlong2* const sqp = sm.qp[HALF] + r0 * TILE_W + tx;
        const int2* const kc = sm.coef[tg] + 8 * HALF;
        auto coef = [&](int j) { const int2 v = kc[j]; return fx::Limbs{v.x, v.y}; };
        const int sc = kc[7].x;
        const int be_own = max((int)(sm.emax[par][HALF] >> 21), 128);
        bad = bad || be_own == 0x7ff || (sm.emax[par][2 + HALF] >> 21) == 0x7ffu;
        const int texp = sc - 2044 - F + (fx::ROW_SHIFT - 28) + sg.yexp;       // unit of y as stored
        // columns of the other half: rows r0 - R .. r0 + RPT + R - 1
        longlong2 col[RPT + 2 * R];
#pragma unroll
        for (int j = 0; j < RPT + 2 * R; ++j) col[j] = oth[(j - R) * W];
        long long v[RPT][2];
        unsigned vor = 0u;                              // the upper words of all |v|, or-ed
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
          const longlong2* const row = oth + k * W;
          fx::Acc s0, s1;
          // upper: (mc^2+V-s-sigma) u + c[-i D_x d - D_y d + (A_x - i A_y) d]
          // lower: (-mc^2+V-s-sigma) d + c[-i D_x u + D_y u + (A_x + i A_y) u]
          {
            // differences along x of (re, im), and along y
            const longlong2 xl = row[-1], xr = row[1];
            long long hxr = xl.x - xr.x, hxi = xr.y - xl.y;          // -D_x re, D_x im
            long long hyr = col[k + R + 1].x - col[k + R - 1].x, hyi = col[k + R + 1].y - col[k + R - 1].y;
            if constexpr (R == 2) {
              const longlong2 xl2 = row[-2], xr2 = row[2];
              hxr -= fx::eighth(xl2.x - xr2.x);
              hxi -= fx::eighth(xr2.y - xl2.y);
              hyr -= fx::eighth(col[k + 2 * R].x - col[k].x);
              hyi -= fx::eighth(col[k + 2 * R].y - col[k].y);
            }
            const fx::Limbs kx = coef(1);
            if constexpr (ISO) {
              s0.mac(fx::split(HALF ? hxi + hyr : hxi - hyr), kx);
              s1.mac(fx::split(HALF ? hxr + hyi : hxr - hyi), kx);
            } else {
              const fx::Limbs ky = coef(2);
              s0.mac(fx::split(hxi), kx);
              s1.mac(fx::split(hxr), kx);
              s0.mac(fx::split(HALF ? hyr : -hyr), ky);
              s1.mac(fx::split(HALF ? hyi : -hyi), ky);
            }
          }
          if (sg.has_ax) {
            const fx::Limbs kax = coef(3);
            s0.mac(fx::split(col[k + R].x), kax);
            s1.mac(fx::split(col[k + R].y), kax);
          }
          if (sg.has_ay) {
            const fx::Limbs kay = coef(4);
            s0.mac(fx::split(HALF ? -col[k + R].y : col[k + R].y), kay);
            s1.mac(fx::split(HALF ? col[k + R].x : -col[k + R].x), kay);
          }
          if (sg.i >= 2) {
            const fx::Limbs ke = coef(5);
            const longlong2 pv = sqp[k * TILE_W];
            s0.mac(fx::split(pv.x), ke);
            s1.mac(fx::split(pv.y), ke);
          }
          {
            const longlong2 cv = own[k * W];
            const fx::Limbs c0 = fx::split(cv.x), c1 = fx::split(cv.y), ka = coef(0);
            s0.mac(c0, ka);
            s1.mac(c1, ka);
            if constexpr (HAS_V) {
              if (const double* const Vp = sg.V) {
                const double pot = k < rows_in ? Vp[idx0 + (unsigned)(k * sg.nx)] : 0.0;
                const fx::Limbs kv = fx::split(fx::to_fixed<60>(pot, max(sc - be_own, 63)));
                s0.mac(c0, kv);
                s1.mac(c1, kv);
              }
            }
          }
          v[k][0] = s0.template value<fx::ROW_SHIFT>();
          v[k][1] = s1.template value<fx::ROW_SHIFT>();
          if (!full && k >= rows_in) v[k][0] = v[k][1] = 0;
          vor |= (unsigned)((v[k][0] ^ (v[k][0] >> 63)) >> 32) | (unsigned)((v[k][1] ^ (v[k][1] >> 63)) >> 32);
          vec4* const y_out = sg.y_out;
          if (y_out && k < rows_in) {
            // components of this half (16 of the site's 32 bytes); zero below the normal range
            double2* const yo = reinterpret_cast<double2*>(y_out + (idx0 + (unsigned)(k * sg.nx))) + HALF;
            *yo = texp >= -1022 ? make_double2(fx::to_double(v[k][0], texp), fx::to_double(v[k][1], texp))
                                : make_double2(0.0, 0.0);
          }
        }
        // the sums: y^ as 60 bits of the warp's largest number (the terms of a
        // row may cancel by many bits), q^ as it is
        const int sl = __clz((int)__reduce_or_sync(0xffffffffu, vor)) - 2;   // 0 .. 30
        fx::Acc aP;
        fx::SqAcc aY, aX;
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
          longlong2 cv = own[k * W];
          if (!full && k >= rows_in) cv.x = cv.y = 0;
          const fx::Limbs c0 = fx::split(cv.x), c1 = fx::split(cv.y);
          const fx::Limbs w0 = fx::split((v[k][0] << sl) >> 2), w1 = fx::split((v[k][1] << sl) >> 2);
          aP.mac(c0, w0);
          aP.mac(c1, w1);
          aY.sqr(w0);
          aY.sqr(w1);
          aX.sqr(c0);
          aX.sqr(c1);
        }
        // |q^| < 2^59 and |w| < 2^60: eight terms of q^ w stay below 2^62 in
        // units of 2^60, of w^2 below 2^63, of q^2 below 2^61
        const int qe = be_own - 1022 - F, ye = texp + 2 - sl;
        const fx::WarpSum wp = fx::warp_sum(aP.template value<28>());
        const fx::WarpSum wy = fx::warp_sum(aY.value()), wx = fx::warp_sum(aX.value());
        const int j = lane - 6 * pend_tiles - 3 * HALF;
        if (j == 0) { pend = wp; pend_e = qe + ye + 60; }
        if (j == 1) { pend = wy; pend_e = 2 * ye + 60; }
        if (j == 2) { pend = wx; pend_e = 2 * qe + 60; }
      };
      half(std::integral_constant<int, 0>{});
      half(std::integral_constant<int, 1>{});
      par ^= 1;
      if (++pend_tiles == 5) {
        acc += fx::scale2(fx::to_double(pend), pend_e);
        pend = {0, 0, 0};
        pend_tiles = 0;
      }
    }
    const int t0 = t;
    t = seg_end;
    acc += fx::scale2(fx::to_double(pend), pend_e);
    if (lane >= 30) acc = 0.0;
    // lanes l, l + 3, .. -> l (one tile: two of them)
    double accP = acc + __shfl_down_sync(0xffffffffu, acc, 3);
    if (seg_end - t0 > SUB) {
      acc += __shfl_down_sync(0xffffffffu, acc, 15);
      accP = acc;
#pragma unroll
      for (int k = 3; k < 15; k += 3) accP += __shfl_down_sync(0xffffffffu, acc, k);
    }
    const double accY = __shfl_sync(0xffffffffu, accP, 1), accX = __shfl_sync(0xffffffffu, accP, 2);
    if (bad) accP = __longlong_as_double(0x7ff8000000000000LL);   // not finite: reported by finish_pass
    if (lane == 0) { red[warp][0] = accP; red[warp][1] = accY; red[warp][2] = accX; }
    pass_sums64<COOP, NW>(lp, pr, sg.i, seg_tiles, red, tot, &last_flag, coop_slots, epoch);
  }
}

template <int R, int TH, bool DIRI, bool HAS_V, bool ISO>
__global__ void __launch_bounds__(fx_threads<TH>(), 1) lanczos_pass64(const __grid_constant__ LaunchParams lp) {
  // programmatic dependent launch: nothing the previous kernel wrote is read
  // before this point
  asm volatile("griddepcontrol.wait;" ::: "memory");
  pass_body64<R, TH, DIRI, HAS_V, ISO, false>(lp, nullptr, nullptr, *lp.step, 0u, nullptr);
  // the next kernel may be scheduled now (it waits for our completion)
  asm volatile("griddepcontrol.launch_dependents;");
}

// ---------------------------------------------------------------------------
// psi <- sum_j C_j q^_j (Eq. 17), q^_1 = psi, q^_j = basis[j-2] for j >= 2.  In
// FP64 the 16 multiply-adds per site and vector took 1024 cycles of a
// sub-partition against the 190 that reading the vector takes; in limbs they
// take somewhat longer than the read (m = 20, us, in brackets the time of the
// reads at the copy bandwidth: 256^2 21 (7), 512^2 56 (26), 1024^2 173 (104),
// 2048^2 649 (415); the FP64 multiply-adds alone would take 530 us at 1024^2).  The upper and the lower component
// of each site have a scale of their own, that of the largest |C_j q^_j| so far
// (the sums are shifted when a batch of D vectors raises it).  A product drops up to
// 2^-56 of that largest term, an eighth of what each of FP64's 2 k multiply-adds may.
// (One scale for both components left the lower one of a slow packet 2^-48 of itself;
// the second costs 0.4 % of a step at 1024^2.)
// ---------------------------------------------------------------------------
struct FxCoef {
  fx::Limbs re, im, mim;   // C_j and -Im C_j as 59-bit fractions of 2^(be - 1022)
  int be;
};
__device__ __forceinline__ FxCoef fx_coef(double re, double im) {
  FxCoef c;
  c.be = max(fx::exp_field(re), fx::exp_field(im));
  const long long i = fx::to_fixed<59>(im, max(c.be, 63));
  c.re = fx::split(fx::to_fixed<59>(re, max(c.be, 63)));
  c.im = fx::split(i);
  c.mim = fx::split(-i);
  return c;
}

template <int D>
__device__ __forceinline__ void recombine_site_fx(vec4* psi, const vec4* basis, size_t n, size_t s, int k,
                                                  const FxCoef* coef) {
  // factors below 2^59: 8 products in x stay below 2^62, all 64 below 2^62 in
  // units of 2^62
  static_assert(D % 4 == 0 && 2 * KMAX <= 64, "bounds of the sums");
  long long sum[4] = {0, 0, 0, 0};
  int beu = 1100, bed = 1100;   // exponent sums of the largest terms (those below 2^-938 count as zero)
  for (int j0 = 1; j0 <= k; j0 += D) {
    vec4 v[D];
#pragma unroll
    for (int u = 0; u < D; ++u) {
      const int j = j0 + u;
      if (j <= k) v[u] = j == 1 ? psi[s] : basis[(size_t)(j - 2) * n + s];
    }
    int nu = beu, nd = bed;
#pragma unroll
    for (int u = 0; u < D; ++u) {
      if (j0 + u <= k) {
        const unsigned a = max((unsigned)__double2hiint(v[u].x) << 1, (unsigned)__double2hiint(v[u].y) << 1);
        const unsigned b = max((unsigned)__double2hiint(v[u].z) << 1, (unsigned)__double2hiint(v[u].w) << 1);
        nu = max(nu, (int)(a >> 21) + coef[j0 + u].be);
        nd = max(nd, (int)(b >> 21) + coef[j0 + u].be);
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) sum[c] = fx::shr_round(sum[c], c < 2 ? nu - beu : nd - bed);
    beu = nu;
    bed = nd;
#pragma unroll
    for (int g = 0; g < D; g += 4) {
      fx::Acc acc[4];
#pragma unroll
      for (int u = g; u < g + 4; ++u) {
        if (j0 + u <= k) {
          const FxCoef cf = coef[j0 + u];
          const int bu = max(beu - cf.be, 63), bd = max(bed - cf.be, 63);
          const fx::Limbs x = fx::split(fx::to_fixed<59>(v[u].x, bu)), y = fx::split(fx::to_fixed<59>(v[u].y, bu));
          const fx::Limbs z = fx::split(fx::to_fixed<59>(v[u].z, bd)), w = fx::split(fx::to_fixed<59>(v[u].w, bd));
          acc[0].mac(x, cf.re);
          acc[0].mac(y, cf.mim);
          acc[1].mac(y, cf.re);
          acc[1].mac(x, cf.im);
          acc[2].mac(z, cf.re);
          acc[2].mac(w, cf.mim);
          acc[3].mac(w, cf.re);
          acc[3].mac(z, cf.im);
        }
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) sum[c] += acc[c].template value<30>();
    }
  }
  const int eu = beu - 2044 - 56, ed = bed - 2044 - 56;   // 2^62 of the products' 2^-118
  vec4 o;
  o.x = fx::to_double(sum[0], eu);
  o.y = fx::to_double(sum[1], eu);
  o.z = fx::to_double(sum[2], ed);
  o.w = fx::to_double(sum[3], ed);
  psi[s] = o;
}


// Blocks are dealt to problems in proportion to their size; three CTAs per SM
// (at most 85 registers), so that enough warps keep loads in flight.
static __global__ void __launch_bounds__(256, 3) recombine64(const __grid_constant__ RecombParams rp) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __shared__ FxCoef fc[KMAX + 2];
  __shared__ int k_s, err_s;
  const int b = rp.blk_prob[blockIdx.x];
  const Problem* pr = rp.probs + b;
  DevState* st = pr->st;
  if (threadIdx.x == 0) { k_s = st->k_used; err_s = st->error; }
  if (threadIdx.x <= KMAX) fc[threadIdx.x] = fx_coef(st->coef_re[threadIdx.x], st->coef_im[threadIdx.x]);
  __syncthreads();
  const int lb = blockIdx.x - pr->rblk_begin;
  if (blockIdx.x == 0 && threadIdx.x == 0) *rp.step += 1;   // the next step's fields
  if (err_s) return;                                         // leave psi untouched
  if (lb == 0 && threadIdx.x == 0) {                         // re-arm the next step
    st->stopped = 0;
    st->cur_pass = 1;
    st->redo_left = rp.redo_budget;
  }
  const int k = k_s;
  const size_t n = (size_t)pr->nx * pr->ny, stride = (size_t)pr->rblk_count * blockDim.x;
  vec4* psi = const_cast<vec4*>(pr->psi);
  for (size_t s = (size_t)lb * blockDim.x + threadIdx.x; s < n; s += stride)
    recombine_site_fx<4>(psi, static_cast<const vec4*>(pr->basis), n, s, k, fc);
  asm volatile("griddepcontrol.launch_dependents;");
}

// One time step of one problem in one cooperative launch: as lanczos_step
// (dirac_kernels.cuh), with the passes and the recombination above.
template <int R, int TH, bool DIRI, bool HAS_V, bool ISO>
__global__ void __launch_bounds__(fx_threads<TH>(), 1)
lanczos_step64(const __grid_constant__ LaunchParams lp, const __grid_constant__ CoopArgs ca) {
  constexpr int NT = fx_threads<TH>();
  __shared__ DevState sst;
  __shared__ FxCoef fc_s[KMAX + 2];
  __shared__ double tot[3], shift_s;
  __shared__ int failed;
  const Problem* pr = lp.probs;
  DevState* gst = lp.states;
  const int warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    failed = 0;
    if constexpr (TH == 16) shift_s = pr->shift;
  }
  {
    const unsigned* src = reinterpret_cast<const unsigned*>(gst);
    unsigned* dst = reinterpret_cast<unsigned*>(&sst);
    for (int w = threadIdx.x; w < (int)(sizeof(DevState) / sizeof(unsigned)); w += NT) dst[w] = __ldcg(src + w);
  }
  const int step = __ldcg(lp.step);
  __syncthreads();
  const int max_iter = lp.m + lp.redo_budget;
  int iter = 0;
  while (!sst.stopped && iter < max_iter) {
    const int i = max(1, sst.cur_pass);
    ++iter;
    unsigned long long* slots = ca.packets + (iter & 1) * 6 * (size_t)ca.cap;
    pass_body64<R, TH, DIRI, HAS_V, ISO, true>(lp, &sst, slots, step, (unsigned)iter, &shift_s);
    // the grid totals, in the same order in every CTA
    collect_partials(slots, ca.bar_count, tot, (unsigned)iter, ca.bar, &failed);
    __syncthreads();
    if (failed) {
      if (threadIdx.x == 0) { gst->error = ERR_BARRIER; gst->stopped = 1; }
      return;   // psi untouched; the host reports the timeout
    }
    if (warp == 0) finish_fast(lp, pr, &sst, i, tot[0], tot[1], tot[2], shift_s);
    __syncthreads();
  }
  const int err = sst.error;
  if (!err) {
    // psi <- sum_j C_j q^_j on this CTA's tiles (no CTA reads psi any more)
    if (threadIdx.x <= KMAX) fc_s[threadIdx.x] = fx_coef(sst.coef_re[threadIdx.x], sst.coef_im[threadIdx.x]);
    __syncthreads();
    const int cq = lp.chunk_q, cr = lp.chunk_r;
    const int t_begin = blockIdx.x * cq + min((int)blockIdx.x, cr);
    const int t_end = t_begin + cq + ((int)blockIdx.x < cr ? 1 : 0);
    const size_t n = (size_t)pr->nx * pr->ny;
    const int k = sst.k_used;
    vec4* psi = const_cast<vec4*>(pr->psi);
    for (int tt = t_begin; tt < t_end; ++tt) {
      const int x0 = (tt % pr->tiles_x) * TILE_W, y0 = (tt / pr->tiles_x) * TH;
      for (int e = threadIdx.x; e < TILE_W * TH; e += NT) {
        const int x = x0 + (e & (TILE_W - 1)), y = y0 + e / TILE_W;
        if (x < pr->nx && y < pr->ny)
          recombine_site_fx<4>(psi, static_cast<const vec4*>(pr->basis), n, (size_t)y * pr->nx + x, k, fc_s);
      }
    }
  }
  if (blockIdx.x == 0) {   // publish the state (identical in every CTA), re-armed for the next step
    __syncthreads();
    if (threadIdx.x == 0) {
      if (!err) { sst.stopped = 0; sst.cur_pass = 1; sst.redo_left = lp.redo_budget; }
      *const_cast<int*>(lp.step) = step + 1;
    }
    __syncthreads();
    const unsigned* src = reinterpret_cast<const unsigned*>(&sst);
    unsigned* dst = reinterpret_cast<unsigned*>(gst);
    for (int w = threadIdx.x; w < (int)(sizeof(DevState) / sizeof(unsigned)); w += NT) dst[w] = src[w];
  }
}

}  // namespace dirac
