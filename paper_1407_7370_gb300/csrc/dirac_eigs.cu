// dirac_eigs.cu -- eigenvalue mode of the Dirac Lanczos library (Sec. 2, Sec. 5)
// and the plain Hamiltonian product.
//
// Lanczos on A = H - s (direct) or A = (H - s - sigma)^2 (shift-folded), with
// full reorthogonalisation by classical Gram-Schmidt applied twice (Sec. 2),
// Ritz values of T_k checked every few iterations against the Eq. 9 bound
// |beta_k t_i^k|, and Ritz vectors Q t_i (Eq. 8) on request.
//
// Iteration i (0-based) with basis slots q^_0..q^_i (q_j = s_j q^_j, s_j the
// reciprocal norm of slot j, so no vector is ever rescaled in memory):
//   apply   z = s_i A q^_i - beta_{i-1} s_{i-1} q^_{i-1}  into slot i+1; the
//           prologue turns the norm partials of slot i into beta_{i-1} and s_i
//           and applies the breakdown test
//   twice:  h_j = <q_j, z> for j <= i  (dot + finish: fixed-order sums)
//           z -= sum_j h_j q_j         (update; the second also yields ||z||^2
//                                       partials for beta_i)
//   alpha_i = Re(h_i) summed over both passes.
// Without reorthogonalisation one pass against q_i alone with the real part
// of h_i only (Fig. 1, Eq. 4).
//
// Every sum is taken in a fixed order (per-CTA partials, then one warp), so
// results are bitwise reproducible.  No kernel waits on another CTA.
//
// The Ritz values come from a Sturm-sequence multisection on T_k (four warps
// per eigenvalue, 128 points per round), their vectors from inverse iteration
// with a partially pivoted LU of T_k - theta (two solves, orthogonalised
// within clusters of close values); T_k is scaled by a power of two so that
// the characteristic-polynomial recurrence stays in range.
#include "dirac.h"
#include "dirac_fixed.cuh"
#include "dirac_internal.h"

#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <numeric>
#include <type_traits>
#include <vector>

namespace dirac {
namespace eig {

using v4 = double4_32a;   // one site: (u.re, u.im, d.re, d.im)

constexpr int RITZ_CAP = DIRAC_EIG_RITZ_MAX;   // Ritz values examined per check
constexpr int MAX_ITER = DIRAC_EIG_ITER_MAX;
constexpr int TILE_W = 32;                     // tile width of the product (one warp)
constexpr int CH_MAX = 256;                    // sites per dot-kernel chunk
constexpr double BREAKDOWN_REL = 1e-12;

struct EigDev {
  int breakdown;   // 1 once beta_i <= 1e-12 * scale (invariant subspace)
  int k_final;     // size of T at the breakdown
  int error;       // 1: non-finite value or zero start vector
  int pad;
  double scale;    // max(|alpha_j + s_a|, beta_j) so far, s_a the shift of A
};

struct RitzOut {
  int k;           // size of T_k
  int n_lo, n_hi;  // eigenvalue indices of T_k in the window (folded: 0, k)
  int n_exam;      // examined: indices n_lo .. n_lo + n_exam - 1
  int breakdown, error, exp2;   // exp2: T was scaled by 2^-exp2
  int pad;
  double beta_last;             // beta_k of Eq. 9
  double g_lo, g_hi;            // Gershgorin interval of the scaled T
  double theta[RITZ_CAP];
  double bound[RITZ_CAP];
};

__device__ __forceinline__ double wsum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Largest |x| of a vector, by the upper 31 bits of its numbers (their exponent
// and 20 bits): max over a block, then one atomic
__device__ __forceinline__ unsigned mag(double x) { return (unsigned)__double2hiint(x) << 1; }
__device__ __forceinline__ unsigned mag4(const v4& v) { return max(max(mag(v.x), mag(v.y)), max(mag(v.z), mag(v.w))); }
__device__ void block_max(unsigned m, unsigned* out) {
  __shared__ unsigned red[32];
  m = __reduce_max_sync(0xffffffffu, m);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) red[warp] = m;
  __syncthreads();
  if (warp == 0) {
    m = __reduce_max_sync(0xffffffffu, lane < (int)(blockDim.x >> 5) ? red[lane] : 0u);
    if (lane == 0) atomicMax(out, m);
  }
}
// exponent field of a recorded maximum (192 and below count as zero)
__device__ __forceinline__ int max_field(unsigned m) { return max((int)(m >> 21), 192); }

__device__ __forceinline__ double wmax(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

__device__ __forceinline__ double wmin(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// ---------------------------------------------------------------------------
// A q: the Hamiltonian of Eq. 12 (electron, central differences) minus e0
// ---------------------------------------------------------------------------
struct ApplyArgs {
  int nx, ny;
  double kx, ky;        // c / (2h) (order 2) or c / (12h) (order 4)
  double cax, cay;      // c A (p - qA = p + A for the electron)
  double au, ad;        // mc^2 - e0, -mc^2 - e0
  const double* V;      // potential energy or null
  const v4* in;
  const v4* sub;        // q^_{i-1} (Lanczos mode) or null
  v4* out;
  EigDev* ed;           // null: plain product out = (H - e0) in
  const double* norm_part;
  int n_part;
  double* beta;
  double* s;
  int iter;
  int prologue;         // 1: s_i and beta_{i-1} from norm_part, breakdown test, scale by s_i
  unsigned* vmax;       // largest number of `out` (or null)
};

template <bool DIRI, class T>
__device__ __forceinline__ void load_site(const v4* __restrict__ in, int gx, int gy, int nx, int ny,
                                          T (&o)[4]) {
  if (DIRI) {
    if (gx < 0 || gx >= nx || gy < 0 || gy >= ny) { o[0] = o[1] = o[2] = o[3] = 0.0; return; }
  } else {
    gx = ((gx % nx) + nx) % nx;
    gy = ((gy % ny) + ny) % ny;
  }
  const v4 v = in[(size_t)gy * nx + gx];
  o[0] = (T)v.x; o[1] = (T)v.y; o[2] = (T)v.z; o[3] = (T)v.w;
}

// The scalars of a product inside the Lanczos iteration: s_i (the scale of the
// input) and the coefficient of q^_{i-1}, from the norm partials of slot i, with
// the breakdown test; false once the iteration has ended.  A plain product leaves
// s_in = 1, csub = 0.  Every thread of the block takes the same branch.
__device__ __forceinline__ bool apply_scalars(const ApplyArgs& a, double& s_in, double& csub) {
  __shared__ double sh_nrm;
  __shared__ int sh_stop;
  s_in = 1.0;
  csub = 0.0;
  if (!a.ed) return true;
  // one read of the flags per block (the lead CTA of a prologue launch may set
  // them meanwhile)
  if (threadIdx.x == 0) sh_stop = a.ed->breakdown | a.ed->error;
  if (a.prologue && threadIdx.x < 32) {
    double nrm = 0.0;
    for (int c = threadIdx.x; c < a.n_part; c += 32) nrm += a.norm_part[c];
    nrm = wsum(nrm);
    if (threadIdx.x == 0) sh_nrm = nrm;
  }
  __syncthreads();
  if (sh_stop) return false;
  const int i = a.iter;
  if (a.prologue) {
    const double bt = sqrt(sh_nrm);          // ||q^_i||: beta_{i-1}, or ||start|| at i = 0
    const bool lead = blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0;
    if (!isfinite(bt) || !(bt > 0.0)) {
      if (lead) a.ed->error = 1;
      return false;
    }
    if (i >= 1 && bt <= BREAKDOWN_REL * a.ed->scale) {
      if (lead) { a.ed->breakdown = 1; a.ed->k_final = i; a.beta[i - 1] = bt; }
      return false;
    }
    s_in = 1.0 / bt;
    if (i >= 1 && a.sub) csub = bt * a.s[i - 1];
    if (lead) {
      a.s[i] = s_in;
      if (i >= 1) a.beta[i - 1] = bt;
    }
  } else if (a.sub && i >= 1) {
    csub = a.beta[i - 1] * a.s[i - 1];
  }
  return true;
}

// One site of the product in floating point.  T = double: FP64.  T = float: the
// mixed-precision product -- the off-diagonal part (differences and vector
// potential) on FP32 copies of the vector, the diagonal (m c^2 + V - e0 and
// -m c^2 + V - e0) on the FP64 vector itself, so that the -2 m c^2 of the lower
// components adds no u32 * 2 m c^2 rounding to the product; the Lanczos
// combination s_i y - c q^_{i-1} in FP64.
template <int R, bool DIRI, bool HAS_V, class T>
__device__ __forceinline__ v4 apply_site(const ApplyArgs& a, int x, int y, double s_in, double csub) {
  const int nx = a.nx, ny = a.ny;
  T C[4], xp[4], xm[4], yp[4], ym[4], dxv[4], dyv[4];
  double C64[4];
  load_site<DIRI>(a.in, x, y, nx, ny, C64);
#pragma unroll
  for (int q = 0; q < 4; ++q) C[q] = (T)C64[q];
  load_site<DIRI>(a.in, x + 1, y, nx, ny, xp);
  load_site<DIRI>(a.in, x - 1, y, nx, ny, xm);
  load_site<DIRI>(a.in, x, y + 1, nx, ny, yp);
  load_site<DIRI>(a.in, x, y - 1, nx, ny, ym);
#pragma unroll
  for (int q = 0; q < 4; ++q) { dxv[q] = xp[q] - xm[q]; dyv[q] = yp[q] - ym[q]; }
  if constexpr (R == 2) {
    load_site<DIRI>(a.in, x + 2, y, nx, ny, xp);
    load_site<DIRI>(a.in, x - 2, y, nx, ny, xm);
    load_site<DIRI>(a.in, x, y + 2, nx, ny, yp);
    load_site<DIRI>(a.in, x, y - 2, nx, ny, ym);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      dxv[q] = fma(T(8), dxv[q], xm[q] - xp[q]);
      dyv[q] = fma(T(8), dyv[q], ym[q] - yp[q]);
    }
  }
  const size_t idx = (size_t)y * nx + x;
  double au = a.au, ad = a.ad;
  if (HAS_V) {
    const double v = a.V[idx];
    au += v;
    ad += v;
  }
  const T kx = (T)a.kx, ky = (T)a.ky, cax = (T)a.cax, cay = (T)a.cay;
  // off-diagonal part
  T ot[4];
  // upper: c[-i D_x d - D_y d + (A_x - i A_y) d]
  ot[0] = kx * dxv[3] - ky * dyv[2] + cax * C[2] + cay * C[3];
  ot[1] = -kx * dxv[2] - ky * dyv[3] + cax * C[3] - cay * C[2];
  // lower: c[-i D_x u + D_y u + (A_x + i A_y) u]
  ot[2] = kx * dxv[1] + ky * dyv[0] + cax * C[0] - cay * C[1];
  ot[3] = -kx * dxv[0] + ky * dyv[1] + cax * C[1] + cay * C[0];
  // plus the diagonal: (mc^2+V-e0) u and (-mc^2+V-e0) d
  const double o[4] = {fma(au, C64[0], (double)ot[0]), fma(au, C64[1], (double)ot[1]),
                       fma(ad, C64[2], (double)ot[2]), fma(ad, C64[3], (double)ot[3])};
  v4 r;
  if (csub != 0.0) {
    const v4 sv = a.sub[idx];
    r.x = fma(s_in, o[0], -csub * sv.x);
    r.y = fma(s_in, o[1], -csub * sv.y);
    r.z = fma(s_in, o[2], -csub * sv.z);
    r.w = fma(s_in, o[3], -csub * sv.w);
  } else {
    r.x = s_in * o[0]; r.y = s_in * o[1]; r.z = s_in * o[2]; r.w = s_in * o[3];
  }
  return r;
}

// The mixed-precision product, one thread per site
template <int R, bool DIRI, bool HAS_V>
__global__ void __launch_bounds__(256) eig_apply32(const ApplyArgs a) {
  double s_in, csub;
  if (!apply_scalars(a, s_in, csub)) return;
  // threads beyond the grid's edge repeat its last site and store nothing
  const int xt = blockIdx.x * 32 + (threadIdx.x & 31), yt = blockIdx.y * 8 + (threadIdx.x >> 5);
  const bool valid = xt < a.nx && yt < a.ny;
  const int x = min(xt, a.nx - 1), y = min(yt, a.ny - 1);
  const v4 r = apply_site<R, DIRI, HAS_V, float>(a, x, y, s_in, csub);
  if (valid) a.out[(size_t)y * a.nx + x] = r;
  if (a.vmax) block_max(valid ? mag4(r) : 0u, a.vmax);
}

// The FP64 product in fixed point (dirac_fixed.cuh), a tile of 32 x 16 sites per
// CTA, four rows per thread (32 x 4 and one row on small grids), LANCZOS: with the
// scale and q^_{i-1} of an iteration; as in the FP64 Lanczos pass (dirac_pass64.cuh):
// exponents of the tile's upper and lower components and of q^_{i-1}, the tile
// and its halo as 59-bit numbers in shared memory, each row of
// the operator one sum of products, then times s_i.  Of the FP64 pipe only the
// four conversions of the result are left; with some 40 multiply-adds a site it
// bounded the product (2048^2 with V: 342 us, 0.9 TB/s; now 110 us, 2.7 TB/s,
// bound by latency and instruction issue).  Tiles with numbers that are not
// finite, or none above 2^-894, take the floating-point form.  So do tiles whose
// V is so uneven that the row of its smallest |V| would have to be computed at a
// scale more than AP_V_LOSS bits above its own terms (a wall, a spike): there the
// shared scale costs the digits that FP64 keeps at the sites of small V.
constexpr int AP_WARPS = 4, AP_THREADS = 32 * AP_WARPS, AP_SLOTS = 16;
constexpr int AP_V_LOSS = 3;   // of the 6 bits more than FP64's 53 that the numbers of a tile have

template <int R, bool DIRI, bool HAS_V, int AP_RPT, bool LANCZOS>
__global__ void __launch_bounds__(AP_THREADS, LANCZOS ? 4 : 5) eig_apply64(const ApplyArgs a) {
  constexpr int AP_TH = AP_WARPS * AP_RPT;
  constexpr int W = TILE_W + 2 * R, F = fx::ROW_BITS;
  constexpr int NH_ROW = 2 * R * TILE_W, NH = NH_ROW + 2 * R * AP_TH, HPT = (NH + AP_THREADS - 1) / AP_THREADS;
  __shared__ __align__(16) longlong2 sq[2][(AP_TH + 2 * R) * W];
  __shared__ int2 kt[AP_SLOTS];
  __shared__ unsigned emax[6];   // largest of u, d, q^_{i-1}'s u and d, |V|, and the complement of the smallest |V|
  double s_in = 1.0, csub = 0.0;
  if (LANCZOS && !apply_scalars(a, s_in, csub)) return;
  if (threadIdx.x < 6) emax[threadIdx.x] = 0u;
  __syncthreads();
  const int nx = a.nx, ny = a.ny;
  const int tx = threadIdx.x & 31, tg = threadIdx.x >> 5, lane = tx;
  const int x0 = blockIdx.x * TILE_W, y0 = blockIdx.y * AP_TH, r0 = tg * AP_RPT;
  const bool full = x0 + TILE_W <= nx && y0 + AP_TH <= ny;
  const int rows_in = x0 + tx < nx ? ny - (y0 + r0) : 0;              // row k is in the grid if k < rows_in
  const size_t idx0 = (size_t)(y0 + r0) * nx + (x0 + tx);             // used where in the grid
  const bool has_sub = LANCZOS && csub != 0.0;
  double q[AP_RPT][4], p[AP_RPT][4], hq[HPT][4], V[AP_RPT];
  int hat[HPT];
#pragma unroll
  for (int k = 0; k < AP_RPT; ++k) {
    V[k] = HAS_V && k < rows_in ? a.V[idx0 + (size_t)k * nx] : 0.0;
    // sites beyond the grid's edge are halo of the sites inside
    if (full) {
      const v4 v = a.in[idx0 + (size_t)k * nx];
      q[k][0] = v.x; q[k][1] = v.y; q[k][2] = v.z; q[k][3] = v.w;
    } else {
      load_site<DIRI>(a.in, x0 + tx, y0 + r0 + k, nx, ny, q[k]);
    }
    p[k][0] = p[k][1] = p[k][2] = p[k][3] = 0.0;
    if (has_sub && k < rows_in) {
      const v4 v = a.sub[idx0 + (size_t)k * nx];
      p[k][0] = v.x; p[k][1] = v.y; p[k][2] = v.z; p[k][3] = v.w;
    }
  }
#pragma unroll
  for (int u = 0; u < HPT; ++u) {
    const int h = threadIdx.x + u * AP_THREADS;
    hat[u] = -1;
    hq[u][0] = hq[u][1] = hq[u][2] = hq[u][3] = 0.0;
    if (h < NH) {
      int hrow, hcol;
      if (h < NH_ROW) {                 // rows above / below
        const int r = h / TILE_W;
        hrow = (r < R) ? r : AP_TH + r;
        hcol = (h % TILE_W) + R;
      } else {                          // columns left / right
        const int h2 = h - NH_ROW;
        hrow = h2 / (2 * R) + R;
        const int c = h2 % (2 * R);
        hcol = (c < R) ? c : TILE_W + c;
      }
      hat[u] = hrow * W + hcol;
      load_site<DIRI>(a.in, x0 + hcol - R, y0 + hrow - R, nx, ny, hq[u]);
    }
  }
  unsigned m0 = 0u, m1 = 0u, m2 = 0u, m3 = 0u;
#pragma unroll
  for (int u = 0; u < HPT; ++u) {
    m0 = max(m0, max(mag(hq[u][0]), mag(hq[u][1])));
    m1 = max(m1, max(mag(hq[u][2]), mag(hq[u][3])));
  }
#pragma unroll
  for (int k = 0; k < AP_RPT; ++k) {
    m0 = max(m0, max(mag(q[k][0]), mag(q[k][1])));
    m1 = max(m1, max(mag(q[k][2]), mag(q[k][3])));
    m2 = max(m2, max(mag(p[k][0]), mag(p[k][1])));
    m3 = max(m3, max(mag(p[k][2]), mag(p[k][3])));
  }
  m0 = __reduce_max_sync(0xffffffffu, m0);
  m1 = __reduce_max_sync(0xffffffffu, m1);
  m2 = __reduce_max_sync(0xffffffffu, m2);
  m3 = __reduce_max_sync(0xffffffffu, m3);
  if (lane < 4) atomicMax(&emax[lane], lane == 0 ? m0 : lane == 1 ? m1 : lane == 2 ? m2 : m3);
  if constexpr (HAS_V) {
    unsigned vhi = 0u, vlo = 0u;
#pragma unroll
    for (int k = 0; k < AP_RPT; ++k) {
      vhi = max(vhi, mag(V[k]));                       // (zero outside the grid)
      if (k < rows_in) vlo = max(vlo, ~mag(V[k]));
    }
    vhi = __reduce_max_sync(0xffffffffu, vhi);
    vlo = __reduce_max_sync(0xffffffffu, vlo);
    if (lane < 2) atomicMax(&emax[4 + lane], lane == 0 ? vhi : vlo);
  }
  __syncthreads();
  // a tile of zeros is exact in fixed point; a largest number that is not finite
  // or below the clamp is not
  bool plain = false;
#pragma unroll
  for (int c = 0; c < 4; ++c) plain = plain || (emax[c] >> 21) == 0x7ffu || (emax[c] != 0u && (emax[c] >> 21) < 128u);
  int be[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) be[c] = max((int)(emax[c] >> 21), 128);
  const int vbe = HAS_V ? (int)(emax[4] >> 21) : 0;   // exponent field of the tile's largest |V| (0: V = 0)
  if constexpr (HAS_V) {
    // the scale that V asks for against that of the other terms with the smallest |V|
    const int vmin = (int)(~emax[5] >> 21), ek = max(fx::exp_field(a.kx), fx::exp_field(a.ky)) + (R == 1 ? 0 : 3);
    const int eo = max(ek, max(fx::exp_field(a.cax), fx::exp_field(a.cay)));
    const int es = has_sub ? fx::exp_field(csub) - fx::exp_field(s_in) + 1023 : -4096;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int others = max(max(vmin, fx::exp_field(h ? a.ad : a.au)) + be[h], max(eo + be[1 - h], es + be[2 + h]));
      plain = plain || (vbe && vbe + be[h] > others + AP_V_LOSS);
    }
  }
  if (plain) {
    unsigned m = 0u;
    for (int k = 0; k < AP_RPT; ++k) {
      if (k >= rows_in) break;
      const v4 o = apply_site<R, DIRI, HAS_V, double>(a, x0 + tx, y0 + r0 + k, s_in, csub);
      a.out[idx0 + (size_t)k * nx] = o;
      m = max(m, mag4(o));
    }
    __syncwarp();
    if (a.vmax) block_max(m, a.vmax);
    return;
  }
  const int at0 = (r0 + R) * W + tx + R;
#pragma unroll
  for (int k = 0; k < AP_RPT; ++k) {
    sq[0][at0 + k * W] = make_longlong2(fx::to_fixed<F>(q[k][0], be[0]), fx::to_fixed<F>(q[k][1], be[0]));
    sq[1][at0 + k * W] = make_longlong2(fx::to_fixed<F>(q[k][2], be[1]), fx::to_fixed<F>(q[k][3], be[1]));
  }
#pragma unroll
  for (int u = 0; u < HPT; ++u) {
    if (hat[u] >= 0) {
      sq[0][hat[u]] = make_longlong2(fx::to_fixed<F>(hq[u][0], be[0]), fx::to_fixed<F>(hq[u][1], be[0]));
      sq[1][hat[u]] = make_longlong2(fx::to_fixed<F>(hq[u][2], be[1]), fx::to_fixed<F>(hq[u][3], be[1]));
    }
  }
  if (tg == 0) {
    // coefficients as 60-bit fractions of the row's largest term: slots 0
    // diagonal, 1 kx, 2 ky, 3 c A_x, 4 c A_y, 5 of q^_{i-1} (before the scaling by
    // s_i), 6 V (its exponent alone), 7 the scale, of the upper and the lower row
    const int j = lane & 7, ch = (lane >> 3) & 1;
    double c = 0.0;
    if (j == 0) c = ch ? a.ad : a.au;
    if (j == 1) c = R == 1 ? a.kx : 8.0 * a.kx;   // of the inner difference
    if (j == 2) c = R == 1 ? a.ky : 8.0 * a.ky;
    if (j == 3) c = a.cax;
    if (j == 4) c = a.cay;
    if (j == 5) c = -csub / s_in;
    const int xe = j == 6 ? vbe : fx::exp_field(c);
    const int be_x = (j == 0 || j == 6) ? be[ch] : (j == 5 ? be[2 + ch] : be[1 - ch]);
    int sc = xe ? xe + be_x : 0;
    sc = max(sc, __shfl_xor_sync(0xffffffffu, sc, 1));
    sc = max(sc, __shfl_xor_sync(0xffffffffu, sc, 2));
    sc = max(sc, __shfl_xor_sync(0xffffffffu, sc, 4));
    if (lane < AP_SLOTS) {
      const fx::Limbs l = fx::split(fx::to_fixed<60>(c, max(sc - be_x, 63)));
      kt[lane] = j == 7 ? make_int2(sc, 0) : make_int2(l.hi, l.lo);
    }
  }
  __syncthreads();
  const int es = fx::exp_field(s_in);
  const fx::Limbs ks = fx::split(fx::to_fixed<60>(s_in, es));
  const bool scaled = LANCZOS && s_in != 1.0;
  unsigned m = 0u;
  long long pot[AP_RPT];      // V as 60-bit fractions of the tile's largest |V|
#pragma unroll
  for (int k = 0; k < AP_RPT; ++k) pot[k] = HAS_V ? fx::to_fixed<60>(V[k], max(vbe, 63)) : 0;
  auto half = [&](auto half_c) {
    constexpr int HALF = decltype(half_c)::value;
    const longlong2* const own = sq[HALF] + at0;
    const longlong2* const oth = sq[1 - HALF] + at0;
    const int2* const kc = kt + 8 * HALF;
    auto coef = [&](int j) { const int2 v = kc[j]; return fx::Limbs{v.x, v.y}; };
    const int sc = kc[7].x;
    const int texp = sc - 2044 - F + (fx::ROW_SHIFT - 28) + (scaled ? es - 1022 : 0);
    const bool normal = texp >= -1022 && texp <= 960;      // no result leaves the normal range
    const int vsh = min(max(sc - be[HALF] - max(vbe, 63), 0), 63);   // V's scale within the row's
    longlong2 col[AP_RPT + 2 * R];
#pragma unroll
    for (int j = 0; j < AP_RPT + 2 * R; ++j) col[j] = oth[(j - R) * W];
#pragma unroll
    for (int k = 0; k < AP_RPT; ++k) {
      const longlong2* const row = oth + k * W;
      const longlong2 xl = row[-1], xr = row[1], cv = own[k * W];
      long long hxr = xl.x - xr.x, hxi = xr.y - xl.y;          // -D_x re, D_x im
      long long hyr = col[k + R + 1].x - col[k + R - 1].x, hyi = col[k + R + 1].y - col[k + R - 1].y;
      if constexpr (R == 2) {
        const longlong2 xl2 = row[-2], xr2 = row[2];
        hxr -= fx::eighth(xl2.x - xr2.x);
        hxi -= fx::eighth(xr2.y - xl2.y);
        hyr -= fx::eighth(col[k + 2 * R].x - col[k].x);
        hyi -= fx::eighth(col[k + 2 * R].y - col[k].y);
      }
      fx::Acc s0, s1;
      s0.mac(fx::split(hxi), coef(1));
      s1.mac(fx::split(hxr), coef(1));
      s0.mac(fx::split(HALF ? hyr : -hyr), coef(2));
      s1.mac(fx::split(HALF ? hyi : -hyi), coef(2));
      const fx::Limbs c0 = fx::split(cv.x), c1 = fx::split(cv.y);
      s0.mac(c0, coef(0));
      s1.mac(c1, coef(0));
      if (a.cax != 0.0) {
        s0.mac(fx::split(col[k + R].x), coef(3));
        s1.mac(fx::split(col[k + R].y), coef(3));
      }
      if (a.cay != 0.0) {
        s0.mac(fx::split(HALF ? -col[k + R].y : col[k + R].y), coef(4));
        s1.mac(fx::split(HALF ? col[k + R].x : -col[k + R].x), coef(4));
      }
      if (has_sub) {
        s0.mac(fx::split(fx::to_fixed<F>(p[k][2 * HALF], be[2 + HALF])), coef(5));
        s1.mac(fx::split(fx::to_fixed<F>(p[k][2 * HALF + 1], be[2 + HALF])), coef(5));
      }
      if constexpr (HAS_V) {
        const fx::Limbs kv = fx::split(pot[k] >> vsh);
        s0.mac(c0, kv);
        s1.mac(c1, kv);
      }
      long long v0 = s0.template value<fx::ROW_SHIFT>(), v1 = s1.template value<fx::ROW_SHIFT>();
      if (scaled) {
        fx::Acc t0, t1;
        t0.mac(fx::split(v0), ks);
        t1.mac(fx::split(v1), ks);
        v0 = t0.template value<28>();
        v1 = t1.template value<28>();
      }
      if (k < rows_in) {
        const double2 o = normal ? make_double2(fx::to_double(v0, texp), fx::to_double(v1, texp))
                                 : make_double2(fx::scale2((double)v0, texp), fx::scale2((double)v1, texp));
        reinterpret_cast<double2*>(a.out + idx0 + (size_t)k * nx)[HALF] = o;
        m = max(m, max(mag(o.x), mag(o.y)));
      }
    }
  };
  half(std::integral_constant<int, 0>{});
  half(std::integral_constant<int, 1>{});
  if (a.vmax) block_max(m, a.vmax);
}

// ---------------------------------------------------------------------------
// h_j = <q^_j, z> for j = j0..j1, and ||z||^2 (z is the basis slot after j1):
// per-CTA partials, the z chunk staged in shared memory, one warp per vector at
// a time.
//
// The products are 58-bit fixed point (dirac_fixed.cuh): in FP64 the eight
// multiply-adds per site and vector occupied a sub-partition for 512 cycles,
// against the 190 in which its share of the memory bandwidth delivers the vector;
// conversion and limb products take about 290.  z has an exponent per site, a
// vector one per 128 sites (its chunk's largest so far), so that a flat floor under
// a peak keeps its share of the sum: a product is off by 2^-58 of the largest
// numbers of its 128 or 256 sites for its truncation and, with either sign, up to
// 2^-54 for the lower limbs' product; over a chunk that is about 2^-53 of its part
// of the norms, the rounding of one FP64 operation.  Chunks are added in FP64.  (With
// one exponent per vector a floor of 2^-29 under a peak, 2^-37 of the squared norm,
// was lost: three vectors were orthogonal to 5e-12; the exponents cost 2.5 % of the
// run, keeping the lower limbs' products instead 7 %.)  The FP64 pipe takes every
// third vector meanwhile, at FP64_SHARE's cost ratio (512 to 290): without that
// share a run was 5 % longer.  100 iterations on 1024^2 with two orthogonalisations:
// 327 ms in FP64 alone, now 149; the reads of both kernels take 100 at the copy
// bandwidth.
// ---------------------------------------------------------------------------
constexpr int FP64_SHARE = 3;   // one vector in so many goes to the FP64 pipe
__device__ __forceinline__ bool fp64_vector(int jj, int nw) { return (jj / nw + jj % nw) % FP64_SHARE == FP64_SHARE - 1; }

struct DotArgs {
  const v4* basis;
  long long n;
  int j0, j1;           // z is slot j1 + 1
  int cs;               // sites per chunk (multiple of 32, <= CH_MAX)
  double2* part;        // [j - j0][CTA], the last row ||z||^2
  const EigDev* ed;
};

// A warp takes four rows of 32 numbers at a time: four pieces of one vector's
// chunk, or (SHORT: chunks of 32 sites, small grids) one piece of each of four
// vectors, so that as many loads are in flight.
template <bool SHORT>
__global__ void __launch_bounds__(256, 4) eig_dot(const DotArgs a) {
  extern __shared__ __align__(32) unsigned char smem[];
  __shared__ unsigned zmax[8];
  if (a.ed->breakdown | a.ed->error) return;
  int4* const zu = reinterpret_cast<int4*>(smem);       // limbs of (x, y), then of (z, w)
  int4* const zd = zu + a.cs;
  v4* const zf = reinterpret_cast<v4*>(zd + a.cs);
  int* const zk = reinterpret_cast<int*>(zf + a.cs);     // exponent of the chunk's z less that of the site
  double2* acc = reinterpret_cast<double2*>(zk + a.cs);
  const int count = a.j1 - a.j0 + 2;
  for (int t = threadIdx.x; t < count; t += blockDim.x) acc[t] = make_double2(0.0, 0.0);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int zbe = 0;                                // exponent field of the largest number of z's chunk
  const long long nchunks = (a.n + a.cs - 1) / a.cs;
  const v4* const z = a.basis + (size_t)(a.j1 + 1) * a.n;
  // limb products of one number of q^ with its z, and the sums of a batch
  auto products = [&](const v4& v, int t, int chunk_be, fx::Acc& ar, fx::Acc& ai, fx::Acc& am) {
    const int be = chunk_be + zk[t];
    const fx::Limbs x = fx::split(fx::to_fixed<58>(v.x, be)), y = fx::split(fx::to_fixed<58>(v.y, be));
    const fx::Limbs z = fx::split(fx::to_fixed<58>(v.z, be)), w = fx::split(fx::to_fixed<58>(v.w, be));
    const int4 s0 = zu[t], s1 = zd[t];
    const fx::Limbs zx{s0.x, s0.y}, zy{s0.z, s0.w}, zz{s1.x, s1.y}, zw{s1.z, s1.w};
    ar.mac(x, zx);
    ar.mac(y, zy);
    ar.mac(z, zz);
    ar.mac(w, zw);
    ai.mac(x, zy);
    ai.mac(z, zw);
    am.mac(y, zx);
    am.mac(w, zz);
  };
  // units: (2^(be - 1022 - 58)) (2^(zbe - 1022 - 58)) 2^60
  auto add_sums = [&](int jj, int be, long long re, long long im) {
    const fx::WarpSum sr = fx::warp_sum(re), si = fx::warp_sum(im);
    if (lane < 2) reinterpret_cast<double*>(acc + jj)[lane] += fx::scale2(fx::to_double(lane == 0 ? sr : si), be + zbe - 2100);
  };
  v4 none;
  none.x = none.y = none.z = none.w = 0.0;
  for (long long ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
    const long long base = ch * a.cs;
    const int len = (int)min((long long)a.cs, a.n - base);
    const int t = threadIdx.x;                // cs <= CH_MAX threads
    const v4 v = t < len ? z[base + t] : none;
    const unsigned m = __reduce_max_sync(0xffffffffu, mag4(v));
    __syncthreads();                          // the chunk before has been read
    if (lane == 0) zmax[warp] = m;
    __syncthreads();
    zbe = max_field(__reduce_max_sync(0xffffffffu, lane < nw ? zmax[lane] : 0u));
    if (t < a.cs) {
      const int sbe = max_field(mag4(v));
      const fx::Limbs x = fx::split(fx::to_fixed<58>(v.x, sbe)), y = fx::split(fx::to_fixed<58>(v.y, sbe));
      const fx::Limbs u = fx::split(fx::to_fixed<58>(v.z, sbe)), w = fx::split(fx::to_fixed<58>(v.w, sbe));
      zu[t] = make_int4(x.hi, x.lo, y.hi, y.lo);
      zd[t] = make_int4(u.hi, u.lo, w.hi, w.lo);
      zf[t] = v;
      zk[t] = zbe - sbe;
    }
    __syncthreads();
    if constexpr (SHORT) {
      for (int j0 = 4 * warp; j0 < count; j0 += 4 * nw) {
        const v4* __restrict__ q = a.basis + (size_t)(a.j0 + j0) * a.n + base;
        v4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = lane < len && j0 + u < count ? q[(size_t)u * a.n + lane] : none;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int jj = j0 + u;
          if (jj < count) {
            const int be = max_field(__reduce_max_sync(0xffffffffu, mag4(v[u])));
            fx::Acc ar, ai, am;
            products(v[u], lane, be, ar, ai, am);
            add_sums(jj, be, ar.template value<28>(), ai.template value<28>() - am.template value<28>());
          }
        }
      }
    } else {
      for (int jj = warp; jj < count; jj += nw) {
        const v4* __restrict__ q = a.basis + (size_t)(a.j0 + jj) * a.n + base;
        if (fp64_vector(jj, nw)) {
          double re = 0.0, im = 0.0;
          for (int t0 = 0; t0 < len; t0 += 128) {
            v4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int t = t0 + 32 * u + lane;
              v[u] = t < len ? q[t] : none;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const v4 zz = zf[min(t0 + 32 * u + lane, a.cs - 1)];
              re = fma(v[u].x, zz.x, fma(v[u].y, zz.y, fma(v[u].z, zz.z, fma(v[u].w, zz.w, re))));
              im = fma(v[u].x, zz.y, fma(-v[u].y, zz.x, fma(v[u].z, zz.w, fma(-v[u].w, zz.z, im))));
            }
          }
          // both sums over the warp with one addition per level: even lanes re, odd lanes im
          double part = (lane & 1 ? im : re) + __shfl_xor_sync(0xffffffffu, lane & 1 ? re : im, 1);
#pragma unroll
          for (int o = 16; o > 1; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
          if (lane < 2) reinterpret_cast<double*>(acc + jj)[lane] += part;
          continue;
        }
        int be = 0;
        long long re = 0, im = 0;   // at most 32 products below 2^56 in units of 2^60
        for (int t0 = 0; t0 < len; t0 += 128) {
          v4 v[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int t = t0 + 32 * u + lane;
            v[u] = t < len ? q[t] : none;
          }
          const int nb = max_field(__reduce_max_sync(0xffffffffu, max(max(mag4(v[0]), mag4(v[1])), max(mag4(v[2]), mag4(v[3])))));
          if (nb > be) {
            re = fx::shr_round(re, nb - be);
            im = fx::shr_round(im, nb - be);
            be = nb;
          }
          fx::Acc ar, ai, am;   // at most 16 products each: cross terms below 2^62
#pragma unroll
          for (int u = 0; u < 4; ++u)
            products(v[u], min(t0 + 32 * u + lane, a.cs - 1), be, ar, ai, am);   // (zero beyond the end)
          re += ar.template value<28>();
          im += ai.template value<28>() - am.template value<28>();
        }
        add_sums(jj, be, re, im);
      }
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < count; t += blockDim.x) a.part[(size_t)t * gridDim.x + blockIdx.x] = acc[t];
}

// <q, z> of one vector in FP64: per-CTA partials (the folded mode's Rayleigh quotients)
__global__ void __launch_bounds__(256) eig_inner(const v4* q, const v4* z, long long n, double2* part) {
  double re = 0.0;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += stride) {
    const v4 a = q[t], b = z[t];
    re = fma(a.x, b.x, fma(a.y, b.y, fma(a.z, b.z, fma(a.w, b.w, re))));
  }
  __shared__ double red[32];
  re = wsum(re);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) red[warp] = re;
  __syncthreads();
  if (warp == 0) {
    re = wsum(lane < (int)(blockDim.x >> 5) ? red[lane] : 0.0);
    if (lane == 0) part[blockIdx.x] = make_double2(re, 0.0);
  }
}

// ---------------------------------------------------------------------------
// grid sums of the dot partials -> update coefficients, alpha_i
// ---------------------------------------------------------------------------
struct FinishArgs {
  const double2* part;
  int n_cta;
  int j0, j1;
  int iter, pass, last, reorth;
  const double* s;
  double2* coef;        // coefficient of q^_j in the update: s_j h_j
  double* alpha;
  const double* beta;
  EigDev* ed;
  double ashift;        // shift of A for the breakdown scale (s direct, 0 folded)
  const unsigned* vmax;
  int4* rec;            // update record of q^_j (eig_update)
};

// A coefficient of the update below this part of ||z|| (by |h_j|) is applied in
// FP32, in sums of at most FP32_RUN vectors that are then added in FP64.  Such a
// sum's terms are at most 2^-38 ||z|| each, so that its 256 roundings come to at most
// 256 2^-24 64 2^-38 ||z||, 2^-55 ||z|| a vector (the truncation of the numbers, 2^-23
// of a term, is far less): an eighth of what the two roundings of the FP64
// multiply-adds may come to, however many vectors there are.  After the first
// orthogonalisation, and for all but the last one or two vectors before it, the
// coefficients are far smaller.  (Runs of 32 vectors made the kernel 5 % slower.)
constexpr double SMALL_COEF = 0x1p-38;
constexpr int FP32_RUN = 128;

__global__ void __launch_bounds__(256) eig_dot_finish(const FinishArgs a) {
  if (a.ed->breakdown | a.ed->error) return;
  const int lane = threadIdx.x & 31;
  const int jj = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  if (jj > a.j1 - a.j0) return;
  double re = 0.0, im = 0.0;
  const double2* p = a.part + (size_t)jj * a.n_cta;
  for (int c = lane; c < a.n_cta; c += 32) { re += p[c].x; im += p[c].y; }
  double zz = 0.0;   // ||z||^2, from the row after the last vector's
  const double2* pz = a.part + (size_t)(a.j1 - a.j0 + 1) * a.n_cta;
  for (int c = lane; c < a.n_cta; c += 32) zz += pz[c].x;
  re = wsum(re);
  im = wsum(im);
  zz = wsum(zz);
  if (lane != 0) return;
  const int j = a.j0 + jj;
  const double sj = a.s[j];
  const double hr = sj * re;                      // h_j = <q_j, z>
  const double hi = a.reorth ? sj * im : 0.0;     // Fig. 1 removes alpha_i q_i, alpha real
  a.coef[jj] = make_double2(sj * hr, sj * hi);
  {
    const unsigned mz = a.vmax[3 * (a.j1 + 1) + a.pass], mq = a.vmax[3 * j + 2];
    const int big = !(hr * hr + hi * hi <= SMALL_COEF * SMALL_COEF * zz);
    const int de = max_field(mq) - max_field(mz);
    a.rec[jj] = make_int4(__float_as_int((float)fx::scale2(sj * hr, de)), __float_as_int((float)fx::scale2(sj * hi, de)),
                          max_field(mq), big);
    if ((mz >> 21) == 0x7ffu || (mq >> 21) == 0x7ffu) a.ed->error = 1;   // not finite
  }
  if (j == a.iter) {
    if (!isfinite(hr) || !isfinite(hi)) a.ed->error = 1;
    const double al = (a.pass == 0 ? 0.0 : a.alpha[j]) + hr;
    a.alpha[j] = al;
    if (a.last) {
      double sc = fmax(a.ed->scale, fabs(al + a.ashift));
      if (j >= 1) sc = fmax(sc, a.beta[j - 1]);
      a.ed->scale = sc;
    }
  }
}

// ---------------------------------------------------------------------------
// z -= sum_j coef_j q^_j; with `last`, per-CTA partials of ||z||^2.  Vectors with
// small coefficients (SMALL_COEF) are accumulated in FP32, as fractions of their
// own largest number and of z's; the rest in FP64.  Eight FP64 multiply-adds per
// site and vector took 512 cycles of a sub-partition against the 190 of the read
// (100 iterations on 1024^2: now 58 ms, the reads 50).
// Record of vector j: coefficient (re, im) as FP32 in units of z's largest number
// over q^_j's, q^_j's exponent field, and 1 for FP64.
// ---------------------------------------------------------------------------
struct UpdArgs {
  v4* z;
  const v4* basis;
  long long n;
  int j0, j1;
  const double2* coef;
  const int4* rec;
  int last;
  double* norm_part;
  const unsigned* zmax; // z's largest number before
  unsigned* zmax_out;   // and after
  const EigDev* ed;
};

// x 2^-(be - 1022) as FP32 (below 1), truncated; zero below 2^-126
__device__ __forceinline__ float to_fp32(double x, int be) {
  const int hi = __double2hiint(x);
  const unsigned t = __funnelshift_l((unsigned)__double2loint(x), (unsigned)hi, 3) - ((unsigned)(be - 126) << 23);
  const bool tiny = (hi & 0x7ff00000) <= ((be - 126) << 20);
  return __int_as_float(tiny ? 0 : (int)((t & 0x7fffffffu) | (hi & 0x80000000u)));
}

__device__ __forceinline__ void axpy_c(v4& z, double cr, double ci, const v4& q) {
  z.x = fma(-cr, q.x, fma(ci, q.y, z.x));
  z.y = fma(-cr, q.y, fma(-ci, q.x, z.y));
  z.z = fma(-cr, q.z, fma(ci, q.w, z.z));
  z.w = fma(-cr, q.w, fma(-ci, q.z, z.w));
}

__device__ void block_partial(double v, double* out) {
  __shared__ double red[32];
  v = wsum(v);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) red[warp] = v;
  __syncthreads();
  if (warp == 0) {
    double t = lane < (int)(blockDim.x >> 5) ? red[lane] : 0.0;
    t = wsum(t);
    if (lane == 0) *out = t;
  }
}

// GROUPS: warps of a CTA that share the vectors of one set of sites.  1: each
// thread has its own sites and walks all vectors.  8 (small grids, where that walk
// is one chain of loads): 32 sites per CTA, vector quads dealt to eight warps,
// whose parts are added in a fixed order.
template <int GROUPS>
__global__ void __launch_bounds__(256, 4) eig_update(const UpdArgs a) {
  if (a.ed->breakdown | a.ed->error) return;
  constexpr int SITES = 256 / GROUPS;
  __shared__ v4 part[GROUPS > 1 ? GROUPS : 1][GROUPS > 1 ? SITES : 1];
  __shared__ float4 fpart[GROUPS > 1 ? GROUPS : 1][GROUPS > 1 ? SITES : 1];
  const int count = a.j1 - a.j0 + 1;
  const int zbe = max_field(*a.zmax);
  const int site = GROUPS > 1 ? (int)threadIdx.x % SITES : (int)threadIdx.x;
  const int grp = GROUPS > 1 ? (int)threadIdx.x / SITES : 0;
  double nrm = 0.0;
  unsigned m = 0u;
  const long long stride = (long long)gridDim.x * SITES;
  for (long long x0 = (long long)blockIdx.x * SITES; x0 < a.n; x0 += stride) {
    const long long x = x0 + site;
    const bool in = x < a.n;
    v4 zv;
    zv.x = zv.y = zv.z = zv.w = 0.0;
    if (grp == 0) zv = a.z[in ? x : 0];
    float f0 = 0.f, f1 = 0.f, f2 = 0.f, f3 = 0.f;
    // the FP32 sums, in units of 2^(zbe - 1022), into z
    auto flush = [&]() {
      const double unit = __hiloint2double(zbe << 20, 0);
      zv.x = fma((double)(-2.f * f0), unit, zv.x);
      zv.y = fma((double)(-2.f * f1), unit, zv.y);
      zv.z = fma((double)(-2.f * f2), unit, zv.z);
      zv.w = fma((double)(-2.f * f3), unit, zv.w);
      f0 = f1 = f2 = f3 = 0.f;
    };
    const v4* __restrict__ q = a.basis + (size_t)a.j0 * a.n + (in ? x : 0);
    auto one = [&](int jj, const v4& v, const int4& rc) {
      if (rc.w) {
        const double2 c = __ldg(a.coef + jj);
        axpy_c(zv, c.x, c.y, v);
      } else {
        const float cr = __int_as_float(rc.x), ci = __int_as_float(rc.y);
        const float qx = to_fp32(v.x, rc.z), qy = to_fp32(v.y, rc.z), qz = to_fp32(v.z, rc.z), qw = to_fp32(v.w, rc.z);
        f0 = fmaf(cr, qx, fmaf(-ci, qy, f0));
        f1 = fmaf(cr, qy, fmaf(ci, qx, f1));
        f2 = fmaf(cr, qz, fmaf(-ci, qw, f2));
        f3 = fmaf(cr, qw, fmaf(ci, qz, f3));
      }
    };
    int jj = 4 * grp, run = 0;
    for (; jj + 4 <= count; jj += 4 * GROUPS) {
      const v4 q0 = q[(size_t)jj * a.n], q1 = q[(size_t)(jj + 1) * a.n];
      const v4 q2 = q[(size_t)(jj + 2) * a.n], q3 = q[(size_t)(jj + 3) * a.n];
      const int4 r0 = __ldg(a.rec + jj), r1 = __ldg(a.rec + jj + 1), r2 = __ldg(a.rec + jj + 2), r3 = __ldg(a.rec + jj + 3);
      one(jj, q0, r0);
      one(jj + 1, q1, r1);
      one(jj + 2, q2, r2);
      one(jj + 3, q3, r3);
      run += 4;
      if (run == FP32_RUN - 4) {     // (up to three more come after the last four)
        flush();
        run = 0;
      }
    }
    for (; jj < count; ++jj) one(jj, q[(size_t)jj * a.n], __ldg(a.rec + jj));   // the last quad's owner
    if constexpr (GROUPS > 1) {
      part[grp][site] = zv;
      fpart[grp][site] = make_float4(f0, f1, f2, f3);
      __syncthreads();
      if (grp == 0) {
#pragma unroll
        for (int g = 1; g < GROUPS; ++g) {
          const v4 p = part[g][site];
          const float4 f = fpart[g][site];
          if (p.x != 0.0 || p.y != 0.0 || p.z != 0.0 || p.w != 0.0) {
            zv.x += p.x; zv.y += p.y; zv.z += p.z; zv.w += p.w;
          }
          f0 += f.x; f1 += f.y; f2 += f.z; f3 += f.w;   // (seven more roundings)
        }
      }
      __syncthreads();
    }
    if (in && grp == 0) {
      flush();
      a.z[x] = zv;
      m = max(m, mag4(zv));
      if (a.last) nrm = fma(zv.x, zv.x, fma(zv.y, zv.y, fma(zv.z, zv.z, fma(zv.w, zv.w, nrm))));
    }
  }
  block_max(m, a.zmax_out);
  if (a.last) block_partial(nrm, a.norm_part + blockIdx.x);
}

// slot 0 = start, with the ||start||^2 partials
__global__ void __launch_bounds__(256) eig_start(const v4* in, v4* out, long long n, double* norm_part,
                                                 unsigned* vmax) {
  double nrm = 0.0;
  unsigned m = 0u;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += stride) {
    const v4 v = in[x];
    out[x] = v;
    m = max(m, mag4(v));
    nrm = fma(v.x, v.x, fma(v.y, v.y, fma(v.z, v.z, fma(v.w, v.w, nrm))));
  }
  block_max(m, vmax);
  block_partial(nrm, norm_part + blockIdx.x);
}

// ---------------------------------------------------------------------------
// Ritz values of T_k (Sec. 2) and the Eq. 9 bounds
// ---------------------------------------------------------------------------
struct RitzArgs {
  int k;
  const double* alpha;
  double* beta;
  const double* norm_part;
  int n_part;
  EigDev* ed;
  double lo, hi;        // examined range (energies of A); use_window = 0: the lowest values
  int use_window;
  int exam_max;         // most Ritz values examined (<= RITZ_CAP)
  double* th_s;         // scaled Ritz values, RITZ_CAP
  double* as;           // scaled T: diagonal, off-diagonal, squared off-diagonal
  double* bs;
  double* b2s;
  RitzOut* out;
  double* X;            // eigenvectors, RITZ_CAP rows of kmax
  double* lu;           // LU scratch, RITZ_CAP x 4 x kmax
  int* piv;             // RITZ_CAP x kmax
  int kmax;
};

// Number of eigenvalues of the scaled T below x: sign changes of the
// characteristic polynomials p_j(x) = det(T_j - x) from the three-term
// recurrence p_j = (a_j - x) p_{j-1} - b_{j-1}^2 p_{j-2}.  The pair is rescaled
// by a power of two every 8 terms; an exact zero takes the sign opposite to
// its predecessor (it counts as an eigenvalue at or below x of T_j).
//
// Signs, zeros and magnitudes are taken from the bits: an FP64 comparison costs as
// much as a multiplication (76 cycles of a sub-partition).
__device__ int sturm_count(const double* __restrict__ as, const double* __restrict__ b2s, int k, double x) {
  double p1 = 1.0, p2 = 0.0;
  int cnt = 0;
  for (int j = 0; j < k; ++j) {
    const double t = (j > 0) ? b2s[j - 1] * p2 : 0.0;
    double p = fma(as[j] - x, p1, -t);
    if (((__double2hiint(p) & 0x7fffffff) | __double2loint(p)) == 0)
      p = (__double2hiint(p1) < 0 ? 1.0 : -1.0) * fabs(p1) * 0x1p-60;
    cnt += (int)((unsigned)(__double2hiint(p) ^ __double2hiint(p1)) >> 31);
    p2 = p1;
    p1 = p;
    if ((j & 7) == 7) {
      const int e = max(fx::exp_field(p1), fx::exp_field(p2)) - 1023;
      if (e > 400 || e < -400) {
        const double f = ldexp(1.0, -e);
        p1 *= f;
        p2 *= f;
      }
    }
  }
  return cnt;
}

// max (or min, with `mx` false) over a block of up to 1024 threads; every
// thread gets the result
__device__ double block_extreme(double v, bool mx) {
  __shared__ double red[32];
  v = mx ? wmax(v) : wmin(v);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double r = red[0];
  for (int w = 1; w < nw; ++w) r = mx ? fmax(r, red[w]) : fmin(r, red[w]);
  return r;
}

__global__ void __launch_bounds__(256) eig_ritz_prep(const RitzArgs a) {
  __shared__ int shk;
  RitzOut* o = a.out;
  if (threadIdx.x < 32) {
    // beta_k: from the last norm partials, or the one that broke down
    const bool broke = a.ed->breakdown != 0;
    const int kb = broke ? a.ed->k_final : a.k;
    double nrm = 0.0;
    if (!broke)
      for (int c = threadIdx.x; c < a.n_part; c += 32) nrm += a.norm_part[c];
    nrm = wsum(nrm);
    if (threadIdx.x == 0) {
      int k = kb;
      const double bt = broke ? a.beta[kb - 1] : sqrt(nrm);
      o->error = 0;
      if (a.ed->error || !isfinite(bt)) {
        o->error = 1;
        a.ed->error = 1;
        k = 0;
      } else if (!broke) {
        a.beta[k - 1] = bt;
        if (bt <= BREAKDOWN_REL * a.ed->scale) { a.ed->breakdown = 1; a.ed->k_final = k; }
      }
      o->k = k;
      o->n_lo = o->n_hi = o->n_exam = 0;
      o->breakdown = a.ed->breakdown;
      o->beta_last = bt;
      shk = k;
    }
  }
  __syncthreads();
  const int k = shk;
  if (k == 0) return;
  // scale T by 2^-e, 2^e above the Gershgorin bound max_j |a_j| + b_{j-1} + b_j,
  // so that the scaled norm is <= 1
  double g = 0.0;
  for (int j = threadIdx.x; j < k; j += blockDim.x) {
    const double bl = j > 0 ? a.beta[j - 1] : 0.0, br = j < k - 1 ? a.beta[j] : 0.0;
    g = fmax(g, fabs(a.alpha[j]) + bl + br);
  }
  g = block_extreme(g, true);
  const int e = g > 0.0 ? ilogb(g) + 1 : 0;
  const double f = ldexp(1.0, -e);
  double glo = 1e300, ghi = -1e300;
  for (int j = threadIdx.x; j < k; j += blockDim.x) {
    const double aj = a.alpha[j] * f;
    const double bl = j > 0 ? a.beta[j - 1] * f : 0.0, br = j < k - 1 ? a.beta[j] * f : 0.0;
    a.as[j] = aj;
    if (j < k - 1) { a.bs[j] = br; a.b2s[j] = br * br; }
    glo = fmin(glo, aj - bl - br);
    ghi = fmax(ghi, aj + bl + br);
  }
  glo = block_extreme(glo, false);
  ghi = block_extreme(ghi, true);
  __syncthreads();   // the scaled arrays are complete
  if (threadIdx.x == 0) {
    // widen by a few ulps so that the interval brackets every eigenvalue
    const double pad = 8.0 * DBL_EPSILON * fmax(1.0, fmax(fabs(glo), fabs(ghi)));
    o->g_lo = glo - pad;
    o->g_hi = ghi + pad;
    o->exp2 = e;
    o->n_lo = a.use_window ? sturm_count(a.as, a.b2s, k, a.lo * f) : 0;
  }
  if (threadIdx.x == 32) o->n_hi = a.use_window ? sturm_count(a.as, a.b2s, k, a.hi * f) : k;
  __syncthreads();
  if (threadIdx.x == 0) o->n_exam = min(o->n_hi - o->n_lo, a.exam_max);
}

// LU of the scaled T - theta with partial pivoting (row interchanges kept in
// piv): rd reciprocals of U's diagonal (one division a row: 434 cycles), u1/u2 its
// first/second superdiagonal, l the multipliers.  One thread; the row being
// eliminated stays in registers.
__device__ void tridiag_lu(const double* __restrict__ as, const double* __restrict__ bs, int k, double theta,
                           double* rd, double* u1, double* u2, double* l, int* piv) {
  const double tiny = DBL_EPSILON;   // T is scaled to norm <= 1
  double d = as[0] - theta, u = k > 1 ? bs[0] : 0.0;
  for (int j = 0; j < k - 1; ++j) {
    const double low = bs[j];                 // entry (j+1, j)
    const double dn = as[j + 1] - theta, un = j + 1 < k - 1 ? bs[j + 1] : 0.0;
    if (fabs(d) >= fabs(low)) {
      const double r = 1.0 / (d == 0.0 ? tiny : d);
      const double m = low * r;
      rd[j] = r;
      u1[j] = u;
      u2[j] = 0.0;
      l[j] = m;
      piv[j] = 0;
      d = fma(-m, u, dn);
      u = un;
    } else {                                  // rows j and j+1 change places
      const double r = 1.0 / low;
      const double m = d * r;
      rd[j] = r;
      u1[j] = dn;
      u2[j] = un;
      l[j] = m;
      piv[j] = 1;
      d = fma(-m, dn, u);
      u = -m * un;
    }
  }
  rd[k - 1] = 1.0 / (d == 0.0 ? tiny : d);
  u1[k - 1] = u2[k - 1] = 0.0;
}

// x <- (T - theta)^{-1} x with the factors of tridiag_lu; one thread
__device__ void tridiag_solve(int k, const double* rd, const double* u1, const double* u2, const double* l,
                              const int* piv, double* x) {
  double c = x[0];
  for (int j = 0; j < k - 1; ++j) {
    double n = x[j + 1];
    if (piv[j]) { const double t = c; c = n; n = t; }
    x[j] = c;
    c = fma(-l[j], c, n);
  }
  double x1 = c * rd[k - 1], x2 = 0.0;      // x[j + 1], x[j + 2]
  x[k - 1] = x1;
  for (int j = k - 2; j >= 0; --j) {
    const double t = fma(-u2[j], x2, fma(-u1[j], x1, x[j])) * rd[j];
    x[j] = t;
    x2 = x1;
    x1 = t;
  }
}

// x /= ||x|| by one warp (x in global memory; the warp is synchronised on return)
__device__ void warp_normalise(double* x, int k) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  double mx = 0.0;
  for (int j = lane; j < k; j += 32) mx = fmax(mx, fabs(x[j]));
  mx = wmax(mx);
  const double inv_mx = mx > 0.0 ? 1.0 / mx : 1.0;
  double nrm = 0.0;
  for (int j = lane; j < k; j += 32) { const double t = x[j] * inv_mx; nrm = fma(t, t, nrm); }
  nrm = wsum(nrm);
  const double f = inv_mx / sqrt(nrm);
  for (int j = lane; j < k; j += 32) x[j] *= f;
  __syncwarp();
}

// Ritz values: multisection for the r-th smallest eigenvalue (0-based) of the
// scaled T, one block of four warps each, 128 Sturm counts per round (8 rounds to
// the last digit, where 32 points took 11)
constexpr int RV_THREADS = 128;

__global__ void __launch_bounds__(RV_THREADS) eig_ritz_values(const RitzArgs a) {
  __shared__ int firsts[RV_THREADS / 32];
  const RitzOut* o = a.out;
  if (o->error || o->k == 0) return;
  const int w = (int)blockIdx.x;
  if (w >= o->n_exam) return;
  const int k = o->k;
  const int r = o->n_lo + w;
  double lo = o->g_lo, hi = o->g_hi;
  auto point = [&](double l, double width, int i) { return l + width * (double)(i + 1) * (1.0 / (RV_THREADS + 1)); };
  for (int round = 0; round < 80; ++round) {
    const double width = hi - lo;
    if (width <= 2.0 * DBL_EPSILON * fmax(fabs(lo), fabs(hi)) + 2.0 * DBL_EPSILON) break;
    const int c = sturm_count(a.as, a.b2s, k, point(lo, width, (int)threadIdx.x));
    const unsigned above = __ballot_sync(0xffffffffu, c > r);   // points past the eigenvalue
    if ((threadIdx.x & 31) == 0) firsts[threadIdx.x >> 5] = above ? __ffs(above) - 1 : 32;
    __syncthreads();
    int f = RV_THREADS;                                         // the first of them
#pragma unroll
    for (int q = RV_THREADS / 32 - 1; q >= 0; --q)
      if (firsts[q] < 32) f = 32 * q + firsts[q];
    __syncthreads();
    const double l0 = lo;
    if (f > 0) lo = point(l0, width, f - 1);
    if (f < RV_THREADS) hi = point(l0, width, f);
  }
  if (threadIdx.x == 0) {
    const double th = 0.5 * (lo + hi);
    a.th_s[w] = th;
    a.out->theta[w] = ldexp(th, o->exp2);
  }
}

// Ritz vectors of T (t_i, for Eq. 9 and Eq. 8) by inverse iteration, two
// solves from a fixed pseudo-random start.  Values closer than CLUSTER (in
// units of the scaled norm) form a cluster, handled by one warp in order:
// each member's iterate is orthogonalised against the members before it
// (modified Gram-Schmidt) and a value equal to its predecessor is nudged by a
// few ulps so that the factorisations differ.
constexpr double CLUSTER = 1e-7;

__global__ void __launch_bounds__(128) eig_ritz_tvecs(const RitzArgs a) {
  const RitzOut* o = a.out;
  if (o->error || o->k == 0) return;
  const int lane = threadIdx.x & 31;
  const int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int ne = o->n_exam;
  if (w >= ne) return;
  if (w > 0 && a.th_s[w] - a.th_s[w - 1] <= CLUSTER) return;   // not the first of its cluster
  const int k = o->k;
  double* lu = a.lu + (size_t)w * 4 * a.kmax;
  double *d = lu, *u1 = lu + a.kmax, *u2 = lu + 2 * a.kmax, *l = lu + 3 * a.kmax;
  int* piv = a.piv + (size_t)w * a.kmax;
  double th_prev = 0.0;
  for (int m = w; m < ne && (m == w || a.th_s[m] - a.th_s[m - 1] <= CLUSTER); ++m) {
    double th = a.th_s[m];
    if (m > w && th - th_prev < 10.0 * DBL_EPSILON) th = th_prev + 10.0 * DBL_EPSILON;
    th_prev = th;
    double* x = a.X + (size_t)m * a.kmax;
    if (lane == 0) tridiag_lu(a.as, a.bs, k, th, d, u1, u2, l, piv);
    for (int j = lane; j < k; j += 32) {
      unsigned h = (unsigned)j * 2654435761u + 0x9e3779b9u;
      h ^= h >> 15; h *= 0x85ebca6bu; h ^= h >> 13;
      x[j] = 0.5 + (double)(h >> 8) * (1.0 / 16777216.0);
    }
    __syncwarp();
    for (int it = 0; it < 2; ++it) {
      if (lane == 0) tridiag_solve(k, d, u1, u2, l, piv, x);
      warp_normalise(x, k);
      for (int p = w; p < m; ++p) {         // against the earlier members of the cluster
        const double* xp = a.X + (size_t)p * a.kmax;
        double dot = 0.0;
        for (int j = lane; j < k; j += 32) dot = fma(xp[j], x[j], dot);
        dot = wsum(dot);
        for (int j = lane; j < k; j += 32) x[j] = fma(-dot, xp[j], x[j]);
        __syncwarp();
      }
      if (m > w) warp_normalise(x, k);
    }
    if (lane == 0) a.out->bound[m] = fabs(o->beta_last * x[k - 1]);
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------
// Ritz vectors y_l = sum_j q_j t_{j,l} = sum_j q^_j (s_j t_{j,l})  (Eq. 8)
// ---------------------------------------------------------------------------
struct RvArgs {
  const v4* basis;
  const double* s;
  const double* X;
  int kmax, k;
  const int* sel;       // rows of X
  int n_sel;
  long long n;
  v4* out;              // n_sel consecutive fields
};

__global__ void __launch_bounds__(256) eig_ritz_vectors(const RvArgs a) {
  __shared__ double w[4][256];
  const long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (int l0 = 0; l0 < a.n_sel; l0 += 4) {
    const int nl = min(4, a.n_sel - l0);
    double acc[4][4];
#pragma unroll
    for (int l = 0; l < 4; ++l) acc[l][0] = acc[l][1] = acc[l][2] = acc[l][3] = 0.0;
    for (int jb = 0; jb < a.k; jb += 256) {
      __syncthreads();
      const int j = jb + threadIdx.x;
#pragma unroll
      for (int l = 0; l < 4; ++l)
        w[l][threadIdx.x] = (l < nl && j < a.k) ? a.s[j] * a.X[(size_t)a.sel[l0 + l] * a.kmax + j] : 0.0;
      __syncthreads();
      if (x < a.n) {
        const int jn = min(256, a.k - jb);
        for (int jj = 0; jj < jn; ++jj) {
          const v4 q = a.basis[(size_t)(jb + jj) * a.n + x];
#pragma unroll
          for (int l = 0; l < 4; ++l) {
            const double c = w[l][jj];
            acc[l][0] = fma(c, q.x, acc[l][0]);
            acc[l][1] = fma(c, q.y, acc[l][1]);
            acc[l][2] = fma(c, q.z, acc[l][2]);
            acc[l][3] = fma(c, q.w, acc[l][3]);
          }
        }
      }
    }
    if (x < a.n) {
      for (int l = 0; l < nl; ++l) {
        v4 r;
        r.x = acc[l][0]; r.y = acc[l][1]; r.z = acc[l][2]; r.w = acc[l][3];
        a.out[(size_t)(l0 + l) * a.n + x] = r;
      }
    }
  }
}

// folded mode: lambda = sigma + sign(rho) sqrt(theta), rho = <y, (H - s - sigma) y>
__global__ void eig_fold_finish(const double2* part, int n_cta, double theta, double bound, double sigma,
                                double* out) {
  double re = 0.0;
  for (int c = threadIdx.x; c < n_cta; c += 32) re += part[c].x;
  re = wsum(re);
  if (threadIdx.x != 0) return;
  const double th = fmax(theta, 0.0), rt = sqrt(th);
  out[0] = sigma + copysign(rt, re);
  out[1] = th > 0.0 ? fmin(sqrt(bound), bound / rt) : sqrt(bound);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct DevMem {
  void* p = nullptr;
  ~DevMem() { if (p) cudaFree(p); }
};

#define EIG_TRY(call)                                                                   \
  do {                                                                                  \
    cudaError_t e_ = (call);                                                            \
    if (e_ != cudaSuccess) return fail(DIRAC_ECUDA, "%s: %s", #call, cudaGetErrorString(e_)); \
  } while (0)

int n_sms() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 1;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 1;
  return std::max(1, n);
}

ApplyArgs apply_args(const CtxView& v, double e0) {
  ApplyArgs a;
  std::memset(&a, 0, sizeof(a));
  const double kfac = v.order == 2 ? 2.0 : 12.0;
  const double mc2 = v.mass * v.c * v.c;
  a.nx = v.nx; a.ny = v.ny;
  a.kx = v.c / (kfac * v.dx);
  a.ky = v.c / (kfac * v.dy);
  a.cax = v.c * v.ax;
  a.cay = v.c * v.ay;
  a.au = mc2 - e0;
  a.ad = -mc2 - e0;
  a.V = v.V;
  return a;
}

template <int R, bool D>
cudaError_t launch_apply_rd(const ApplyArgs& a, cudaStream_t s, bool f32) {
  if (f32) {
    const dim3 grid((a.nx + 31) / 32, (a.ny + 7) / 8);
    if (a.V) eig_apply32<R, D, true><<<grid, 256, 0, s>>>(a);
    else eig_apply32<R, D, false><<<grid, 256, 0, s>>>(a);
  } else {
    // four rows a thread, or one on grids of less than two tall tiles per SM,
    // where the time of one tile counts
    const int tiles_x = (a.nx + TILE_W - 1) / TILE_W;
    const bool tall = (long long)tiles_x * ((a.ny + 4 * AP_WARPS - 1) / (4 * AP_WARPS)) >= 2LL * n_sms();
    const int th = tall ? 4 * AP_WARPS : AP_WARPS;
    const dim3 grid(tiles_x, (a.ny + th - 1) / th);
    auto go = [&](auto rpt, auto lanczos) {
      constexpr int P = decltype(rpt)::value;
      constexpr bool L = decltype(lanczos)::value;
      if (a.V) eig_apply64<R, D, true, P, L><<<grid, AP_THREADS, 0, s>>>(a);
      else eig_apply64<R, D, false, P, L><<<grid, AP_THREADS, 0, s>>>(a);
    };
    using std::integral_constant;
    if (tall) {
      if (a.ed) go(integral_constant<int, 4>{}, std::true_type{});
      else go(integral_constant<int, 4>{}, std::false_type{});
    } else {
      if (a.ed) go(integral_constant<int, 1>{}, std::true_type{});
      else go(integral_constant<int, 1>{}, std::false_type{});
    }
  }
  return cudaGetLastError();
}

// f32: the mixed-precision product (the Lanczos steps of a DIRAC_MIXED context)
cudaError_t launch_apply(const CtxView& v, const ApplyArgs& a, bool f32 = false) {
  const bool d = v.boundary == DIRAC_DIRICHLET;
  if (v.order == 2) return d ? launch_apply_rd<1, true>(a, v.stream, f32) : launch_apply_rd<1, false>(a, v.stream, f32);
  return d ? launch_apply_rd<2, true>(a, v.stream, f32) : launch_apply_rd<2, false>(a, v.stream, f32);
}

// Device time per kernel kind from CUDA events recorded between consecutive
// launches on one stream (active only while the context is profiling).
enum { K_APPLY = 0, K_DOT = 1, K_UPDATE = 2, K_OTHER = 3, K_START = -1 };

struct KindTimer {
  bool on = false;
  cudaStream_t s = nullptr;
  std::vector<cudaEvent_t> ev;
  std::vector<int> kind;      // kind of the kernel that ends at event j
  size_t used = 0;
  double ms[4] = {0.0, 0.0, 0.0, 0.0};
  long long n = 0;            // kernels launched (counted also when not timing)

  // after a launch of `k` (K_START: before the first launch of a segment)
  cudaError_t mark(int k) {
    if (k >= 0) ++n;
    if (!on) return cudaSuccess;
    if (used == ev.size()) {
      cudaEvent_t e;
      cudaError_t r = cudaEventCreate(&e);
      if (r != cudaSuccess) return r;
      ev.push_back(e);
      kind.push_back(k);
    }
    kind[used] = k;
    return cudaEventRecord(ev[used++], s);
  }
  // after the stream has been synchronised: add up and start a new segment
  cudaError_t flush() {
    if (!on) return cudaSuccess;
    for (size_t j = 1; j < used; ++j) {
      if (kind[j] < 0) continue;
      float t = 0.f;
      cudaError_t r = cudaEventElapsedTime(&t, ev[j - 1], ev[j]);
      if (r != cudaSuccess) return r;
      ms[kind[j]] += t;
    }
    used = 0;
    return cudaSuccess;
  }
  ~KindTimer() {
    for (cudaEvent_t e : ev) cudaEventDestroy(e);
  }
};

}  // namespace eig
}  // namespace dirac

using namespace dirac;
using namespace dirac::eig;

extern "C" {

dirac_status dirac_apply_hamiltonian(dirac_ctx* ctx, const void* in_dev, void* out_dev) {
  CtxView v;
  dirac_status st = ctx_view(ctx, &v);
  if (st != DIRAC_OK) return st;
  if (!v.fields_set) return fail(DIRAC_ESTATE, "dirac_set_fields has not been called");
  if (!in_dev || !out_dev) return fail(DIRAC_EINVAL, "null vector");
  if ((reinterpret_cast<uintptr_t>(in_dev) | reinterpret_cast<uintptr_t>(out_dev)) & 31u)
    return fail(DIRAC_EINVAL, "vectors must be 32-byte aligned");
  if (in_dev == out_dev) return fail(DIRAC_EINVAL, "in and out must not alias");
  ApplyArgs a = apply_args(v, v.shift);
  a.in = static_cast<const v4*>(in_dev);
  a.out = static_cast<v4*>(out_dev);
  EIG_TRY(launch_apply(v, a));
  ++*v.launches;
  return DIRAC_OK;
}

dirac_status dirac_lanczos_eigs(dirac_ctx* ctx, const void* start_dev, int n_want, int max_iter,
                                int check_every, double tol, double e_lo, double e_hi, int reorth,
                                int fold, double sigma, double* eigs_out, double* bounds_out,
                                void* vecs_dev, dirac_eig_info* info) {
  dirac::TraceRange trace("dirac_lanczos_eigs");
  CtxView v;
  dirac_status st = ctx_view(ctx, &v);
  if (st != DIRAC_OK) return st;
  if (!v.fields_set) return fail(DIRAC_ESTATE, "dirac_set_fields has not been called");
  if (!start_dev || (reinterpret_cast<uintptr_t>(start_dev) & 31u))
    return fail(DIRAC_EINVAL, "start vector must be a non-null 32-byte aligned device pointer");
  if (vecs_dev && (reinterpret_cast<uintptr_t>(vecs_dev) & 31u))
    return fail(DIRAC_EINVAL, "vecs_dev must be 32-byte aligned");
  if (n_want < 1 || n_want > RITZ_CAP) return fail(DIRAC_EINVAL, "n_want must be 1..%d", RITZ_CAP);
  if (max_iter < 1 || max_iter > MAX_ITER) return fail(DIRAC_EINVAL, "max_iter must be 1..%d", MAX_ITER);
  if (check_every < 1) return fail(DIRAC_EINVAL, "check_every must be >= 1");
  if (!(tol >= 0.0) || !std::isfinite(tol)) return fail(DIRAC_EINVAL, "tol must be finite and >= 0");
  if (!fold && !(e_lo < e_hi)) return fail(DIRAC_EINVAL, "window needs e_lo < e_hi");
  if (fold && !std::isfinite(sigma)) return fail(DIRAC_EINVAL, "fold sigma must be finite");
  if (!eigs_out || !bounds_out) return fail(DIRAC_EINVAL, "null output array");
  if (info) std::memset(info, 0, sizeof(*info));

  const long long n = (long long)v.nx * v.ny;
  const size_t vb = sizeof(v4) * (size_t)n;
  const int kmax = max_iter;
  const int sm = n_sms();
  cudaStream_t s = v.stream;

  // launch geometry, fixed for the call
  int cs = (int)std::min<long long>(CH_MAX, std::max<long long>(32, (n + 4LL * sm - 1) / (4LL * sm)));
  cs = (cs + 31) / 32 * 32;
  const int n_dot = (int)std::min<long long>(4LL * sm, (n + cs - 1) / cs);
  // update: one thread per site where that fills the GPU (a CTA per SM), else eight
  const int upd_groups = n < 256LL * sm ? 8 : 1;
  const int upd_sites = 256 / upd_groups;
  const int n_upd = (int)std::min<long long>(4LL * sm, std::max<long long>(1, (n + upd_sites - 1) / upd_sites));
  const size_t z_smem = (size_t)cs * (2 * sizeof(v4) + sizeof(int));   // a chunk of z: limbs, numbers, exponents
  const size_t dot_smem_max = z_smem + sizeof(double2) * (size_t)(kmax + 2);
  EIG_TRY(cudaFuncSetAttribute(eig_dot<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dot_smem_max));
  EIG_TRY(cudaFuncSetAttribute(eig_dot<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dot_smem_max));

  // device memory: basis slots 0..max_iter, then (folded) one product buffer
  // and the n_want Ritz vectors before sorting
  const size_t n_vec = (size_t)kmax + 1 + (fold ? 1 + (size_t)n_want : 0);
  size_t free_b = 0, total_b = 0;
  EIG_TRY(cudaMemGetInfo(&free_b, &total_b));
  if (vb * n_vec > free_b)
    return fail(DIRAC_ENOMEM, "eigen mode needs %.3g GB for %zu vectors, %.3g GB free", vb * n_vec / 1e9,
                n_vec, free_b / 1e9);
  DevMem basis_mem, small_mem;
  EIG_TRY(cudaMalloc(&basis_mem.p, vb * n_vec));
  v4* basis = static_cast<v4*>(basis_mem.p);
  v4* tmp = fold ? basis + (size_t)(kmax + 1) * n : nullptr;
  v4* fold_vecs = fold ? tmp + n : nullptr;

  // small arrays
  size_t off = 0;
  auto take = [&](size_t bytes) { const size_t o = off; off += (bytes + 255) & ~size_t(255); return o; };
  const size_t o_ed = take(sizeof(EigDev));
  const size_t o_ro = take(sizeof(RitzOut));
  const size_t o_alpha = take(sizeof(double) * (kmax + 1));
  const size_t o_beta = take(sizeof(double) * (kmax + 1));
  const size_t o_s = take(sizeof(double) * (kmax + 1));
  const size_t o_coef = take(sizeof(double2) * (kmax + 1));
  const size_t o_dpart = take(sizeof(double2) * (size_t)n_dot * (kmax + 2));
  const size_t o_rec = take(sizeof(int4) * (kmax + 1));
  const size_t o_vmax = take(sizeof(unsigned) * 3 * (kmax + 2));
  const size_t o_npart = take(sizeof(double) * n_upd);
  const size_t o_as = take(sizeof(double) * kmax);
  const size_t o_bs = take(sizeof(double) * kmax);
  const size_t o_b2s = take(sizeof(double) * kmax);
  const size_t o_X = take(sizeof(double) * (size_t)RITZ_CAP * kmax);
  const size_t o_lu = take(sizeof(double) * (size_t)RITZ_CAP * 4 * kmax);
  const size_t o_piv = take(sizeof(int) * (size_t)RITZ_CAP * kmax);
  const size_t o_sel = take(sizeof(int) * RITZ_CAP);
  const size_t o_fres = take(sizeof(double) * 2 * RITZ_CAP);
  const size_t o_ths = take(sizeof(double) * RITZ_CAP);
  EIG_TRY(cudaMalloc(&small_mem.p, off));
  char* sb = static_cast<char*>(small_mem.p);
  EigDev* ed = reinterpret_cast<EigDev*>(sb + o_ed);
  RitzOut* ro = reinterpret_cast<RitzOut*>(sb + o_ro);
  double* alpha = reinterpret_cast<double*>(sb + o_alpha);
  double* beta = reinterpret_cast<double*>(sb + o_beta);
  double* sarr = reinterpret_cast<double*>(sb + o_s);
  double2* coef = reinterpret_cast<double2*>(sb + o_coef);
  double2* dpart = reinterpret_cast<double2*>(sb + o_dpart);
  double* npart = reinterpret_cast<double*>(sb + o_npart);
  int4* rec = reinterpret_cast<int4*>(sb + o_rec);
  unsigned* vmax = reinterpret_cast<unsigned*>(sb + o_vmax);   // largest numbers by slot: after the product, the first
                                                               // update, and at the end
  int* d_sel = reinterpret_cast<int*>(sb + o_sel);
  double* d_fres = reinterpret_cast<double*>(sb + o_fres);
  EIG_TRY(cudaMemsetAsync(ed, 0, sizeof(EigDev), s));
  EIG_TRY(cudaMemsetAsync(vmax, 0, sizeof(unsigned) * 3 * (kmax + 2), s));
  EIG_TRY(cudaMemsetAsync(alpha, 0, sizeof(double) * (kmax + 1), s));
  EIG_TRY(cudaMemsetAsync(beta, 0, sizeof(double) * (kmax + 1), s));

  RitzArgs ra;
  ra.alpha = alpha; ra.beta = beta; ra.norm_part = npart; ra.n_part = n_upd; ra.ed = ed;
  ra.lo = e_lo; ra.hi = e_hi; ra.use_window = fold ? 0 : 1;
  ra.exam_max = fold ? n_want : RITZ_CAP;
  ra.as = reinterpret_cast<double*>(sb + o_as);
  ra.bs = reinterpret_cast<double*>(sb + o_bs);
  ra.b2s = reinterpret_cast<double*>(sb + o_b2s);
  ra.out = ro;
  ra.X = reinterpret_cast<double*>(sb + o_X);
  ra.lu = reinterpret_cast<double*>(sb + o_lu);
  ra.piv = reinterpret_cast<int*>(sb + o_piv);
  ra.th_s = reinterpret_cast<double*>(sb + o_ths);
  ra.kmax = kmax;

  KindTimer tm;
  tm.on = v.profiling;
  tm.s = s;
  // every exit from here on adds the launches to the context and fills info
  struct Finish {
    KindTimer& tm;
    CtxView& v;
    dirac_eig_info* info;
    ~Finish() {
      *v.launches += tm.n;
      if (info) {
        info->launches = tm.n;
        info->ms_apply = tm.ms[K_APPLY];
        info->ms_dot = tm.ms[K_DOT];
        info->ms_update = tm.ms[K_UPDATE];
        info->ms_other = tm.ms[K_OTHER];
      }
    }
  } finish_guard{tm, v, info};

  EIG_TRY(tm.mark(K_START));
  eig_start<<<n_upd, 256, 0, s>>>(static_cast<const v4*>(start_dev), basis, n, npart, vmax + 2);
  EIG_TRY(cudaGetLastError());
  EIG_TRY(tm.mark(K_OTHER));

  const double e0 = v.shift + (fold ? sigma : 0.0);   // A = H - e0 (direct) or (H - e0)^2
  const double ashift = fold ? 0.0 : v.shift;
  std::vector<unsigned char> ro_host(sizeof(RitzOut));
  RitzOut& h = *reinterpret_cast<RitzOut*>(ro_host.data());
  std::vector<int> sel;
  int k_done = 0;
  bool finished = false;

  for (int i = 0; i < max_iter && !finished; ++i) {
    v4* z = basis + (size_t)(i + 1) * n;
    const v4* qi = basis + (size_t)i * n;
    const v4* qim = i >= 1 ? basis + (size_t)(i - 1) * n : nullptr;
    ApplyArgs a = apply_args(v, e0);
    a.ed = ed; a.norm_part = npart; a.n_part = n_upd; a.beta = beta; a.s = sarr; a.iter = i;
    a.prologue = 1;
    a.in = qi;
    const bool f32 = v.precision == DIRAC_MIXED;
    if (!fold) {
      a.sub = qim;
      a.out = z;
      a.vmax = vmax + 3 * (i + 1);
      EIG_TRY(launch_apply(v, a, f32));
      EIG_TRY(tm.mark(K_APPLY));
    } else {
      a.sub = nullptr;
      a.out = tmp;
      EIG_TRY(launch_apply(v, a, f32));
      EIG_TRY(tm.mark(K_APPLY));
      a.prologue = 0;
      a.in = tmp;
      a.sub = qim;
      a.out = z;
      a.vmax = vmax + 3 * (i + 1);
      EIG_TRY(launch_apply(v, a, f32));
      EIG_TRY(tm.mark(K_APPLY));
    }
    const int passes = reorth ? 2 : 1;
    const int j0 = reorth ? 0 : i;
    const int count = i - j0 + 1;
    for (int p = 0; p < passes; ++p) {
      DotArgs da{basis, n, j0, i, cs, dpart, ed};
      const size_t smem = z_smem + sizeof(double2) * (size_t)(count + 1);
      if (cs == 32) eig_dot<true><<<n_dot, 256, smem, s>>>(da);
      else eig_dot<false><<<n_dot, 256, smem, s>>>(da);
      EIG_TRY(cudaGetLastError());
      EIG_TRY(tm.mark(K_DOT));
      FinishArgs fa{dpart, n_dot, j0, i, i, p, p == passes - 1, reorth ? 1 : 0, sarr, coef, alpha, beta, ed, ashift,
                    vmax, rec};
      eig_dot_finish<<<(count + 7) / 8, 256, 0, s>>>(fa);
      EIG_TRY(cudaGetLastError());
      EIG_TRY(tm.mark(K_OTHER));
      const bool last = p == passes - 1;
      UpdArgs ua{z, basis, n, j0, i, coef, rec, last ? 1 : 0, npart, vmax + 3 * (i + 1) + p,
                 vmax + 3 * (i + 1) + (last ? 2 : 1), ed};
      if (upd_groups == 8) eig_update<8><<<n_upd, 256, 0, s>>>(ua);
      else eig_update<1><<<n_upd, 256, 0, s>>>(ua);
      EIG_TRY(cudaGetLastError());
      EIG_TRY(tm.mark(K_UPDATE));
    }
    const int it = i + 1;
    if (it % check_every != 0 && it != max_iter) continue;

    ra.k = it;
    eig_ritz_prep<<<1, 256, 0, s>>>(ra);
    EIG_TRY(cudaGetLastError());
    eig_ritz_values<<<RITZ_CAP, RV_THREADS, 0, s>>>(ra);
    EIG_TRY(cudaGetLastError());
    eig_ritz_tvecs<<<(RITZ_CAP + 3) / 4, 128, 0, s>>>(ra);
    EIG_TRY(cudaGetLastError());
    EIG_TRY(tm.mark(K_OTHER));
    tm.n += 2;
    EIG_TRY(cudaMemcpyAsync(ro_host.data(), ro, sizeof(RitzOut), cudaMemcpyDeviceToHost, s));
    EIG_TRY(cudaStreamSynchronize(s));
    EIG_TRY(tm.flush());
    EIG_TRY(tm.mark(K_START));
    if (h.error) return fail(DIRAC_ENONFINITE, "eigen mode: non-finite value or zero start vector");
    k_done = h.k;
    const int n_exam = h.n_exam;
    std::vector<int> conv;
    for (int w = 0; w < n_exam; ++w) {
      const double th = h.theta[w];
      bool c = h.bound[w] <= tol * std::max(1.0, std::fabs(th));
      if (!fold) c = c && th > e_lo && th < e_hi;
      if (c) conv.push_back(w);
    }
    const bool done = it >= max_iter || h.breakdown;
    bool ok;
    if (!fold) {
      ok = (int)conv.size() >= n_want;
    } else {
      ok = n_exam >= n_want && (int)conv.size() >= n_want && conv[n_want - 1] == n_want - 1;
    }
    if (info) {
      info->iterations = k_done;
      info->n_in_window = h.n_hi - h.n_lo;
      info->n_converged = (int)conv.size();
      info->breakdown = h.breakdown;
    }
    if (ok || done) {
      finished = true;
      if (!fold) {
        sel.assign(conv.begin(), conv.begin() + std::min<size_t>(conv.size(), (size_t)n_want));
      } else {
        for (int w : conv) if (w < n_want) sel.push_back(w);
      }
    }
  }
  const int n_sel = (int)sel.size();
  if (info) info->n_found = n_sel;
  if (n_sel == 0) return DIRAC_OK;

  const int vgrid = (int)((n + 255) / 256);
  if (!fold) {
    for (int l = 0; l < n_sel; ++l) {
      eigs_out[l] = h.theta[sel[l]];
      bounds_out[l] = h.bound[sel[l]];
    }
    if (vecs_dev) {
      EIG_TRY(cudaMemcpyAsync(d_sel, sel.data(), sizeof(int) * n_sel, cudaMemcpyHostToDevice, s));
      RvArgs rv{basis, sarr, ra.X, kmax, k_done, d_sel, n_sel, n, static_cast<v4*>(vecs_dev)};
      eig_ritz_vectors<<<vgrid, 256, 0, s>>>(rv);
      EIG_TRY(cudaGetLastError());
      EIG_TRY(tm.mark(K_OTHER));
      EIG_TRY(cudaStreamSynchronize(s));
      EIG_TRY(tm.flush());
    }
    return DIRAC_OK;
  }

  // folded: Ritz vectors, the sign of each from its Rayleigh quotient with
  // H - s - sigma, lambda ascending
  EIG_TRY(cudaMemcpyAsync(d_sel, sel.data(), sizeof(int) * n_sel, cudaMemcpyHostToDevice, s));
  RvArgs rv{basis, sarr, ra.X, kmax, k_done, d_sel, n_sel, n, fold_vecs};
  eig_ritz_vectors<<<vgrid, 256, 0, s>>>(rv);
  EIG_TRY(cudaGetLastError());
  EIG_TRY(tm.mark(K_OTHER));
  for (int l = 0; l < n_sel; ++l) {
    ApplyArgs a = apply_args(v, e0);
    a.in = fold_vecs + (size_t)l * n;
    a.out = tmp;
    EIG_TRY(launch_apply(v, a));
    EIG_TRY(tm.mark(K_APPLY));
    eig_inner<<<n_dot, 256, 0, s>>>(fold_vecs + (size_t)l * n, tmp, n, dpart);
    EIG_TRY(cudaGetLastError());
    EIG_TRY(tm.mark(K_DOT));
    eig_fold_finish<<<1, 32, 0, s>>>(dpart, n_dot, h.theta[sel[l]], h.bound[sel[l]], sigma, d_fres + 2 * l);
    EIG_TRY(cudaGetLastError());
    EIG_TRY(tm.mark(K_OTHER));
  }
  std::vector<double> fres(2 * n_sel);
  EIG_TRY(cudaMemcpyAsync(fres.data(), d_fres, sizeof(double) * 2 * n_sel, cudaMemcpyDeviceToHost, s));
  EIG_TRY(cudaStreamSynchronize(s));
  EIG_TRY(tm.flush());
  std::vector<int> order(n_sel);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int p, int q) { return fres[2 * p] < fres[2 * q]; });
  for (int l = 0; l < n_sel; ++l) {
    eigs_out[l] = fres[2 * order[l]];
    bounds_out[l] = fres[2 * order[l] + 1];
    if (vecs_dev)
      EIG_TRY(cudaMemcpyAsync(static_cast<v4*>(vecs_dev) + (size_t)l * n, fold_vecs + (size_t)order[l] * n, vb,
                              cudaMemcpyDeviceToDevice, s));
  }
  EIG_TRY(cudaStreamSynchronize(s));
  return DIRAC_OK;
}

}  // extern "C"
