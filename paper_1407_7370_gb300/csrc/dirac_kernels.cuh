// dirac_kernels.cuh -- device code of the GB300 Dirac Lanczos propagator.
//
// One time step (Sec. 4, Eq. 17) is m launches of `lanczos_pass` (one Lanczos
// iteration each, Fig. 1 / Eq. 4) and one launch of `recombine`.  Every launch
// covers a table of independent problems (grids of any size); a single
// propagation is a table of one.  For a single problem the same pass body can
// instead run inside `lanczos_step`, one cooperative launch per time step
// whose passes are separated by grid-wide barriers (see there).
//
// Pass i (1-based) works on unnormalised vectors whose scales are tracked by
// device scalars:
//   q^_1 = psi                                  (no copy: psi is read in place)
//   q^_i = g_{i-1} (y^_{i-1} - d_{i-1} q^_{i-1})  formed on the fly, i >= 2
//   y^_i = (H - s - sigma_i) q^_i - e_i q^_{i-1}  the stencil product
// and reduces P = Re<q^_i, y^_i>, Y = ||y^_i||^2, X = ||q^_i||^2 in the same
// pass.  With q_i = q^_i / nu_i (nu_i = sqrt X) one has y^_i = nu_i (z_i -
// sigma_i q_i), z_i = A q_i - beta_{i-1} q_{i-1} being the vector of Fig. 1,
// so that exactly (in exact arithmetic)
//   alpha_i  = sigma_i + P / X                         (Eq. 4)
//   d_i      = P / X,   ||z_i - alpha_i q_i||^2 nu_i^2 = Y - P d_i =: s2_i
//   beta_{i-1} = nu_i / (g_{i-1} nu_{i-1})               (a posteriori, exact)
//   g_i = 1 / sqrt(s2_i),  e_{i+1} = sqrt(s2_i) / X.
// The stencil shift sigma_i only moves rounding: any value gives the same T
// in exact arithmetic.  It predicts alpha_i so that s2 is free of
// cancellation (Y ~ s2): the previous step's alpha_i where there is one (T
// changes little between steps), else alpha_{i-2} (the Krylov vectors of a
// packet with a negative-energy admixture alternate between the two bands),
// else alpha_{i-1}.  beta_{i-1} is taken from the measured norm of the next
// vector rather than from s2, so the tridiagonal T of Fig. 1 is reproduced
// to rounding.
//
// Work split: the tiles of all problems form one list of T tiles; persistent
// CTA c of G takes a contiguous chunk of T / G or T / G + 1 tiles.  A CTA may hold SUB independent tile workers (groups
// of warps with their own tile buffer and named barrier) that take the
// chunk's tiles in turn, so that one CTA per SM still overlaps one worker's
// loads with another's arithmetic.  Per problem it touches, a CTA writes one
// partial (P, Y, X) into slot c - (first CTA of that problem) and adds its
// tile count to the problem's ticket; the CTA that completes a problem sums
// that problem's slots in a fixed order (deterministic, no floating-point
// atomics) and updates its scalars.
//
// exp(-i T dt) e_1 (Sec. 4) is evaluated on one warp by a Chebyshev expansion
// over an a-priori spectral interval of H (Jacobi-Anger coefficients computed
// on the host).  The paper diagonalises T; on this GPU FP64 division and
// square root have latencies of several hundred cycles, which would make a
// serial eigensolver dominate small steps, while the Chebyshev recurrence is
// FMA-only and warp-parallel.  Both give exp(-i T dt) e_1 to rounding.
//
// Precision: S = double is the FP64 path (complex128 fields; the products in
// 60-bit fixed point, dirac_fixed.cuh).  S = float is the mixed path:
// complex64 basis and y^, FP32 stencil, warp sums converted to FP64, FP64
// scalars; q^_1 is the complex128 state itself (passes 1-2 read it).
#pragma once
#include <cuda.h>           // CUtensorMap (the type only; the library calls the driver through the runtime)
#include <cuda_runtime.h>
#include <stdint.h>

#include <cuda/atomic>
#include <type_traits>

#include "dirac_fixed.cuh"

namespace dirac {

constexpr int KMAX = 32;        // Krylov dimension limit (one warp holds T)
constexpr int CHEB_MAX = 160;   // Chebyshev terms limit
constexpr int ERR_NONFINITE = 4;
constexpr int TILE_W = 32;      // tile width in sites (one warp)

using vec4 = double4_32a;       // one site: (u.re, u.im, d.re, d.im)

// Coefficients one pass needs, prepared by the finisher of the pass before
// (FP64 values and FP32 copies, so that no thread converts on the FP64 pipe).
struct PassCoef {
  double g, gd, e, au0, ad0;          // q^ = g y^ - gd q^_prev; y^ -= e q^_prev; diagonals
  float gf, gdf, ef, au_hi, au_lo, ad_hi, ad_lo;
  float yexp;                         // FP64 path: the pass stores 2^yexp y^ (an integer; 0 on the mixed path)
};

__host__ __device__ inline PassCoef make_coef(double g, double gd, double e, double au0, double ad0,
                                              float yexp = 0.f) {
  PassCoef c;
  c.g = g; c.gd = gd; c.e = e; c.au0 = au0; c.ad0 = ad0;
  c.gf = (float)g; c.gdf = (float)gd; c.ef = (float)e;
  // the diagonals (up to ~2 m c^2) as a rounded float plus its remainder, so
  // that on the FP32 path their rounding does not act as a constant
  // perturbation of the mass term
  c.au_hi = (float)au0; c.au_lo = (float)(au0 - (double)c.au_hi);
  c.ad_hi = (float)ad0; c.ad_lo = (float)(ad0 - (double)c.ad_hi);
  c.yexp = yexp;
  return c;
}

struct DevState {
  PassCoef pc_cur;          // coefficients of the next pass to run
  PassCoef pc_prev;         // those of the last accepted pass (its stencil shift and coupling)
  int cur_pass;             // the next pass to run (1-based; 0 reads as 1)
  int redo_left;            // re-runs of a pass still allowed in this step
  double alpha[KMAX + 2];   // T diagonal of H - s, index 1..k
  double beta[KMAX + 2];    // beta[i] couples i and i+1; beta[k] = beta_k estimate
  double nu[KMAX + 2];      // ||q^_i||
  double inv_nu[KMAX + 2];  // 1 / ||q^_i||
  double sigma[KMAX + 2];   // stencil shift of pass i
  double coef_re[KMAX + 2]; // recombination coefficients C_j, j = 1..k
  double coef_im[KMAX + 2];
  double scale;             // running max(|alpha_j + s|, beta_j) for breakdown
  double psi_norm, energy, err_est, cum_err, beta_last, kappa_max;
  int stopped;              // passes of this step are done (or an error is pending)
  int k_used, breakdown, error, sigma_valid;
  unsigned counter;         // tiles of the running pass completed so far
};

struct ChebParams {
  int n;                    // number of terms
  double c0;                // centre of the spectral interval of H - s
  double inv_half;          // 1 / half width
  double ph_re, ph_im;      // exp(-i (c0 + s) dt)
  double cr[CHEB_MAX];      // eps_n (-i)^n J_n(half * dt), real part
  double ci[CHEB_MAX];      //                               imaginary part
};

// c * A of one step (electron: p - qA = p + A), FP64 and as FP32 pairs
// (rounded value and remainder)
struct FieldStep {
  double cAx, cAy;
  float cAxf, cAyf, cAxf_lo, cAyf_lo;
};

// One independent propagation problem.
struct Problem {
  int nx, ny, tiles_x, tile_begin, ntiles;   // tiles of TILE_W x TH sites
  int rblk_begin, rblk_count;                // recombination blocks
  const vec4* psi;          // the state (complex128), q^_1
  void* basis;              // q^_2 .. q^_m
  void* ybuf0;              // y^ ping-pong
  void* ybuf1;
  const void* V;            // potential energy in S, or NULL
  const void* Vlo;          // mixed path: V - (float)V as float, or NULL
  DevState* st;
  double* partials;         // 3 doubles per slot
  const ChebParams* cheb;
  double kx, ky, shift;     // c/(2dx) (order 2) or c/(12dx) (order 4); energy shift
  float kxf, kyf;           // kx, ky rounded to FP32
  float kxf_lo, kyf_lo;     // and their remainders
  int tma;                  // the mixed one-launch step stages tiles by tensor copies (maps valid)
  int vbe;                  // FP64 path: exponent field of max |V| (0: V = 0)
  PassCoef probe_coef;      // coefficients of the probe pass (stencil shift 0)
};

// Tensor maps of one problem for the bulk tensor copies of the mixed
// one-launch step, each with a box of one tile and its halo and zeros
// outside the grid: `basis` covers the complex64 basis vectors q^_2 ..
// (packed, nx ny 16 bytes apart) as a 3D FP32 tensor {4 nx, ny, vectors},
// `ybuf` the two y^ buffers as {4 nx, ny, 2}, `psi` the complex128 state as a
// 2D FP64 tensor {4 nx, ny}.
struct TmaMaps {
  CUtensorMap basis;
  CUtensorMap ybuf;
  CUtensorMap psi;
};

struct LaunchParams {
  const Problem* probs;
  const TmaMaps* maps;      // one per problem (mixed one-launch step only), else NULL
  int redo_budget;          // re-runs allowed per step (the spare launches)
  double kappa_redo;        // re-run a pass whose ||y^||^2 / s2 exceeds this
  DevState* states;         // one per problem, same order
  const FieldStep* fields;  // fields[step * fstride + problem]
  int fstride;              // 0: one FieldStep per problem for every step
  int nprob, total_tiles;
  int chunk_q, chunk_r;     // tiles per CTA: q + 1 for the first r CTAs, then q
  int pass, m, probe;
  int conj_coef;            // 1: backward step (dt < 0): exp(+i H |dt|), the conjugate coefficients
  int async_tiles;          // FP32 basis: stage passes >= 3 by asynchronous copies (many tiles per CTA)
  int iso;                  // FP64 path: kx = ky in every problem (host: picks the kernel)
  int diri;                 // Dirichlet boundaries (kernels that take the boundary at run time)
  double mcc, dt, tol;      // dt = |dt|
  const int* step;          // step counter of the running call (index into fields)
};

struct RecombParams {
  const Problem* probs;
  const int* blk_prob;      // problem of each block
  int* step;                // advanced once per step
  int redo_budget;
};

// ---------------------------------------------------------------------------
// small helpers
// ---------------------------------------------------------------------------
template <class S>
__device__ __forceinline__ S warp_sum(S v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---------------------------------------------------------------------------
// compensated FP32 arithmetic (value s plus error accumulator e)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& r) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  r = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// s + e  +=  (kh + kl) * a
__device__ __forceinline__ void acc_prod(float kh, float kl, float a, float& s, float& e) {
  const float p = __fmul_rn(kh, a);
  const float pe = fmaf(kh, a, -p);
  float t, r;
  two_sum(s, p, t, r);
  s = t;
  e = __fadd_rn(e, __fadd_rn(pe, r));
  e = fmaf(kl, a, e);
}
// grid coordinate -> array index; `outside` marks a Dirichlet zero
template <bool DIRI>
__device__ __forceinline__ int wrap(int g, int n, bool& outside) {
  if (g >= 0 && g < n) { outside = false; return g; }
  if (DIRI) { outside = true; return 0; }
  outside = false;
  int r = g % n;
  return r < 0 ? r + n : r;
}

// asynchronous 16-byte global -> shared copy (bytes = 0: zero fill, nothing read)
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem, int bytes) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(gmem), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit_wait() {
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

// read-only (non-coherent) loads: the inputs of a pass are not written
// during it, and the compiler may then move these loads ahead of the shared
// memory stores in between
__device__ __forceinline__ vec4 ldg4(const vec4* p) {
  const double2* q = reinterpret_cast<const double2*>(p);
  const double2 a = __ldg(q), b = __ldg(q + 1);
  vec4 r;
  r.x = a.x; r.y = a.y; r.z = b.x; r.w = b.y;
  return r;
}
__device__ __forceinline__ float4 ldg4(const float4* p) { return __ldg(p); }

// plain (coherent) loads for the one-launch step: its own earlier passes
// wrote the data, so the read-only path may not serve it; the grid barrier's
// acquire orders these loads after the other CTAs' stores
__device__ __forceinline__ vec4 ldw4(const vec4* p) {
  const double2* q = reinterpret_cast<const double2*>(p);
  const double2 a = q[0], b = q[1];
  vec4 r;
  r.x = a.x; r.y = a.y; r.z = b.x; r.w = b.y;
  return r;
}
__device__ __forceinline__ float4 ldw4(const float4* p) { return *p; }

template <bool COHERENT, class T>
__device__ __forceinline__ T ld4(const T* p) {
  if constexpr (COHERENT) return ldw4(p);
  else return ldg4(p);
}

template <class To, class From>
__device__ __forceinline__ void cvt4(const From& a, To (&o)[4]) {
  o[0] = (To)a.x; o[1] = (To)a.y; o[2] = (To)a.z; o[3] = (To)a.w;
}

// ---------------------------------------------------------------------------
// exp(-i T dt) e_1 on one warp: lane j holds component j+1 (k <= 32).
// X = (T - c0) / half has its spectrum in [-1, 1]; exp(-i R X) with
// R = half * dt is sum_n eps_n (-i)^n J_n(R) T_n(X) (Jacobi-Anger), summed
// with the three-term Chebyshev recurrence T_{n+1} = 2 X T_n - T_{n-1}.
// ---------------------------------------------------------------------------
__device__ inline void cheb_expm_e1(const ChebParams& cp, int k, double alpha_j, double beta_lo,
                                    double beta_hi, double& vr, double& vi) {
  // lane j holds alpha_{j+1} and the couplings to its neighbours (0 outside)
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  double a = 0.0, bl = 0.0, bh = 0.0;
  if (lane < k) {
    a = (alpha_j - cp.c0) * cp.inv_half;
    if (lane >= 1) bl = beta_lo * cp.inv_half;
    if (lane + 1 < k) bh = beta_hi * cp.inv_half;
  }
  double t0 = (lane == 0) ? 1.0 : 0.0;
  double up = __shfl_up_sync(full, t0, 1);
  double dn = __shfl_down_sync(full, t0, 1);
  double t1 = fma(a, t0, fma(bl, up, bh * dn));
  double r = cp.cr[0] * t0 + cp.cr[1] * t1;
  double im = cp.ci[0] * t0 + cp.ci[1] * t1;
  const double a2 = 2.0 * a, bl2 = 2.0 * bl, bh2 = 2.0 * bh;
  for (int n = 2; n < cp.n; ++n) {
    up = __shfl_up_sync(full, t1, 1);
    dn = __shfl_down_sync(full, t1, 1);
    const double t2 = fma(a2, t1, fma(bl2, up, fma(bh2, dn, -t0)));
    r = fma(cp.cr[n], t2, r);
    im = fma(cp.ci[n], t2, im);
    t0 = t1;
    t1 = t2;
  }
  vr = r * cp.ph_re - im * cp.ph_im;
  vi = r * cp.ph_im + im * cp.ph_re;
}

// ---------------------------------------------------------------------------
// Scalar update of one problem after pass i: run by one warp with the grid
// totals P, Y, X in every lane.  Values written by earlier launches are read
// with plain loads up front; new values travel by shuffles.  rsqrt gives
// sqrt(X), 1/X, sqrt(s2) and 1/sqrt(s2) with few dependent FP64 operations.
// ---------------------------------------------------------------------------
// FX (the FP64 path): the pass stores 2^yexp y^ with yexp an integer chosen
// before it, and g = 1 on that vector: forming q^ then takes one multiply-add
// per number instead of two, and no scale can overflow.  P and Y come in for
// the scaled vector.
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }
// floor(log2 x) of a positive normal number; 0 for zero
__device__ __forceinline__ int log2_floor(double x) { return x > 0.0 ? fx::exp_field(x) - 1023 : 0; }
__device__ __forceinline__ float next_yexp(double beta_pred, double nu) {
  const int e = -(log2_floor(beta_pred) + log2_floor(nu));
  return (float)max(-1000, min(1000, e));
}

template <bool FX>
__device__ inline void finish_pass(const LaunchParams& lp, const Problem* pr, DevState* st, int i, double P,
                                   double Y, double X) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const double shift = pr->shift;
  const bool ok = isfinite(P) && isfinite(Y) && isfinite(X) && X > 0.0;
  // psi = 0 exactly: exp(-i H dt) 0 = 0, a step that changes nothing
  const bool zero = X == 0.0 && P == 0.0 && Y == 0.0;
  if (lp.probe) {   // Rayleigh quotient of psi: the first stencil shift
    if (lane == 0) {
      if (ok || zero) {
        const double s1 = ok ? P / X : 0.0;   // the probe ran with stencil shift 0
        st->sigma[1] = s1;
        st->pc_cur = make_coef(1.0, 0.0, 0.0, lp.mcc - shift - s1, -lp.mcc - shift - s1,
                               FX && ok ? next_yexp(sqrt(Y / X), sqrt(X)) : 0.f);
        st->cur_pass = 1;
        st->redo_left = lp.redo_budget;
        st->sigma_valid = 1;
      } else {
        st->error = ERR_NONFINITE; st->stopped = 1;
      }
    }
    return;
  }
  if (zero && i == 1) {   // recombination with C_1 = 0 keeps psi = 0
    if (lane == 0) {
      st->nu[1] = 0.0;
      st->inv_nu[1] = 0.0;
      st->alpha[1] = st->sigma[1];
      st->beta[1] = 0.0;
      st->coef_re[1] = 0.0;
      st->coef_im[1] = 0.0;
      st->psi_norm = 0.0;
      st->energy = 0.0;          // no state, no energy
      st->err_est = 0.0;
      st->k_used = 1;
      st->breakdown = 1;
      st->beta_last = 0.0;
      st->pc_cur = make_coef(1.0, 0.0, 0.0, lp.mcc - shift - st->sigma[1], -lp.mcc - shift - st->sigma[1]);
      st->sigma_valid = 1;
      st->stopped = 1;
    }
    return;
  }
  if (!ok) {
    if (lane == 0) { st->error = ERR_NONFINITE; st->stopped = 1; }
    return;
  }
  // earlier T entries (lane j: component j+1), issued before the scalar chain
  const double a_old = (lane + 1 < i) ? st->alpha[lane + 1] : 0.0;
  const double b_old = (lane + 2 < i) ? st->beta[lane + 1] : 0.0;   // exact beta_{j+1}
  const double invnu_old = (lane + 1 < i) ? st->inv_nu[lane + 1] : 0.0;
  const double sigma = st->sigma[i];
  const double scale_old = (i == 1) ? 0.0 : st->scale;
  const double bhat_prev = (i == 1) ? 0.0 : st->beta[i - 1];       // estimate from pass i-1
  const double nu1_old = (i == 1) ? 0.0 : st->nu[1];
  const double alpha1_old = (i == 1) ? 0.0 : st->alpha[1];
  const double psi_norm_old = st->psi_norm, cum_old = st->cum_err;
  const int redo_left = st->redo_left;
  // candidates for the next pass's stencil shift: alpha_{i+1} of the previous
  // step (still in place: this step has not reached pass i + 1) and
  // alpha_{i-1} of this one
  const int k_prev = st->k_used;
  const double alpha_next_prev = (i + 1 <= k_prev && i + 1 <= KMAX) ? st->alpha[i + 1] : 0.0;
  const double alpha_im1 = (i >= 2) ? st->alpha[i - 1] : 0.0;
  const PassCoef pc_now = st->pc_cur;
  // FX: 2^-yexp of this pass and of the one before, the last estimate of
  // beta_{i+1} and 1 / nu_{i-1}
  const double unscale = FX ? pow2(-(int)pc_now.yexp) : 1.0;
  const double unscale_prev = (FX && i >= 2) ? pow2(-(int)st->pc_prev.yexp) : 1.0;
  const double invnu_im1 = (FX && i >= 2) ? st->inv_nu[i - 1] : 0.0;
  const double beta_next_prev = (FX && i + 1 <= k_prev && i + 1 <= KMAX) ? st->beta[i + 1] : 0.0;
  const double beta1_old = (FX && i >= 2) ? st->beta[1] : 0.0;
  __syncwarp();   // every lane has read the state before lane 0 updates it

  // scalar chain (every lane computes it; no broadcast needed)
  const double y = rsqrt(X);            // 1 / nu_i
  const double nu = X * y;
  const double rX = y * y;
  const double dd = P * rX;             // alpha_i - sigma_i
  const double alpha = FX ? fma(dd, unscale, sigma) : sigma + dd;
  const double s2 = fma(-P, dd, Y);     // nu_i^2 beta_i^2 (estimate)
  const double rs = s2 > 0.0 ? rsqrt(s2) : 0.0;
  const double sq = s2 > 0.0 ? s2 * rs : 0.0;
  const double beta_hat = FX ? sq * y * unscale : sq * y;
  // exact beta_{i-1} from the measured norm
  const double bprev = FX ? nu * invnu_im1 * unscale_prev : nu * bhat_prev;
  // The stencil shift sigma_i was too far from alpha_i for the precision of
  // y^ (s2 is then cancellation noise): run pass i again with sigma_i =
  // alpha_i, which makes s2 ~ Y.  Everything derived from X (nu, beta_{i-1})
  // is unchanged by the re-run.
  if ((!(s2 > 0.0) || Y > lp.kappa_redo * s2) && redo_left > 0) {
    if (lane == 0) {
      st->redo_left = redo_left - 1;
      st->sigma[i] = alpha;
      st->pc_cur = make_coef(pc_now.g, pc_now.gd, pc_now.e, lp.mcc - shift - alpha,
                             -lp.mcc - shift - alpha, pc_now.yexp);
      if (s2 > 0.0) st->kappa_max = fmax(st->kappa_max, Y * rs * rs);
    }
    return;
  }
  double scale = fmax(scale_old, fabs(alpha + shift));
  if (i > 1) scale = fmax(scale, bprev);
  const int brk = beta_hat <= 1e-12 * scale;
  int stop = (i >= lp.m) || brk;
  const double nu1 = (i == 1) ? nu : nu1_old;
  const double psi_norm = (i == 1) ? nu : psi_norm_old;
  if (lane == 0) {
    st->nu[i] = nu;
    st->inv_nu[i] = y;
    st->alpha[i] = alpha;
    st->beta[i] = beta_hat;
    if (i > 1) st->beta[i - 1] = bprev;
    st->scale = scale;
    if (i == 1) { st->psi_norm = nu; st->energy = alpha + shift; }
    if (s2 > 0.0) st->kappa_max = fmax(st->kappa_max, Y * rs * rs);
    if (!stop) {
      // The stencil shift of pass i + 1, a prediction of alpha_{i+1} (any
      // value is exact; a close one keeps s2 free of cancellation).  T hardly
      // changes from one step to the next -- for static fields its entries
      // are moments of H in psi, which the propagation conserves -- so the
      // previous step's alpha_{i+1} is the best guess when that step got so
      // far.  Else alpha_{i-1}: the Krylov vectors of a positive-energy packet
      // with a small negative-energy admixture alternate between the two
      // bands, so alpha_{i+1} is close to alpha_{i-1}, not to alpha_i.
      const double sig = (i + 1 <= k_prev) ? alpha_next_prev : (i >= 2 ? alpha_im1 : alpha);
      st->sigma[i + 1] = sig;
      st->pc_prev = pc_now;
      if constexpr (FX)
        st->pc_cur = make_coef(1.0, dd, s2 * rX * unscale, lp.mcc - shift - sig, -lp.mcc - shift - sig,
                               next_yexp(beta_next_prev > 0.0 ? beta_next_prev : beta_hat, sq));
      else
        st->pc_cur = make_coef(rs, rs * dd, sq * rX, lp.mcc - shift - sig, -lp.mcc - shift - sig);
      st->cur_pass = i + 1;
    }
  }
  // this lane's row of T^(i)
  const double a_j = (lane + 1 == i) ? alpha : a_old;
  const double b_hi = (lane + 2 == i) ? bprev : b_old;               // couples j+1, j+2
  const double b_lo = __shfl_up_sync(full, b_hi, 1);                 // couples j, j+1
  const double inv_nu_j = (lane + 1 == i) ? y : invnu_old;
  double vr = 0.0, vi = 0.0;
  bool have_v = false;
  if (!stop && lp.tol > 0.0) {   // adaptive Krylov dimension (Sec. 4, Eq. 18)
    cheb_expm_e1(*pr->cheb, i, a_j, b_lo, b_hi, vr, vi);
    have_v = true;
    const double vk = __shfl_sync(full, sqrt(vr * vr + vi * vi), i - 1);
    stop = (beta_hat * lp.dt * vk <= lp.tol);
  }
  if (!stop) return;
  if (!have_v) cheb_expm_e1(*pr->cheb, i, a_j, b_lo, b_hi, vr, vi);
  // C_j = nu_1 / nu_j * v_j applied to q^_j; Eq. 18 estimate from v_k
  const double vk = __shfl_sync(full, sqrt(vr * vr + vi * vi), i - 1);
  if (lane < i) {
    const double f = nu1 * inv_nu_j;
    st->coef_re[lane + 1] = f * vr;
    st->coef_im[lane + 1] = lp.conj_coef ? -f * vi : f * vi;   // T real: exp(+iT dt) e_1 = conj(exp(-iT dt) e_1)
  }
  if (lane == 0) {
    const double err = lp.dt * beta_hat * psi_norm * vk;
    st->err_est = err;
    st->cum_err = cum_old + err;
    st->k_used = i;
    st->breakdown = brk;
    st->beta_last = beta_hat;
    const double s1 = (i == 1) ? alpha : alpha1_old;   // next step's first shift
    st->sigma[1] = s1;
    const double b1 = (i == 1) ? beta_hat : (i == 2 ? bprev : beta1_old);
    st->pc_cur = make_coef(1.0, 0.0, 0.0, lp.mcc - shift - s1, -lp.mcc - shift - s1,
                           FX ? next_yexp(b1, nu1) : 0.f);
    st->sigma_valid = 1;
    st->stopped = 1;
  }
}

// ---------------------------------------------------------------------------
// One Lanczos iteration over every problem of the table: stencil product
// with fused reductions.
//
// S    arithmetic type of the stencil (double: FP64 path; float: mixed path)
// R    stencil half width (1: order 2, 2: order 4)
// TH   tile height in sites (tiles are TILE_W x TH; TH / RPT warps per tile
//      worker, RPT rows per thread)
//
// Each problem runs its own next pass (DevState::cur_pass), so that a pass
// can be re-run (see finish_pass) without the host knowing.  q^_{i-1} (and
// psi) are complex128 on the FP64 path and in passes 1-2 of the mixed path
// (whose q^_1 is the FP64 state itself), else complex64.
//
// Thread (tx, tg) handles column tx and rows tg, tg + NG, ..., so every warp
// touches one contiguous row segment per access.  The tile and a
// cross-shaped halo of q^_i are formed in shared memory from y^_{i-1} and
// q^_{i-1}.
// ---------------------------------------------------------------------------
// CTAs per SM of the FP32 pass (128 or 256 threads each)
template <int TH>
__host__ __device__ constexpr int min_blocks() { return TH == 32 ? 4 : 8; }

// rows per thread: four, except two on FP64 16-row tiles, which keep eight
// warps per tile worker and halve the unit of work: a grid of a few tiles per
// worker then ends with a shorter partial round
template <class S, int TH>
__host__ __device__ constexpr int rows_per_thread() { return (sizeof(S) == sizeof(double) && TH == 16) ? 2 : 4; }

// tile workers per CTA: two on the FP64 path (one CTA per SM), one otherwise
template <class S>
__host__ __device__ constexpr int sub_workers() { return sizeof(S) == sizeof(double) ? 2 : 1; }

// shared memory of one FP64 tile worker: q^_i on the tile and its halo in
// fixed point, the upper and the lower components in separate halves (16 bytes
// per site each, so that a warp's row is read without bank conflicts), then a
// table of coefficients per warp and the exponents of two tiles
constexpr int COEF_SLOTS = 16;   // eight per half
template <int R, int TH>
__host__ __device__ constexpr int half_sites() { return (TH + 2 * R) * (TILE_W + 2 * R); }
template <int R, int TH>
__host__ __device__ constexpr size_t worker_bytes() {
  return 2 * sizeof(longlong2) * half_sites<R, TH>() +
         sizeof(int2) * COEF_SLOTS * (TH / rows_per_thread<double, TH>()) + 32;
}

// Chunks of the tile list: CTA c takes q + 1 tiles if c < r, else q (q = T / G,
// r = T % G), starting at c q + min(c, r).  The CTA whose chunk holds tile t:
__device__ __forceinline__ int cta_of_tile(int t, int q, int r) {
  const int big = r * (q + 1);
  return t < big ? t / (q + 1) : r + (t - big) / q;
}

// Dynamic shared memory of a pass kernel (the FP32 pass keeps its tile in a
// static array)
template <class S, int R, int TH, int SUB>
__host__ __device__ constexpr size_t dyn_smem_bytes() {
  return sizeof(S) == sizeof(float) ? 0 : SUB * worker_bytes<R, TH>();
}

// This CTA's share of a problem, the warps' sums in red[], -> one partial per
// (problem, CTA) slot.  COOP = false: then the problem's ticket, and the CTA
// that completes the problem sums its slots and updates its scalars.  COOP =
// true (one-launch step): the partial goes to coop_slots[3 blockIdx.x ..] and
// the caller goes on.
template <bool FX, bool COOP, int NW>
__device__ __forceinline__ void pass_sums(const LaunchParams& lp, const Problem* pr, int i, int seg_tiles,
                                          double (*red)[3], int* last_flag, double* coop_slots) {
  constexpr int NT = 32 * NW;
  const int cq = lp.chunk_q, cr = lp.chunk_r;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (warp == 0) {
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    if (lane < NW) { s0 = red[lane][0]; s1 = red[lane][1]; s2 = red[lane][2]; }
#pragma unroll
    for (int o = (NW > 16 ? 16 : 8); o > 0; o >>= 1) {   // NW <= 32 warps
      s0 += __shfl_xor_sync(0xffffffffu, s0, o);
      s1 += __shfl_xor_sync(0xffffffffu, s1, o);
      s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    }
    if (lane == 0) {
      if constexpr (COOP) {
        coop_slots[3 * blockIdx.x + 0] = s0;
        coop_slots[3 * blockIdx.x + 1] = s1;
        coop_slots[3 * blockIdx.x + 2] = s2;
        *last_flag = 0;
      } else {
        const int slot = blockIdx.x - cta_of_tile(pr->tile_begin, cq, cr);
        pr->partials[3 * slot + 0] = s0;
        pr->partials[3 * slot + 1] = s1;
        pr->partials[3 * slot + 2] = s2;
        // release our partial / acquire everybody else's
        cuda::atomic_ref<unsigned, cuda::thread_scope_device> ticket(pr->st->counter);
        *last_flag = (ticket.fetch_add((unsigned)seg_tiles, cuda::memory_order_acq_rel) + seg_tiles ==
                     (unsigned)pr->ntiles);
      }
    }
  }
  __syncthreads();
  if (!COOP && *last_flag) {
    // the problem is complete: the whole CTA sums its slots in a fixed
    // order (thread-strided, the warp tree, then the warps in turn), the
    // loads of SB slots per thread in flight at once, so that a pass of
    // eight CTAs per SM waits for two L2 round trips here, not five
    const int cta_lo = cta_of_tile(pr->tile_begin, cq, cr);
    const int nslots = cta_of_tile(pr->tile_begin + pr->ntiles - 1, cq, cr) - cta_lo + 1;
    constexpr int SB = 5;
    double t0 = 0.0, t1 = 0.0, t2 = 0.0;
    for (int s0 = threadIdx.x; s0 < nslots; s0 += SB * NT) {
      double v[SB][3];
#pragma unroll
      for (int k = 0; k < SB; ++k) {
        const int s = s0 + k * NT;
        const double* ps = pr->partials + 3 * (s < nslots ? s : 0);
        v[k][0] = s < nslots ? __ldcg(ps + 0) : 0.0;
        v[k][1] = s < nslots ? __ldcg(ps + 1) : 0.0;
        v[k][2] = s < nslots ? __ldcg(ps + 2) : 0.0;
      }
#pragma unroll
      for (int k = 0; k < SB; ++k) { t0 += v[k][0]; t1 += v[k][1]; t2 += v[k][2]; }
    }
    t0 = warp_sum(t0);
    t1 = warp_sum(t1);
    t2 = warp_sum(t2);
    if (lane == 0) { red[warp][0] = t0; red[warp][1] = t1; red[warp][2] = t2; }
    __syncthreads();
    if (warp == 0) {
      t0 = red[0][0]; t1 = red[0][1]; t2 = red[0][2];
#pragma unroll
      for (int w = 1; w < NW; ++w) { t0 += red[w][0]; t1 += red[w][1]; t2 += red[w][2]; }
      if (lane == 0) pr->st->counter = 0u;
      finish_pass<FX>(lp, pr, pr->st, i, t0, t1, t2);
    }
  }
  __syncthreads();
}

// The body of one FP32 pass over this CTA's chunk (the mixed path).
template <int R, int TH, bool DIRI, bool HAS_V>
__device__ __forceinline__ void pass_body(const LaunchParams& lp, int step) {
  using S = float;
  using T4 = float4;                        // storage of y^ and of q^_i, i >= 2
  constexpr int RPT = rows_per_thread<S, TH>();
  constexpr int NG = TH / RPT;              // row groups = warps
  constexpr int NT = 32 * NG;               // threads
  constexpr int W = TILE_W + 2 * R;
  __shared__ double red[NG][3];
  __shared__ int last_flag;

  const int cq = lp.chunk_q, cr = lp.chunk_r;
  const int t_begin = blockIdx.x * cq + min((int)blockIdx.x, cr);
  const int t_end = t_begin + cq + ((int)blockIdx.x < cr ? 1 : 0);
  const int ltid = (int)threadIdx.x;
  const int tx = ltid & 31, tg = ltid >> 5;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __shared__ __align__(32) S tile[TH + 2 * R][W][4];
  // passes >= 3: q^_{i-1} on the tile and halo, copied asynchronously
  __shared__ __align__(16) float4 qbuf[(TH + 2 * R) * W];

  // problem of the first tile (problems are sorted by tile_begin)
  int b = 0;
  {
    int lo = 0, hi = lp.nprob - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (lp.probs[mid].tile_begin <= t_begin) lo = mid; else hi = mid - 1;
    }
    b = lo;
  }
  for (int t = t_begin; t < t_end; ++b) {
    const Problem* pr = lp.probs + b;
    const DevState* st = lp.states + b;
    // independent loads first (all addresses are valid), then the branch
    const int stopped = st->stopped;
    const int i = lp.probe ? 1 : max(1, st->cur_pass);
    const PassCoef pc = lp.probe ? pr->probe_coef : st->pc_cur;
    const FieldStep fs = lp.fields[step * lp.fstride + b];
    const int seg_end = min(t_end, pr->tile_begin + pr->ntiles);
    const int seg_tiles = seg_end - t;
    if (stopped) { t = seg_end; continue; }
    const S gS = pc.gf;
    const S gdS = pc.gdf;
    const S eS = pc.ef;
    const S kx = pr->kxf, ky = pr->kyf;
    const S cAx = fs.cAxf, cAy = fs.cAyf;
    const S au_hi = pc.au_hi, au_lo = pc.au_lo;
    const S ad_hi = pc.ad_hi, ad_lo = pc.ad_lo;
    // FP32: remainders of the stencil and vector-potential coefficients
    const S kx_lo = pr->kxf_lo, ky_lo = pr->kyf_lo;
    const S cAx_lo = fs.cAxf_lo, cAy_lo = fs.cAyf_lo;
    const int nx = pr->nx, ny = pr->ny;
    const size_t n = (size_t)nx * ny;
    // this pass's vectors
    constexpr int SB = (int)sizeof(float4);
    const char* basis = static_cast<const char*>(pr->basis);
    const void* y_prev = (i >= 2) ? (((i - 1) & 1) ? pr->ybuf1 : pr->ybuf0) : nullptr;
    const void* q_prev = (i == 2) ? (const void*)pr->psi
                                  : (i >= 3 ? (const void*)(basis + (size_t)(i - 3) * n * SB) : nullptr);
    void* q_out = (i >= 2) ? (void*)(basis + (size_t)(i - 2) * n * SB) : nullptr;
    void* y_out = (i < lp.m) ? ((i & 1) ? pr->ybuf1 : pr->ybuf0) : nullptr;
    const T4* yprev = static_cast<const T4*>(y_prev);
    const bool q64 = i <= 2;                // q^_{i-1} stored as complex128
    const S* Vp = static_cast<const S*>(pr->V);   // NULL: V = 0 for this problem
    const float* Vlo = static_cast<const float*>(pr->Vlo);   // mixed path: V - (float)V, or NULL

    // q^_i at grid point (gx, gy) (zero outside for Dirichlet) into smem slot
    auto form = [&](int gx, int gy, int row, int col, S (&qp)[4]) {
      bool ox, oy;
      const int ix = wrap<DIRI>(gx, nx, ox), iy = wrap<DIRI>(gy, ny, oy);
      S q[4] = {S(0), S(0), S(0), S(0)};
      qp[0] = qp[1] = qp[2] = qp[3] = S(0);
      if (!(ox || oy)) {
        const size_t idx = (size_t)iy * nx + ix;
        if (q64) {
          const vec4* qsrc = (i == 1) ? pr->psi : static_cast<const vec4*>(q_prev);
          cvt4(ldg4(qsrc + idx), qp);
        } else {
          cvt4(ldg4(static_cast<const float4*>(q_prev) + idx), qp);
        }
        if (i == 1) {
#pragma unroll
          for (int c = 0; c < 4; ++c) q[c] = qp[c];
        } else {
          S yv[4];
          cvt4(ldg4(yprev + idx), yv);
#pragma unroll
          for (int c = 0; c < 4; ++c) q[c] = fma(-gdS, qp[c], gS * yv[c]);
        }
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) tile[row][col][c] = q[c];
    };

    S accP = S(0), accY = S(0), accX = S(0);
    // y^_i at one site from q^_i there (C) and its differences, q^_{i-1}
    // (qp) and V; stores q^_i and y^_i and accumulates P, Y, X
    auto site_update = [&](size_t idx, const S (&C)[4], const S (&dxv)[4], const S (&dyv)[4],
                           const S (&qp)[4]) {
      S au, ad, aul = au_lo, adl = ad_lo;
      if (HAS_V && Vp != nullptr) {   // V stored in S (float copy on the mixed path)
        const S v = Vp[idx];
        {
          // the FP32 sum with the diagonal (up to 2 m c^2) rounds differently at
          // every site: its error and V's own remainder go into the low part
          float ru, rd;
          two_sum(au_hi, v, au, ru);
          two_sum(ad_hi, v, ad, rd);
          const float vl = Vlo ? Vlo[idx] : 0.f;
          aul = au_lo + vl + ru;
          adl = ad_lo + vl + rd;
        }
      } else {
        au = au_hi;
        ad = ad_hi;
      }
      // C = (u.re, u.im, d.re, d.im); dxv/dyv likewise
      S yv[4];
      // upper: (mc^2+V-s-sigma) u + c[-i D_x d - D_y d + (A_x - i A_y) d]
      yv[0] = au * C[0] + kx * dxv[3] - ky * dyv[2] + cAx * C[2];
      yv[1] = au * C[1] - kx * dxv[2] - ky * dyv[3] + cAx * C[3];
      // lower: (-mc^2+V-s-sigma) d + c[-i D_x u + D_y u + (A_x + i A_y) u]
      yv[2] = ad * C[2] + kx * dxv[1] + ky * dyv[0] + cAx * C[0];
      yv[3] = ad * C[3] - kx * dxv[0] + ky * dyv[1] + cAx * C[1];
      {
        yv[0] = fma(cAy, C[3], yv[0]);
        yv[1] = fma(-cAy, C[2], yv[1]);
        yv[2] = fma(-cAy, C[1], yv[2]);
        yv[3] = fma(cAy, C[0], yv[3]);
      }
      {
        yv[0] = fma(aul, C[0], fma(kx_lo, dxv[3], fma(-ky_lo, dyv[2], fma(cAx_lo, C[2], yv[0]))));
        yv[1] = fma(aul, C[1], fma(-kx_lo, dxv[2], fma(-ky_lo, dyv[3], fma(cAx_lo, C[3], yv[1]))));
        yv[2] = fma(adl, C[2], fma(kx_lo, dxv[1], fma(ky_lo, dyv[0], fma(cAx_lo, C[0], yv[2]))));
        yv[3] = fma(adl, C[3], fma(-kx_lo, dxv[0], fma(ky_lo, dyv[1], fma(cAx_lo, C[1], yv[3]))));
        {
          yv[0] = fma(cAy_lo, C[3], yv[0]);
          yv[1] = fma(-cAy_lo, C[2], yv[1]);
          yv[2] = fma(-cAy_lo, C[1], yv[2]);
          yv[3] = fma(cAy_lo, C[0], yv[3]);
        }
      }
      if (i >= 2) {
#pragma unroll
        for (int q = 0; q < 4; ++q) yv[q] = fma(-eS, qp[q], yv[q]);
      }
      if (!lp.probe) {
        if (q_out) {
          T4 o; o.x = C[0]; o.y = C[1]; o.z = C[2]; o.w = C[3];
          static_cast<T4*>(q_out)[idx] = o;
        }
        if (y_out) {
          T4 o; o.x = yv[0]; o.y = yv[1]; o.z = yv[2]; o.w = yv[3];
          static_cast<T4*>(y_out)[idx] = o;
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        accP = fma(C[q], yv[q], accP);
        accY = fma(yv[q], yv[q], accY);
        accX = fma(C[q], C[q], accX);
      }
    };
    // the stencil on the formed tile; qprev(k, r, c) gives q^_{i-1} of row k
    auto stencil_rows = [&](int x0, int y0, auto&& qprev) {
#pragma unroll
      for (int k = 0; k < RPT; ++k) {
        const int ry = tg + k * NG;
        const int x = x0 + tx, y = y0 + ry;
        if (x < nx && y < ny) {
          const size_t idx = (size_t)y * nx + x;
          const int r = ry + R, c = tx + R;
          S C[4], dxv[4], dyv[4], qp[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            C[q] = tile[r][c][q];
            dxv[q] = tile[r][c + 1][q] - tile[r][c - 1][q];
            dyv[q] = tile[r + 1][c][q] - tile[r - 1][c][q];
            if constexpr (R == 2) {
              dxv[q] = fma(S(8), dxv[q], tile[r][c - 2][q] - tile[r][c + 2][q]);
              dyv[q] = fma(S(8), dyv[q], tile[r - 2][c][q] - tile[r + 2][c][q]);
            }
          }
          qprev(k, r, c, qp);
          site_update(idx, C, dxv, dyv, qp);
        }
      }
    };

    bool done_async = false;
    {
     if (!q64 && lp.async_tiles) {
      done_async = true;
      // mixed path, passes >= 3: y^_{i-1} and q^_{i-1} of the tile and its
      // halo (a full rectangle) go to shared memory by asynchronous copies,
      // all in flight at once and without registers; q^_i is formed in place
      constexpr int NS = (TH + 2 * R) * W;
      float4* const tf = reinterpret_cast<float4*>(&tile[0][0][0]);
      const float4* const qsrc = static_cast<const float4*>(q_prev);
      for (int tt = t; tt < seg_end; ++tt) {
        const int lt = tt - pr->tile_begin;
        const int x0 = (lt % pr->tiles_x) * TILE_W;
        const int y0 = (lt / pr->tiles_x) * TH;
        for (int e = ltid; e < NS; e += NT) {
          const int r = e / W, c = e - r * W;
          bool ox, oy;
          const int ix = wrap<DIRI>(x0 - R + c, nx, ox), iy = wrap<DIRI>(y0 - R + r, ny, oy);
          const bool in = !(ox || oy);
          const size_t idx = in ? (size_t)iy * nx + ix : 0;
          cp_async16(tf + e, reinterpret_cast<const float4*>(yprev) + idx, in ? 16 : 0);
          cp_async16(qbuf + e, qsrc + idx, in ? 16 : 0);
        }
        cp_async_commit_wait();
        __syncthreads();
        for (int e = ltid; e < NS; e += NT) {
          const float4 yv = tf[e], qp = qbuf[e];
          tf[e] = make_float4(fmaf(-(float)gdS, qp.x, (float)gS * yv.x), fmaf(-(float)gdS, qp.y, (float)gS * yv.y),
                              fmaf(-(float)gdS, qp.z, (float)gS * yv.z), fmaf(-(float)gdS, qp.w, (float)gS * yv.w));
        }
        __syncthreads();
        stencil_rows(x0, y0, [&](int, int r, int c, S (&qp)[4]) {
          const float4 v = qbuf[r * W + c];
          qp[0] = (S)v.x; qp[1] = (S)v.y; qp[2] = (S)v.z; qp[3] = (S)v.w;
        });
        __syncthreads();   // tile and qbuf are reused next
      }
     }
    }
    if (!done_async) {
      for (int tt = t; tt < seg_end; ++tt) {
        const int lt = tt - pr->tile_begin;
        const int x0 = (lt % pr->tiles_x) * TILE_W;
        const int y0 = (lt / pr->tiles_x) * TH;
        S qprev[RPT][4];
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
          const int r = tg + k * NG;
          form(x0 + tx, y0 + r, r + R, tx + R, qprev[k]);
        }
        constexpr int NH_ROW = 2 * R * TILE_W, NH = NH_ROW + 2 * R * TH;
        for (int h = ltid; h < NH; h += NT) {
          int row, col;
          if (h < NH_ROW) {               // rows above / below
            const int r = h / TILE_W;
            row = (r < R) ? r : TH + r;
            col = (h % TILE_W) + R;
          } else {                        // columns left / right
            const int h2 = h - NH_ROW;
            row = h2 / (2 * R) + R;
            const int c = h2 % (2 * R);
            col = (c < R) ? c : TILE_W + c;
          }
          S dummy[4];
          form(x0 + col - R, y0 + row - R, row, col, dummy);
        }
        __syncthreads();
        stencil_rows(x0, y0, [&](int k, int, int, S (&qp)[4]) {
#pragma unroll
          for (int q = 0; q < 4; ++q) qp[q] = qprev[k][q];
        });
        __syncthreads();   // the tile buffer is reused next
      }
    }
    t = seg_end;

    // this CTA's share of the problem: thread -> warp in FP32, the rest in FP64
    accP = warp_sum(accP);
    accY = warp_sum(accY);
    accX = warp_sum(accX);
    if (lane == 0) { red[warp][0] = (double)accP; red[warp][1] = (double)accY; red[warp][2] = (double)accX; }
    pass_sums<false, false, NG>(lp, pr, i, seg_tiles, red, &last_flag, nullptr);
  }
}

// The body of one FP64 pass over this CTA's chunk.  COOP = false: a launch of
// its own (lanczos_pass).  COOP = true: inside the one-launch step
// (lanczos_step): one problem, the state read from `coop_st`, and the CTA's
// partial sums written to coop_slots; the caller synchronises the grid and
// finishes.
//
// The fields are complex128 in memory; per site and pass only the formation of
// q^_i (one FP64 multiply-add per number, the scale of y^ being a power of two)
// and the final conversion of y^_i use the FP64 pipe.  The stencil, the
// coupling to q^_{i-1} and the three sums are 60-bit fixed point
// (dirac_fixed.cuh): a tile (with its halo) shares one exponent for the upper
// and one for the lower components of q^_i, another pair for q^_{i-1}, taken
// from their largest numbers; every row of the operator is one exact sum of
// products, rounded to 2^-60 of its largest term.  The sums run per tile in
// integers and over the tiles of a worker at a common exponent.
//
// Measured (GB300, FP64 step with its recombination): 1024^2, m = 20, 2.50 ->
// 1.89 ms; 4096^2, m = 10, 17.3 -> 10.7 ms; twelve problems of 93^2 .. 301^2 in
// a batch 1.18 -> 0.94 ms, against the same passes in FP64 multiply-adds, whose
// 1160 instructions a site and step kept the FP64 pipe 79 % busy.
//
// Per tile: load and form (all loads of a thread in flight at once), exponents
// -> barrier -> fixed point into shared memory, coefficients at the tile's
// scale -> barrier -> the upper, then the lower components.
template <int R, int TH, bool DIRI, bool HAS_V, bool ISO, bool COOP, int SUB>
__device__ __forceinline__ void pass_body_fx(const LaunchParams& lp, const DevState* coop_st, double* coop_slots,
                                             int step) {
  constexpr int RPT = rows_per_thread<double, TH>();
  constexpr int NG = TH / RPT;              // row groups = warps of a worker
  constexpr int NTS = 32 * NG;              // threads of a worker
  constexpr int NW = SUB * NG;              // warps
  constexpr int W = TILE_W + 2 * R;
  // bits of q^ and q^_{i-1}: the differences (2 x 2 terms; order 4: 36) and
  // the row sums then stay below 2^62
  constexpr int F = R == 1 ? 58 : 55;
  constexpr int NH_ROW = 2 * R * TILE_W, NH = NH_ROW + 2 * R * TH;
  static_assert(NH <= NTS, "one halo site per thread");
  static_assert(2 * RPT <= 8, "bounds of the per-tile sums");
  extern __shared__ __align__(32) unsigned char dyn_smem[];
  __shared__ double red[NW][3];
  __shared__ int last_flag;

  const int cq = lp.chunk_q, cr = lp.chunk_r;
  const int t_begin = blockIdx.x * cq + min((int)blockIdx.x, cr);
  const int t_end = t_begin + cq + ((int)blockIdx.x < cr ? 1 : 0);
  const int sub = (int)threadIdx.x / NTS;   // this thread's worker
  const int ltid = (int)threadIdx.x - sub * NTS;
  const int tx = ltid & 31, tg = ltid >> 5;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char* const my_smem = dyn_smem + sub * worker_bytes<R, TH>();
  longlong2* const half_u = reinterpret_cast<longlong2*>(my_smem);
  longlong2* const half_d = half_u + half_sites<R, TH>();
  int2* const kt = reinterpret_cast<int2*>(half_d + half_sites<R, TH>()) + COEF_SLOTS * tg;
  unsigned* const emax = reinterpret_cast<unsigned*>(reinterpret_cast<int2*>(half_d + half_sites<R, TH>()) +
                                                     COEF_SLOTS * NG);   // [2][4]
  auto sub_sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + sub), "r"(NTS) : "memory"); };
  if (ltid < 8) emax[ltid] = 0u;
  sub_sync();
  int par = 0;                              // which exponents the tile uses

  // problem of the first tile (problems are sorted by tile_begin)
  int b = 0;
  {
    int lo = 0, hi = lp.nprob - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (lp.probs[mid].tile_begin <= t_begin) lo = mid; else hi = mid - 1;
    }
    b = lo;
  }
  for (int t = t_begin; t < t_end; ++b) {
    const Problem* pr = lp.probs + b;
    const DevState* st = COOP ? coop_st : lp.states + b;
    // independent loads first (all addresses are valid), then the branch
    const int stopped = st->stopped;
    const int i = lp.probe ? 1 : max(1, st->cur_pass);
    const PassCoef& pc = lp.probe ? pr->probe_coef : st->pc_cur;
    const int seg_end = min(t_end, pr->tile_begin + pr->ntiles);
    const int seg_tiles = seg_end - t;
    if (stopped) { t = seg_end; continue; }
    const double gd = pc.gd;
    const int yexp = (int)pc.yexp;
    const int nx = pr->nx, ny = pr->ny;
    const size_t n = (size_t)nx * ny;
    // this pass's vectors
    vec4* const basis = static_cast<vec4*>(pr->basis);
    const vec4* const yprev = static_cast<const vec4*>((i & 1) ? pr->ybuf0 : pr->ybuf1);
    const vec4* const qsrc = i <= 2 ? pr->psi : basis + (size_t)(i - 3) * n;   // q^_{i-1} (q^_1 if i = 1)
    vec4* const q_out = (i >= 2 && !lp.probe) ? basis + (size_t)(i - 2) * n : nullptr;
    vec4* const y_out = (i < lp.m && !lp.probe) ? static_cast<vec4*>((i & 1) ? pr->ybuf1 : pr->ybuf0) : nullptr;
    const double* const Vp = static_cast<const double*>(pr->V);   // NULL: V = 0 for this problem
    const FieldStep* const fs = lp.fields + step * lp.fstride + b;
    const bool has_ax = fs->cAx != 0.0, has_ay = fs->cAy != 0.0;
    // this lane's coefficient: slots 0 diagonal, 1 kx, 2 ky, 3 c A_x, 4 c A_y,
    // 5 coupling, 6 V (its exponent alone) of the upper (lanes 0-7) and the
    // lower row (8-15)
    const int cj = lane & 7, ch = (lane >> 3) & 1;
    double my_coef = 0.0;
    if (cj == 0) my_coef = ch ? pc.ad0 : pc.au0;
    if (cj == 1) my_coef = pr->kx;
    if (cj == 2) my_coef = pr->ky;
    if (cj == 3) my_coef = fs->cAx;
    if (cj == 4) my_coef = fs->cAy;
    if (cj == 5) my_coef = i >= 2 ? pc.e : 0.0;
    const int my_xe = cj == 6 ? (HAS_V && Vp ? pr->vbe : 0) : fx::exp_field(my_coef);
    bool bad = __any_sync(0xffffffffu, my_xe == 0x7ff);

    // q^_i at a site, and q^_{i-1} there (zero if i = 1)
    auto load = [&](size_t idx, double (&q)[4], double (&qp)[4]) {
      cvt4(ld4<COOP>(qsrc + idx), qp);
      if (i == 1) {
#pragma unroll
        for (int c = 0; c < 4; ++c) { q[c] = qp[c]; qp[c] = 0.0; }
      } else {
        double yv[4];
        cvt4(ld4<COOP>(yprev + idx), yv);
#pragma unroll
        for (int c = 0; c < 4; ++c) q[c] = fma(-gd, qp[c], yv[c]);
      }
    };
    // the same at grid point (gx, gy), wrapped, or zero outside for Dirichlet
    auto form = [&](int gx, int gy, double (&q)[4], double (&qp)[4]) {
      bool ox, oy;
      const int ix = wrap<DIRI>(gx, nx, ox), iy = wrap<DIRI>(gy, ny, oy);
      q[0] = q[1] = q[2] = q[3] = 0.0;
      qp[0] = qp[1] = qp[2] = qp[3] = 0.0;
      if (ox || oy) return;
      load((size_t)iy * nx + ix, q, qp);
    };
    auto mag = [](double x) { return (unsigned)__double2hiint(x) << 1; };   // orders by |x| (to 20 bits)

    // lane 0-5 of each warp: P, Y, X of the upper, then of the lower components
    double acc = 0.0;
    for (int tt = t + sub; tt < seg_end; tt += SUB) {
      const int lt = tt - pr->tile_begin;
      const int x0 = (lt % pr->tiles_x) * TILE_W;
      const int y0 = (lt / pr->tiles_x) * TH;
      const int r0 = tg * RPT;                  // this thread's rows of the tile
      const bool full = x0 + TILE_W <= nx && y0 + TH <= ny;
      const bool in_x = x0 + tx < nx;
      const int rows_in = in_x ? ny - (y0 + r0) : 0;              // row k is in the grid if k < rows_in
      const size_t idx0 = (size_t)(y0 + r0) * nx + (x0 + tx);     // row 0 (used where in the grid)
      double q[RPT][4], qp[RPT][4], hq[4];
      int hat = 0;                              // the halo site's place in the tile
      if (full) {
#pragma unroll
        for (int k = 0; k < RPT; ++k) load(idx0 + (size_t)k * nx, q[k], qp[k]);
      } else {
#pragma unroll
        for (int k = 0; k < RPT; ++k) form(x0 + tx, y0 + r0 + k, q[k], qp[k]);
      }
      if (ltid < NH) {
        int hrow, hcol;
        if (ltid < NH_ROW) {                    // rows above / below
          const int r = ltid / TILE_W;
          hrow = (r < R) ? r : TH + r;
          hcol = (ltid % TILE_W) + R;
        } else {                                // columns left / right
          const int h2 = ltid - NH_ROW;
          hrow = h2 / (2 * R) + R;
          const int c = h2 % (2 * R);
          hcol = (c < R) ? c : TILE_W + c;
        }
        hat = hrow * W + hcol;
        double unused[4];
        form(x0 + hcol - R, y0 + hrow - R, hq, unused);
      } else {
        hq[0] = hq[1] = hq[2] = hq[3] = 0.0;
      }
      // the largest numbers of the tile
      unsigned m0 = max(mag(hq[0]), mag(hq[1])), m1 = max(mag(hq[2]), mag(hq[3])), m2 = 0u, m3 = 0u;
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
      if (lane < 4) atomicMax(emax + 4 * par + lane, lane == 0 ? m0 : lane == 1 ? m1 : lane == 2 ? m2 : m3);
      if (q_out) {
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
          if (k < rows_in) {
            vec4 o;
            o.x = q[k][0]; o.y = q[k][1]; o.z = q[k][2]; o.w = q[k][3];
            q_out[idx0 + (size_t)k * nx] = o;
          }
        }
      }
      sub_sync();   // the exponents are complete, and the previous tile has been read
      // exponents of 128 and below (numbers under 2^-894) count as zero
      const int be_u = max((int)(emax[4 * par] >> 21), 128), be_d = max((int)(emax[4 * par + 1] >> 21), 128);
      const int be_pu = max((int)(emax[4 * par + 2] >> 21), 128), be_pd = max((int)(emax[4 * par + 3] >> 21), 128);
      bad = bad || be_u == 0x7ff || be_d == 0x7ff || be_pu == 0x7ff || be_pd == 0x7ff;
      if (ltid < 4) emax[4 * (par ^ 1) + ltid] = 0u;
      par ^= 1;
      const int at0 = (r0 + R) * W + tx + R;    // this thread's first site in the tile
#pragma unroll
      for (int k = 0; k < RPT; ++k) {
        // sites beyond the grid's edge are halo of the sites inside, but not summed
        half_u[at0 + k * W] = make_longlong2(fx::to_fixed<F>(q[k][0], be_u), fx::to_fixed<F>(q[k][1], be_u));
        half_d[at0 + k * W] = make_longlong2(fx::to_fixed<F>(q[k][2], be_d), fx::to_fixed<F>(q[k][3], be_d));
      }
      if (ltid < NH) {
        half_u[hat] = make_longlong2(fx::to_fixed<F>(hq[0], be_u), fx::to_fixed<F>(hq[1], be_u));
        half_d[hat] = make_longlong2(fx::to_fixed<F>(hq[2], be_d), fx::to_fixed<F>(hq[3], be_d));
      }
      {
        // this warp's coefficient table: row scale = the largest term's, the
        // coefficients of a row as 60-bit fractions of it
        const int be_own = ch ? be_d : be_u, be_oth = ch ? be_u : be_d, be_p = ch ? be_pd : be_pu;
        const int be_x = (cj == 0 || cj == 6) ? be_own : (cj == 5 ? be_p : be_oth);
        int sc = my_xe ? my_xe + be_x : 0;
        sc = max(sc, __shfl_xor_sync(0xffffffffu, sc, 1));
        sc = max(sc, __shfl_xor_sync(0xffffffffu, sc, 2));
        sc = max(sc, __shfl_xor_sync(0xffffffffu, sc, 4));
        if (lane < COEF_SLOTS) {
          const fx::Limbs l = fx::split(fx::to_fixed<60>(my_coef, max(sc - be_x, 63)));
          kt[lane] = cj == 7 ? make_int2(sc, 0) : make_int2(l.hi, l.lo);
        }
      }
      sub_sync();   // tile and coefficients are in shared memory

      fx::WarpSum ws[6];
      int we[6];
      auto half = [&](auto half_c) {
        constexpr int HALF = decltype(half_c)::value;
        const longlong2* const own = (HALF ? half_d : half_u) + at0;
        const longlong2* const oth = (HALF ? half_u : half_d) + at0;
        const int2* const kc = kt + 8 * HALF;
        auto coef = [&](int j) { const int2 v = kc[j]; return fx::Limbs{v.x, v.y}; };
        const int sc = kc[7].x;
        const int be_own = HALF ? be_d : be_u, be_p = HALF ? be_pd : be_pu;
        const int se = sc - 2044;                       // the row's scale: |terms| < 2^se
        const int texp = se - F + yexp;                 // unit of y as stored
        const bool live = texp >= -1022;                // else below the normal range: zero
        // columns of the other half: rows r0 - R .. r0 + RPT + R - 1
        longlong2 col[RPT + 2 * R];
#pragma unroll
        for (int j = 0; j < RPT + 2 * R; ++j) col[j] = oth[(j - R) * W];
        long long v[RPT][2];
        unsigned vor = 0u;                              // the upper words of all |v|, or-ed
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
          const longlong2* const row = oth + k * W;
          // differences along x of (re, im), and along y
          const longlong2 xl = row[-1], xr = row[1];
          long long hxr = xl.x - xr.x, hxi = xr.y - xl.y;          // -D_x re, D_x im
          long long hyr = col[k + R + 1].x - col[k + R - 1].x, hyi = col[k + R + 1].y - col[k + R - 1].y;
          if constexpr (R == 2) {
            const longlong2 xl2 = row[-2], xr2 = row[2];
            hxr = 8 * hxr - (xl2.x - xr2.x);
            hxi = 8 * hxi - (xr2.y - xl2.y);
            hyr = 8 * hyr - (col[k + 2 * R].x - col[k].x);
            hyi = 8 * hyi - (col[k + 2 * R].y - col[k].y);
          }
          // upper: (mc^2+V-s-sigma) u + c[-i D_x d - D_y d + (A_x - i A_y) d]
          // lower: (-mc^2+V-s-sigma) d + c[-i D_x u + D_y u + (A_x + i A_y) u]
          const longlong2 cv = own[k * W];
          const fx::Limbs c0 = fx::split(cv.x), c1 = fx::split(cv.y);
          fx::Acc s0, s1;
          {
            const fx::Limbs ka = coef(0);
            s0.mac(c0, ka);
            s1.mac(c1, ka);
          }
          if constexpr (ISO) {
            const fx::Limbs kx = coef(1);
            s0.mac(fx::split(HALF ? hxi + hyr : hxi - hyr), kx);
            s1.mac(fx::split(HALF ? hxr + hyi : hxr - hyi), kx);
          } else {
            const fx::Limbs kx = coef(1), ky = coef(2);
            s0.mac(fx::split(hxi), kx);
            s1.mac(fx::split(hxr), kx);
            s0.mac(fx::split(HALF ? hyr : -hyr), ky);
            s1.mac(fx::split(HALF ? hyi : -hyi), ky);
          }
          if (has_ax) {
            const fx::Limbs kax = coef(3);
            s0.mac(fx::split(col[k + R].x), kax);
            s1.mac(fx::split(col[k + R].y), kax);
          }
          if (has_ay) {
            const fx::Limbs kay = coef(4);
            s0.mac(fx::split(HALF ? -col[k + R].y : col[k + R].y), kay);
            s1.mac(fx::split(HALF ? col[k + R].x : -col[k + R].x), kay);
          }
          if (i >= 2) {
            const fx::Limbs ke = coef(5);
            s0.mac(fx::split(-fx::to_fixed<F>(qp[k][2 * HALF], be_p)), ke);
            s1.mac(fx::split(-fx::to_fixed<F>(qp[k][2 * HALF + 1], be_p)), ke);
          }
          if constexpr (HAS_V) {
            if (Vp) {
              const double pot = k < rows_in ? Vp[idx0 + (size_t)k * nx] : 0.0;
              const fx::Limbs kv = fx::split(fx::to_fixed<60>(pot, max(sc - be_own, 63)));
              s0.mac(c0, kv);
              s1.mac(c1, kv);
            }
          }
          v[k][0] = s0.template value<28>();
          v[k][1] = s1.template value<28>();
          if (!full && k >= rows_in) v[k][0] = v[k][1] = 0;
          vor |= (unsigned)((v[k][0] ^ (v[k][0] >> 63)) >> 32) | (unsigned)((v[k][1] ^ (v[k][1] >> 63)) >> 32);
          if (y_out && k < rows_in) {
            // components of this half (16 of the site's 32 bytes)
            double2* const yo = reinterpret_cast<double2*>(y_out + idx0 + (size_t)k * nx) + HALF;
            *yo = live ? make_double2(fx::to_double(v[k][0], texp), fx::to_double(v[k][1], texp))
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
          const fx::Limbs c0 = fx::split(cv.x << (58 - F)), c1 = fx::split(cv.y << (58 - F));
          const fx::Limbs w0 = fx::split((v[k][0] << sl) >> 2), w1 = fx::split((v[k][1] << sl) >> 2);
          aP.mac(c0, w0);
          aP.mac(c1, w1);
          aY.sqr(w0);
          aY.sqr(w1);
          aX.sqr(c0);
          aX.sqr(c1);
        }
        // |q^| < 2^58 and |w| < 2^60: eight terms of q^ w stay below 2^61 in
        // units of 2^60, of w^2 below 2^63, of q^2 below 2^59
        const int qe = be_own - 1022 - 58, ye = texp + 2 - sl;
        ws[3 * HALF] = fx::warp_sum(aP.template value<28>());
        ws[3 * HALF + 1] = fx::warp_sum(aY.value());
        ws[3 * HALF + 2] = fx::warp_sum(aX.value());
        we[3 * HALF] = qe + ye + 60;
        we[3 * HALF + 1] = 2 * ye + 60;
        we[3 * HALF + 2] = 2 * qe + 60;
      };
      half(std::integral_constant<int, 0>{});
      half(std::integral_constant<int, 1>{});
      // one conversion for all six sums: each by its lane
      fx::WarpSum mine = ws[0];
      int me = we[0];
#pragma unroll
      for (int j = 1; j < 6; ++j) {
        if (lane == j) { mine = ws[j]; me = we[j]; }
      }
      acc += scalbn(fx::to_double(mine), me);
    }
    t = seg_end;
    double accP = acc + __shfl_down_sync(0xffffffffu, acc, 3);
    const double accY = __shfl_sync(0xffffffffu, accP, 1), accX = __shfl_sync(0xffffffffu, accP, 2);
    if (bad) accP = __longlong_as_double(0x7ff8000000000000LL);   // not finite: reported by finish_pass
    if (lane == 0) { red[warp][0] = accP; red[warp][1] = accY; red[warp][2] = accX; }
    pass_sums<true, COOP, NW>(lp, pr, i, seg_tiles, red, &last_flag, coop_slots);
  }
}

// threads of a pass kernel (S = double: all tile workers of the CTA)
template <class S, int TH>
__host__ __device__ constexpr int pass_threads() { return sub_workers<S>() * 32 * (TH / rows_per_thread<S, TH>()); }

// FLAG: kx = ky (S = double); not used by S = float
template <class S, int R, int TH, bool DIRI, bool HAS_V, bool FLAG>
__global__ void __launch_bounds__(pass_threads<S, TH>(), sizeof(S) == sizeof(float) ? min_blocks<TH>() : 1)
lanczos_pass(const __grid_constant__ LaunchParams lp) {
  // programmatic dependent launch: nothing the previous kernel wrote is read
  // before this point
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if constexpr (sizeof(S) == sizeof(float))
    pass_body<R, TH, DIRI, HAS_V>(lp, *lp.step);
  else
    pass_body_fx<R, TH, DIRI, HAS_V, FLAG, false, sub_workers<S>()>(lp, nullptr, nullptr, *lp.step);
  // the next kernel may be scheduled now (it waits for our completion)
  asm volatile("griddepcontrol.launch_dependents;");
}

// psi <- C_1 psi + sum_{j >= 2} C_j q^_j at site s: the complex64 basis
// terms accumulated in compensated FP32 (coefficients as FP32 pairs, exact
// products, two-sum accumulation), added to the FP64 term C_1 psi at the end.
// Loads of DEPTH basis vectors are issued before their products (more loads
// in flight per thread, against more registers).
template <int DEPTH>
__device__ __forceinline__ void recombine_site_df(vec4* psi, const float4* basis, size_t n, size_t s, int k,
                                                  const double* cr, const double* ci, const float* crh,
                                                  const float* crl, const float* cih, const float* cil) {
  float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f, e0 = 0.f, e1 = 0.f, e2 = 0.f, e3 = 0.f;
  for (int j0 = 2; j0 <= k; j0 += DEPTH) {
    float4 v[DEPTH];
#pragma unroll
    for (int u = 0; u < DEPTH; ++u)
      if (j0 + u <= k) v[u] = __ldcs(basis + (size_t)(j0 + u - 2) * n + s);
#pragma unroll
    for (int u = 0; u < DEPTH; ++u) {
      if (j0 + u <= k) {
        const int j = j0 + u;
        const float ah = crh[j], al = crl[j], bh = cih[j], bl = cil[j];
        // (a + i b)(q.re + i q.im) for the upper (x, y) and lower (z, w) component
        acc_prod(ah, al, v[u].x, s0, e0);
        acc_prod(-bh, -bl, v[u].y, s0, e0);
        acc_prod(ah, al, v[u].y, s1, e1);
        acc_prod(bh, bl, v[u].x, s1, e1);
        acc_prod(ah, al, v[u].z, s2, e2);
        acc_prod(-bh, -bl, v[u].w, s2, e2);
        acc_prod(ah, al, v[u].w, s3, e3);
        acc_prod(bh, bl, v[u].z, s3, e3);
      }
    }
  }
  const vec4 q = psi[s];
  const double ar = cr[1], ai = ci[1];
  vec4 o;
  o.x = fma(ar, q.x, fma(-ai, q.y, (double)s0 + (double)e0));
  o.y = fma(ar, q.y, fma(ai, q.x, (double)s1 + (double)e1));
  o.z = fma(ar, q.z, fma(-ai, q.w, (double)s2 + (double)e2));
  o.w = fma(ar, q.w, fma(ai, q.z, (double)s3 + (double)e3));
  psi[s] = o;
}

// ---------------------------------------------------------------------------
// psi <- sum_j C_j q^_j (Eq. 17), q^_1 = psi, q^_j = basis[j-2] for j >= 2.
// Mixed path: the basis is complex64; C_1 psi is formed in FP64 so that the
// FP32 rounding of the basis only enters the (small) Krylov corrections, and
// those are summed with compensation (recombine_site_df): plain FP32
// accumulation of the corrections was the largest error of the mixed path on
// fast packets.
//
// FP64 path: complex128 fields, the sums in fixed point (dirac_fixed.cuh): in
// FP64 the 16 multiply-adds per site and vector took 1024 cycles of a
// sub-partition against the 190 that reading the vector takes; in limbs they
// take about as long as the read.  Each site has its own scale, that of its
// largest |C_j q^_j| so far (the sums are shifted when a batch of D vectors
// raises it), so the relative error of every site is about 2^-54 of its
// largest term.
// Blocks are dealt to problems in proportion to their size.
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
  int be = 1100;   // exponent sum of the largest term (terms below 2^-938 count as zero)
  for (int j0 = 1; j0 <= k; j0 += D) {
    vec4 v[D];
#pragma unroll
    for (int u = 0; u < D; ++u) {
      const int j = j0 + u;
      if (j <= k) v[u] = j == 1 ? psi[s] : basis[(size_t)(j - 2) * n + s];
    }
    int nb = be;
#pragma unroll
    for (int u = 0; u < D; ++u) {
      if (j0 + u <= k) {
        const unsigned a = max((unsigned)__double2hiint(v[u].x) << 1, (unsigned)__double2hiint(v[u].y) << 1);
        const unsigned b = max((unsigned)__double2hiint(v[u].z) << 1, (unsigned)__double2hiint(v[u].w) << 1);
        nb = max(nb, (int)(max(a, b) >> 21) + coef[j0 + u].be);
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) sum[c] = fx::shr_round(sum[c], nb - be);
    be = nb;
#pragma unroll
    for (int g = 0; g < D; g += 4) {
      fx::Acc acc[4];
#pragma unroll
      for (int u = g; u < g + 4; ++u) {
        if (j0 + u <= k) {
          const FxCoef cf = coef[j0 + u];
          const int bq = max(be - cf.be, 63);
          const fx::Limbs x = fx::split(fx::to_fixed<59>(v[u].x, bq)), y = fx::split(fx::to_fixed<59>(v[u].y, bq));
          const fx::Limbs z = fx::split(fx::to_fixed<59>(v[u].z, bq)), w = fx::split(fx::to_fixed<59>(v[u].w, bq));
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
  const int e = be - 2044 - 56;   // 2^62 of the products' 2^-118
  vec4 o;
  o.x = fx::to_double(sum[0], e);
  o.y = fx::to_double(sum[1], e);
  o.z = fx::to_double(sum[2], e);
  o.w = fx::to_double(sum[3], e);
  psi[s] = o;
}

// Three CTAs per SM (at most 85 registers), so that enough warps keep loads
// in flight: the compensated sums make the mixed form arithmetic-heavy.
template <bool MIXED>
__global__ void __launch_bounds__(256, 3) recombine(const __grid_constant__ RecombParams rp) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __shared__ double cr[MIXED ? KMAX + 2 : 1], ci[MIXED ? KMAX + 2 : 1];
  __shared__ float fr[MIXED ? KMAX + 2 : 1], fi[MIXED ? KMAX + 2 : 1];
  __shared__ float frl[MIXED ? KMAX + 2 : 1], fil[MIXED ? KMAX + 2 : 1];
  __shared__ FxCoef fc[MIXED ? 1 : KMAX + 2];
  __shared__ int k_s, err_s;
  const int b = rp.blk_prob[blockIdx.x];
  const Problem* pr = rp.probs + b;
  DevState* st = pr->st;
  if (threadIdx.x == 0) { k_s = st->k_used; err_s = st->error; }
  if (threadIdx.x <= KMAX) {
    const double a = st->coef_re[threadIdx.x], c = st->coef_im[threadIdx.x];
    if constexpr (MIXED) {
      cr[threadIdx.x] = a;
      ci[threadIdx.x] = c;
      fr[threadIdx.x] = (float)a;
      fi[threadIdx.x] = (float)c;
      frl[threadIdx.x] = (float)(a - (double)fr[threadIdx.x]);
      fil[threadIdx.x] = (float)(c - (double)fi[threadIdx.x]);
    } else {
      fc[threadIdx.x] = fx_coef(a, c);
    }
  }
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
  const long long n = (long long)pr->nx * pr->ny;
  const long long stride = (long long)pr->rblk_count * blockDim.x;
  vec4* psi = const_cast<vec4*>(pr->psi);
  for (long long s = (long long)lb * blockDim.x + threadIdx.x; s < n; s += stride) {
    if constexpr (MIXED)
      recombine_site_df<8>(psi, static_cast<const float4*>(pr->basis), (size_t)n, (size_t)s, k, cr, ci, fr, frl,
                           fi, fil);
    else
      recombine_site_fx<4>(psi, static_cast<const vec4*>(pr->basis), (size_t)n, (size_t)s, k, fc);
  }
  asm volatile("griddepcontrol.launch_dependents;");
}

// ---------------------------------------------------------------------------
// One time step of one problem in one cooperative launch (every CTA
// resident): the passes separated by grid-wide barriers instead of kernel
// boundaries, then the recombination.  After each pass every CTA sums all
// CTA partials in the same fixed order and runs the scalar update on its own
// shared-memory copy of the state, so that all copies stay identical
// (bitwise: same inputs, same operations) and no second barrier is needed.
// Partials are double-buffered by pass parity: a CTA can run at most one
// pass ahead of the slowest one, which is still reading the other buffer.
// ---------------------------------------------------------------------------
constexpr int ERR_BARRIER = 8;                    // a grid barrier timed out
constexpr unsigned GRID_SYNC_SPIN_MAX = 1u << 20; // polls (~100 ns nap + an L2 round trip each: about a second)
constexpr int GRID_SYNC_WORDS = 4;                // arrivals, generation, timeout flag, spare

struct CoopArgs {
  double* slots;   // 2 x 3 x cap doubles: CTA partials (P, Y, X) by pass parity
  unsigned* bar;   // GRID_SYNC_WORDS words, zeroed before each launch
  int G;           // CTAs of the launch
  int cap;         // CTAs the slot buffer holds
  int bar_count;   // CTAs each grid barrier waits for: G (G + 1 only in the timeout test)
};

// Barrier of all CTAs of a cooperative launch.  Thread 0 of each CTA arrives
// (release of the CTA's writes, ordered by the __syncthreads before it) and
// waits for the generation to advance (acquire).  False after a timeout
// (bar[2] set), after which every waiting CTA gives up as well.  One counter
// and one polled word serve the one-CTA-per-SM launches of the FP64 path
// well; with many CTAs per SM their contention outweighs what the launch
// boundaries cost, which is why the FP32 path keeps per-pass launches.
__device__ __forceinline__ bool grid_sync(unsigned* bar, unsigned G) {
  __shared__ int ok_s;
  __syncthreads();
  if (threadIdx.x == 0) {
    cuda::atomic_ref<unsigned, cuda::thread_scope_device> arrived(bar[0]), gen(bar[1]), timeout(bar[2]);
    const unsigned g0 = gen.load(cuda::memory_order_acquire);
    int ok = 1;
    __threadfence();
    if (arrived.fetch_add(1u, cuda::memory_order_acq_rel) == G - 1u) {
      arrived.store(0u, cuda::memory_order_relaxed);
      gen.store(g0 + 1u, cuda::memory_order_release);
    } else {
      unsigned spins = 0;
      while (gen.load(cuda::memory_order_acquire) == g0) {
        if (timeout.load(cuda::memory_order_relaxed) != 0u || ++spins > GRID_SYNC_SPIN_MAX) {
          timeout.store(1u, cuda::memory_order_relaxed);
          ok = 0;
          break;
        }
        __nanosleep(100);
      }
    }
    __threadfence();
    ok_s = ok;
  }
  __syncthreads();
  return ok_s != 0;
}

template <int R, int TH, bool DIRI, bool HAS_V, bool ISO>
__global__ void __launch_bounds__(pass_threads<double, TH>(), 1)
lanczos_step(const __grid_constant__ LaunchParams lp, const __grid_constant__ CoopArgs ca) {
  constexpr int SUB = sub_workers<double>();
  constexpr int NT = pass_threads<double, TH>();
  __shared__ DevState sst;
  __shared__ FxCoef fc_s[KMAX + 2];
  const Problem* pr = lp.probs;
  DevState* gst = lp.states;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
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
    double* slots = ca.slots + (iter & 1) * 3 * ca.G;
    pass_body_fx<R, TH, DIRI, HAS_V, ISO, true, SUB>(lp, &sst, slots, step);
    ++iter;
    if (!grid_sync(ca.bar, (unsigned)ca.bar_count)) {
      if (threadIdx.x == 0) { gst->error = ERR_BARRIER; gst->stopped = 1; }
      return;   // psi untouched; the host reports the timeout
    }
    if (warp == 0) {   // the grid totals, in the same order in every CTA
      constexpr int SB = 4;   // loads in flight per lane
      double t0 = 0.0, t1 = 0.0, t2 = 0.0;
      for (int c0 = lane; c0 < ca.G; c0 += SB * 32) {
        double v[SB][3];
#pragma unroll
        for (int k = 0; k < SB; ++k) {
          const int c = c0 + k * 32;
          const double* ps = slots + 3 * (c < ca.G ? c : 0);
          v[k][0] = c < ca.G ? __ldcg(ps) : 0.0;
          v[k][1] = c < ca.G ? __ldcg(ps + 1) : 0.0;
          v[k][2] = c < ca.G ? __ldcg(ps + 2) : 0.0;
        }
#pragma unroll
        for (int k = 0; k < SB; ++k) { t0 += v[k][0]; t1 += v[k][1]; t2 += v[k][2]; }
      }
      t0 = warp_sum(t0);
      t1 = warp_sum(t1);
      t2 = warp_sum(t2);
      finish_pass<true>(lp, pr, &sst, i, t0, t1, t2);
    }
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
          recombine_site_fx<8>(psi, static_cast<const vec4*>(pr->basis), n, (size_t)y * pr->nx + x, k, fc_s);
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

// ---------------------------------------------------------------------------
// test hook: exp(-i T dt) e_1 for a given T with the device routine
// ---------------------------------------------------------------------------
static __global__ void debug_tridiag_expm(const __grid_constant__ ChebParams cp, int k, const double* alpha1,
                                   const double* beta1, double* out_re, double* out_im) {
  double vr, vi;
  const int lane = threadIdx.x & 31;
  const double a = lane < k ? alpha1[lane + 1] : 0.0;
  const double bl = (lane >= 1 && lane < k) ? beta1[lane] : 0.0;
  const double bh = (lane + 1 < k) ? beta1[lane + 1] : 0.0;
  cheb_expm_e1(cp, k, a, bl, bh, vr, vi);
  if (lane < k) { out_re[lane] = vr; out_im[lane] = vi; }
}

}  // namespace dirac
