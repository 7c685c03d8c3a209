// Fused ICRS magnification kernel (one CUDA thread block per light-curve
// epoch, persistent over a contiguous chunk of epochs) and the C ABI of
// include/icrs.h.
//
// Method: Miyazaki & Kawahara, arXiv:2510.02639.  Per epoch:
//   1. source-limb points w_k = w_c + rho e^{2 pi i k/N_limb}      (Sec. 3.2)
//   2. all roots of the lens polynomial at each limb point by Ehrlich-Aberth
//      iteration, validated against the lens equation     (Secs. 2.1, 3.1)
//   3. image-limb points binned in theta and r into image-centred polar
//      sectors                                                    (Sec. 3.2)
//   4. a fixed N_r x N_theta polar grid per sector, every ray mapped through
//      the lens equation, inclusion flags, cubic boundary crossings and the
//      uniform / limb-darkened per-point rule, radial sum, 1/rho^2
//                                                 (Sec. 3.3, Appendix A)
//
// Precision design (GB300: FP64 issues at ~1/64 of the FP32 rate):
//   * roots are found in FP32 on the polynomial written about the lightest
//     lens, warm-started from the previous epoch of the same light curve;
//   * every discrete decision (is a root an image, which bin holds a point,
//     which point is a sector's extreme, is a ray inside the source, which
//     branch of f(delta)) is taken in FP32 only when the FP32 error bound
//     cannot change it; otherwise the point or ray is recomputed in FP64, so
//     the decisions equal those of an FP64 evaluation of the same method;
//   * rays are mapped in FP32 in a difference form about FP64 anchors placed
//     on the sector, so the FP32 error stays relative to the source size.
#include <type_traits>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include "icrs.h"
#include "icrs_common.cuh"
#include "icrs_df64.cuh"
#include "icrs_sectors.cuh"
#include "icrs_ps.cuh"
#include "icrs_rays.cuh"
#include "icrs_rays_der.cuh"

namespace icrs {

// Threads per block (one block per SM): 512, 128 registers each.  The ray
// stage is bound by the FP32 pipes and the dependency latency of its chains:
// registers for independent column pairs pay more than further warps.
constexpr int NT_BASE = 512;
constexpr int NW_MAX = NT_BASE / 32;  // warps per block
static_assert(TASK_WARPS == NW_MAX, "the ray stage's chunks are cut for this many warps");
constexpr int QMAX = 2048;       // work queue
constexpr int PMAX_MIN = 512;    // FP64-polished image-limb points per epoch (at least)
constexpr int MAXT = 32;         // theta runs (more: ICRS_ST_OVERFLOW)
constexpr int MAXRB = 32;        // r bins per theta run
constexpr int MAXCELL = 96;      // (theta run, r run) cells
constexpr int MAXBOX = 96;       // candidate sectors before merging
constexpr int MAXCELL_D = 32;    // cells with tracked derivatives
constexpr int MAXBOX_D = 32;     // candidate sectors with tracked derivatives
constexpr float TINY_EXTENT = 3e-4f;  // images smaller than this x rho skip FP64 decisions
// A refined FP32 image whose error bound exceeds EE_SUSPECT max(1, r), or two
// images of one limb point closer than DUP_TOL max(1, r), send the limb point
// to the FP64 re-solve.
constexpr float EE_SUSPECT = 1e-6f;
constexpr float DUP_TOL = 1e-6f;
// Two roots of a limb point that are not images, closer than PAIR_TOL
// max(1, |z|), send it to the FP64 re-solve as well (binary lens; the
// point-source solver's tolerance).
constexpr float PAIR_TOL = (float)PS_PAIR_TOL;

// Meta bits of an image-limb slot.
constexpr uint8_t M_VALID = 1, M_EXACT = 2, M_UNSURE = 4, M_CAND = 8, M_CANDT = 16;

struct Shared {
  // ---- per parameter set
  Lens L;
  double rho, u1, u2;
  double pa[4];        // a1..a4, the power series in mu^(1/2)
  float I0, c0f, c1f, c2f;  // brightness coefficients of the set's law (see the set-up)
  float c1h, c3h;      // their half-integer-power brightness coefficients (ray stage)
  int half;            // c1h or c3h nonzero
  // spot: centre (rho units), radius^2 and contrast; 1 / (1 - c F_spot) and
  // its u1 derivative over itself times c F_spot' ... (see the chain);
  // spot_new: the set changed and has a spot; generic: half or spot
  double spot_x, spot_y, spot_r, spot_c, spot_norm, spot_gu, spot_acc[2];
  float spot_rr32, spot_f32;  // its radius, and 1 - contrast
  int spot, spot_bad, spot_new, generic;
  float eps32[3];
  cf aj32[3][3];       // [frame j][lens i]: a_i - a_j (FP32)
  cf D32[3][4], E32[3][3];  // polynomial parts in frame j (FP32)
  cd D64[3][4], E64[3][3];  // the same in FP64
  df adf[3][3][2];     // [frame j][lens i][x/y]: a_i - a_j (double-float)
  df adf_ll[2];        // a_ll (original frame, double-float)
  df epsdf[3];
  df rhodf;
  int cur_set;
  int l2;              // second lightest lens (triple) or -1
  cf anc[32][10];      // roots of the cold-start anchor limb points
  // ---- per epoch
  cd wc;
  cf wcj32[3];         // w_c - a_j (FP32)
  df wcdf[3][2];       // w_c - a_j (double-float)
  uint32_t status;
  int warm;            // roots[] hold the previous epoch of this set
  int qn, pn;
  double ht;           // width of a theta bin
  float htf;
  unsigned int tocc[4];         // occupied theta bins (up to 128)
  int nT, full;
  signed char runT[128];
  int startT[MAXT];
  unsigned int t_rlo_u[MAXT], t_rhi_l[MAXT];
  unsigned long long t_rlo[MAXT], t_rhi[MAXT];
  unsigned int t_s[MAXT][2];                // FP32 keys of the refined radius: rmin_hi, rmax_lo
  double rlo[MAXT], hr[MAXT];
  float rlh[MAXT], rll[MAXT], ihr[MAXT];  // rlo as a float pair, 1 / hr
  int rsmall[MAXT];    // 1: hr > 0 but the run is below TINY_EXTENT rho; 2: hr = 0
  unsigned int rocc[MAXT];
  unsigned int tmask[MAXT][MAXRB][4];  // theta bins of each (run, r bin)
  signed char rrun[MAXT][MAXRB];
  int cellbase[MAXT + 1];
  int ncell;
  int origin_in;
  int c_cnt[MAXCELL];
  unsigned int c_u[MAXCELL][4];             // FP32 keys: rmin_hi, rmax_lo, tmin_hi, tmax_lo
  unsigned int c_s[MAXCELL][4];             // FP32 keys of the refined radius and angle: rmin_hi, rmax_lo, tmin_hi, tmax_lo
  float2 c_ref[MAXCELL][2];                 // direction of the FP32 angle extremes
  unsigned long long c_x[MAXCELL][4];       // FP64 keys: rmin, rmax, tmin, tmax
  int nbox;
  Box box[MAXBOX];
  int probe_hit;
  int cnt[16];         // diagnostics: FP64 polishes, FP64 validations, FP64 rays, FP64 crossings, phase clocks
  long long clk0;
  // ---- ray stage (current sector)
  double red[NW_MAX];
};

// Derivative-mode state (binary lens), in the dynamic shared memory of that
// instantiation only.
struct DerShared {
  int cell_arg[MAXCELL_D][4];  // slot of the point that sets each cell extreme
  double Gb[MAXBOX_D][4];   // dS / d(r_lo, r_hi, th_lo, width) of each sector
  double H[8];              // dS / d(w_c.x, w_c.y, rho, u1, a1.x, a2.x, eps1, eps2)
  cd dwc[4];                // d w_c / d(t0, tE, u0, alpha)
  double dadp[2][2];        // d a_j.x / d(s, q)
  double depsq[2];          // d eps_j / d q
  DualD cx[MAXCELL_D * 4];  // cell extremes with tangents
  BoxT<DualD> box[MAXBOX_D];  // sectors with tangents
};

// Order-preserving integer keys for signed FP32 / FP64 values.
__device__ __forceinline__ unsigned int fkey(float v) {
  unsigned int u = __float_as_uint(v);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float fkey_inv(unsigned int k) {
  unsigned int u = (k & 0x80000000u) ? (k & 0x7fffffffu) : ~k;
  return __uint_as_float(u);
}
__device__ __forceinline__ unsigned long long dkey(double v) {
  unsigned long long u = (unsigned long long)__double_as_longlong(v);
  return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}
__device__ __forceinline__ double dkey_inv(unsigned long long k) {
  unsigned long long u = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
  return __longlong_as_double((long long)u);
}


// ---------------------------------------------------------------- FP64 paths
// Limb point k in FP64 (Sec. 3.2).
__device__ inline cd limb_point64(const Shared& sh, int k, int n_limb) {
  double s, c;
  sincospi(2.0 * (double)k / (double)n_limb, &s, &c);
  return mk(sh.wc.x + sh.rho * c, sh.wc.y + sh.rho * s);
}

// Index of the lens nearest to z (original frame).
template <int NL>
__device__ inline int nearest_lens64(const Lens& L, cd z) {
  int j = 0;
  double best = abs2(z - L.a[0]);
  for (int i = 1; i < NL; ++i) {
    double d = abs2(z - L.a[i]);
    if (d < best) { best = d; j = i; }
  }
  return j;
}

// FP64 polish of an image-limb root by Newton's method on the lens equation
// in the frame of its nearest lens; returns (r, theta) of the image.
template <int NL>
__device__ inline void polish_image64(const Shared& sh, cd z0, cd w, double* r, double* th) {
  int j = nearest_lens64<NL>(sh.L, z0);
  double eps[NL];
  cd a[NL];
  for (int i = 0; i < NL; ++i) { eps[i] = sh.L.eps[i]; a[i] = sh.L.a[i] - sh.L.a[j]; }
  cd x = z0 - sh.L.a[j];
  cd wj = w - sh.L.a[j];
  for (int it = 0; it < 4; ++it) {
    cd st = lens_newton_step<NL, double>(eps, a, x, wj);
    x = x + st;
    if (abs2(st) <= 1e-32 * fmax(1e-20, abs2(x))) break;
  }
  cd z = x + sh.L.a[j];
  *r = sqrt(z.x * z.x + z.y * z.y);
  *th = atan2(z.y, z.x);
}

// FP64 validation of an ambiguous root: Newton's method on the polynomial
// written about the root's nearest lens, then the lens-equation residual in
// that frame against img_tol.  Returns 1 (image) or 0; (r, theta) if image.
// *conv (if given) is cleared when the Newton steps had not converged: next to
// a near-double root Newton converges only linearly, and an iterate still
// ~1e-4 from the root can pass the residual test there (the lens map is flat
// across the critical curve).
template <int NL>
__device__ inline int validate_root64(const Shared& sh, cd z0, cd w, double img_tol, double* r, double* th,
                                      int* conv = nullptr) {
  constexpr int N = NL * NL + 1;
  int j = nearest_lens64<NL>(sh.L, z0);
  double eps[NL];
  cd a[NL];
  for (int i = 0; i < NL; ++i) { eps[i] = sh.L.eps[i]; a[i] = sh.L.a[i] - sh.L.a[j]; }
  cd b[N + 1];
  cd wj = w - sh.L.a[j];
  lens_poly<NL, double>(eps, a, sh.D64[j], sh.E64[j], wj, b);
  cd x = z0 - sh.L.a[j];
  bool done = false;
  for (int it = 0; it < 8; ++it) {
    cd p, dp;
    horner2<N, double>(b, x, p, dp);
    if (!(abs2(dp) > 0.0)) break;
    cd st = dv(p, dp);
    x = x - st;
    if (abs2(st) <= 1e-30 * fmax(1.0, abs2(x))) { done = true; break; }
  }
  if (conv) *conv = done ? 1 : 0;
  cd F = lens_map<NL, double>(eps, a, x) - wj;
  double res = sqrt(abs2(F));
  if (!(res <= img_tol)) return 0;
  cd z = x + sh.L.a[j];
  *r = sqrt(z.x * z.x + z.y * z.y);
  *th = atan2(z.y, z.x);
  return 1;
}

// Sine of the angle from direction X to the angle th, in FP64 (out of line: a
// rare fallback).
__device__ __noinline__ float sine_from64(float2 X, double th) {
  double s, c;
  sincos(th, &s, &c);
  return (float)((double)X.x * s - (double)X.y * c);
}

// Tangents of an image-limb point z = r e^{i th} (the image of the source-limb
// point w_c + rho u) with respect to (t0, tE, u0, alpha, s, q, rho, u1), binary
// lens: the implicit derivative of the lens equation F(z; p) = f(z; p) - w(p)
// = 0, dz = -J^{-1} dF/dp at fixed z, J the real 2x2 Jacobian of f (the root
// derivative of Sec. 3.5, written for the lens equation rather than the
// polynomial so that it holds in any frame).  Returns d r / dp and d th / dp.
__device__ inline void point_tangents(const Shared& sh, const DerShared& ds, double r, double th, cd u, double* dr,
                                      double* dth) {
  double sn, cs;
  sincos(th, &sn, &cs);
  const cd z = mk(r * cs, r * sn);
  cd gm = mk(0.0, 0.0), cA[2], cE[2];
  for (int j = 0; j < 2; ++j) {
    cd iv = inv(z - sh.L.a[j]);
    cd iv2 = iv * iv;
    gm = gm + scl(iv2, sh.L.eps[j]);
    cA[j] = scl(cj(iv2), -sh.L.eps[j]);  // df/da_j.x = -eps_j / conj(z - a_j)^2
    cE[j] = scl(cj(iv), -1.0);           // df/deps_j = -1 / conj(z - a_j)
  }
  // df = dz + conj(gamma) conj(dz):  J = [[1 + g.x, -g.y], [-g.y, 1 - g.x]]
  const double j11 = 1.0 + gm.x, j12 = -gm.y, j22 = 1.0 - gm.x;
  const double det = j11 * j22 - j12 * j12;
  for (int q = 0; q < NPAR; ++q) {
    cd dF = mk(0.0, 0.0);
    if (q < 4) dF = scl(ds.dwc[q], -1.0);
    else if (q == 4) dF = scl(cA[0], ds.dadp[0][0]) + scl(cA[1], ds.dadp[1][0]);
    else if (q == 5) dF = scl(cA[0], ds.dadp[0][1]) + scl(cA[1], ds.dadp[1][1]) + scl(cE[0], ds.depsq[0]) + scl(cE[1], ds.depsq[1]);
    else if (q == 6) dF = scl(u, -1.0);
    double dx = -(j22 * dF.x - j12 * dF.y) / det;
    double dy = -(-j12 * dF.x + j11 * dF.y) / det;
    dr[q] = (z.x * dx + z.y * dy) / r;
    dth[q] = (z.x * dy - z.y * dx) / (r * r);
  }
}

// FP64 Ehrlich-Aberth by one warp, root j of limb point g on lane g N + j (np
// points): the same iteration, operation by operation, as one thread's over
// all roots.  With one point the differences 1 / (z_k - z_j) are spread over
// the lanes besides.  b: this lane's point's polynomial.  Returns whether this
// lane's point converged.
template <int N>
__device__ inline bool ehrlich_aberth_f64_warp(const cd* b, cd* zj, int np, int max_iter) {
  constexpr int NP2 = N * (N - 1), R = (NP2 + 31) / 32;
  const int lane = threadIdx.x & 31;
  const bool act = lane < np * N;
  const int g = act ? lane / N : 0, k = act ? lane - g * N : 0;
  const unsigned mine = ((1u << N) - 1u) << (g * N);  // the lanes of this point
  // |b_l| of the lane's point: lane k of the point forms |b_k|, all form |b_N|
  double ab[N + 1];
  {
    cd bk = b[0];
#pragma unroll
    for (int l = 1; l < N; ++l) if (k == l) bk = b[l];
    const double m = sqrt(abs2(bk));
#pragma unroll
    for (int l = 0; l < N; ++l) ab[l] = __shfl_sync(0xffffffffu, m, g * N + l);
    ab[N] = sqrt(abs2(b[N]));
  }
  cd z = *zj;
  bool done = false;
#pragma unroll 1
  for (int it = 0; it < max_iter; ++it) {
    cd S = mk(0.0, 0.0);
    if (np == 1) {
      cd iv[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int t = min(lane + 32 * r, NP2 - 1), kk = t / (N - 1), jj = t % (N - 1), j = jj + (jj >= kk ? 1 : 0);
        const cd a = mk(__shfl_sync(0xffffffffu, z.x, kk), __shfl_sync(0xffffffffu, z.y, kk));
        const cd c = mk(__shfl_sync(0xffffffffu, z.x, j), __shfl_sync(0xffffffffu, z.y, j));
        iv[r] = inv(a - c);
      }
#pragma unroll
      for (int jj = 0; jj < N - 1; ++jj) {  // j = 0 .. N - 1 without k, in order
        const int t = k * (N - 1) + jj;
        cd v = mk(0.0, 0.0);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const cd u = mk(__shfl_sync(0xffffffffu, iv[r].x, t & 31), __shfl_sync(0xffffffffu, iv[r].y, t & 31));
          if ((t >> 5) == r) v = u;
        }
        S = S + v;
      }
    } else {
#pragma unroll 1
      for (int jj = 0; jj < N - 1; ++jj) {
        const int j = g * N + jj + (jj >= k ? 1 : 0);
        const cd c = mk(__shfl_sync(0xffffffffu, z.x, j), __shfl_sync(0xffffffffu, z.y, j));
        S = S + inv(z - c);
      }
    }
    cd p, dp;
    horner2<N, double>(b, z, p, dp);
    const cd W = dv(p, dp);
    cd dz = dv(W, mk(1.0, 0.0) - W * S);
    if (!(abs2(p) > 0.0)) dz = mk(0.0, 0.0);
    const bool rnd = ea64_at_rounding<N>(ab, z, dz, dp);
    if (!done) z = z - dz;
    const bool conv = rnd || ea64_small(z, dz);
    const unsigned cb = __ballot_sync(0xffffffffu, conv);  // (every lane votes, done or not)
    done = done || (cb & mine) == mine;
    if (__all_sync(0xffffffffu, done)) break;
  }
  *zj = z;
  return done;
}

// FP64 re-solve of the limb points queue[0 .. np - 1] (all roots, FP64
// Ehrlich-Aberth warm-started from the FP32 roots in the lightest lens's
// frame, FP64 validation of each root) by one warp, one root per lane;
// rewrites the points' slots and flags an illegal image count.  It runs only
// for limb points with an untrustworthy FP32 image set, but with a thread for
// each a single one held its block for 400k cycles (an FP64 division takes 570,
// an iteration 35 of them).
template <int NL>
__device__ __noinline__ void resolve_limb_points64(Shared& sh, const int* queue, int np, int K, int max_iter,
                                                   double img_tol, int PMAX, cf* phi, float* r32, float* rl32, float* t32,
                                                   float* e32, short* pidx, uint8_t* meta, double* pr, double* pt) {
  constexpr int N = NL * NL + 1;
  const int lane = threadIdx.x & 31;
  const bool act = lane < np * N;
  const int g = act ? lane / N : 0, jr = act ? lane - g * N : 0;
  const int k = queue[g];
  const int ll = sh.L.ll;
  const cd w = limb_point64(sh, k, K);
  cd b[N + 1], zj;
  {
    double eps[NL];
    cd a[NL], z[N];
    for (int i2 = 0; i2 < NL; ++i2) { eps[i2] = sh.L.eps[i2]; a[i2] = sh.L.a[i2] - sh.L.a[ll]; }
    lens_poly<NL, double>(eps, a, sh.D64[ll], sh.E64[ll], w - sh.L.a[ll], b);
    for (int j = 0; j < N; ++j) z[j] = tod(phi[k * N + j]);
    // separate coincident starts
    for (int j = 1; j < N; ++j)
      for (int i2 = 0; i2 < j; ++i2)
        if (abs2(z[j] - z[i2]) < 1e-20) z[j] = z[j] + mk(1e-7 * (j + 1), 1e-7 * j);
    zj = z[0];
#pragma unroll
    for (int j = 1; j < N; ++j) if (jr == j) zj = z[j];
  }
  __syncwarp();
  if (!ehrlich_aberth_f64_warp<N>(b, &zj, np, max_iter) && act) atomicOr(&sh.status, ICRS_ST_NONCONV);
  bool img = false;
  if (act) {
    const int ps = k * N + jr;
    phi[ps] = tof(zj);
    pidx[ps] = -1;
    uint8_t mm = 0;
    double r, th;
    if (validate_root64<NL>(sh, zj + sh.L.a[ll], w, img_tol, &r, &th)) {
      img = true;
      const int pi = atomicAdd(&sh.pn, 1);
      const float rh = (float)r;
      r32[ps] = rh; rl32[ps] = (float)(r - (double)rh); t32[ps] = (float)th;
      if (pi < PMAX) { pr[pi] = r; pt[pi] = th; pidx[ps] = (short)pi; e32[ps] = 0.f; mm = M_VALID | M_EXACT; }
      else { e32[ps] = 1e-12f; mm = M_VALID; atomicOr(&sh.status, ICRS_ST_OVERFLOW); }
    }
    meta[ps] = mm;
  }
  const int m = __popc(__ballot_sync(0xffffffffu, img) & (((1u << N) - 1u) << (g * N)));
  const bool legal = (NL == 2) ? (m == 3 || m == 5) : (m == 4 || m == 6 || m == 8 || m == 10);
  if (act && !legal) atomicOr(&sh.status, ICRS_ST_IMGCOUNT);
}

// The same for one limb point by one thread, for queues that fill the warps:
// the FP64 pipe then bounds either form, and this one forms a point's
// polynomial once.  Returns the image count.
template <int NL>
__device__ __noinline__ int resolve_limb_point64(Shared& sh, int k, int K, int max_iter, double img_tol, int PMAX,
                                                 cf* phi, float* r32, float* rl32, float* t32, float* e32, short* pidx,
                                                 uint8_t* meta, double* pr, double* pt) {
  constexpr int N = NL * NL + 1;
  const int ll = sh.L.ll;
  const cd w = limb_point64(sh, k, K);
  double eps[NL];
  cd a[NL], b[N + 1], z[N];
  for (int i2 = 0; i2 < NL; ++i2) { eps[i2] = sh.L.eps[i2]; a[i2] = sh.L.a[i2] - sh.L.a[ll]; }
  lens_poly<NL, double>(eps, a, sh.D64[ll], sh.E64[ll], w - sh.L.a[ll], b);
  for (int j = 0; j < N; ++j) z[j] = tod(phi[k * N + j]);
  // separate coincident starts
  for (int j = 1; j < N; ++j)
    for (int i2 = 0; i2 < j; ++i2)
      if (abs2(z[j] - z[i2]) < 1e-20) z[j] = z[j] + mk(1e-7 * (j + 1), 1e-7 * j);
  if (ehrlich_aberth_f64<N>(b, z, max_iter) < 0) atomicOr(&sh.status, ICRS_ST_NONCONV);
  int m = 0;
#pragma unroll 1
  for (int j = 0; j < N; ++j) {
    const int ps = k * N + j;
    phi[ps] = tof(z[j]);
    pidx[ps] = -1;
    uint8_t mm = 0;
    double r, th;
    if (validate_root64<NL>(sh, z[j] + sh.L.a[ll], w, img_tol, &r, &th)) {
      const int pi = atomicAdd(&sh.pn, 1);
      const float rh = (float)r;
      r32[ps] = rh; rl32[ps] = (float)(r - (double)rh); t32[ps] = (float)th;
      if (pi < PMAX) { pr[pi] = r; pt[pi] = th; pidx[ps] = (short)pi; e32[ps] = 0.f; mm = M_VALID | M_EXACT; }
      else { e32[ps] = 1e-12f; mm = M_VALID; atomicOr(&sh.status, ICRS_ST_OVERFLOW); }
      ++m;
    }
    meta[ps] = mm;
  }
  return m;
}

// ---------------------------------------------------------------- queue
__device__ __forceinline__ void q_push(Shared& sh, int* queue, int v) {
  int i = atomicAdd(&sh.qn, 1);
  if (i < QMAX) queue[i] = v;
  else atomicOr(&sh.status, ICRS_ST_OVERFLOW);
}

// ---------------------------------------------------------------- kernel
// A set whose law has half-integer powers of mu (a1 or a3, on a limb-darkened
// grid) or a spot: the binary forward launch gives these sets to the kernel's
// generic instantiation and all others to the linear one, which carries none
// of their code.
__device__ inline bool generic_law(const icrs_params& p, const icrs_grid& g) {
  return p.spot_c != 0.0 || (!g.uniform && (p.a1 != 0.0 || p.a3 != 0.0));
}

// LAW = 0: only the sets without a generic law (their code compiled out);
// LAW = 1: only the sets with one; LAW = 2: every set, the law decided at run
// time.
// DER = true: also the derivative of A with respect to (t0, tE, u0, alpha, s,
// q, rho, u1) (binary lens): reverse mode over the rays (adjoint seeds per
// ray, then each seeded ray's gradient), forward mode (8 tangents) over the
// sector bounds via the implicit derivative of the extremal image points.
struct DerOut {
  const double* gA;    // [S][E] upstream dL/dA, or NULL
  const double* yobs;  // [S][E] data for chi^2 (with sig), or NULL
  const double* sig;   // [S][E]
  double* dA;          // [S][E][8] or NULL
  double* grad;        // [S][8] accumulated, or NULL
  double* chi2;        // [S] accumulated, or NULL
};

template <int NL, bool DER, int NTB, int LAW>
__global__ void __launch_bounds__(NTB, 1)
mag_kernel(const icrs_params* __restrict__ P, int S, const double* __restrict__ T_, int E,
           icrs_grid g, int tiles_per_block, double* __restrict__ A_out, uint32_t* __restrict__ st_out,
           double* __restrict__ diag_sect, int32_t* __restrict__ diag_cnt, float* __restrict__ diag_pts, int PMAX,
           int has_plo, int tabcap, int ccap, int tcap, DerOut dout, const int32_t* __restrict__ items, int n_items) {
  constexpr int N = NL * NL + 1;
  constexpr int NT = NTB;
  constexpr int NW = NT / 32;
  static_assert(NT % 32 == 0 && NW <= NW_MAX && (!DER || NW == NW_MAX), "per-warp tables are sized for these block sizes");
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ Shared sh;
  __shared__ RayShared rays_sh;
  __shared__ typename std::conditional<DER, DerRays, char>::type der_sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int K = g.n_limb, NP = K * N;
  const int BT = g.n_bins_theta, BR = g.n_bins_r;
  // dynamic shared memory carve-up
  unsigned char* p = dyn;
  // per image-limb slot: root / refined image position in the lightest
  // lens's frame (also the next epoch's warm start), FP32 (r, theta), FP32
  // error bound, flags, bins, index into the FP64 table
  cf* phi = (cf*)p;              p += sizeof(cf) * NP;
  cf* plo = (cf*)p;              p += has_plo ? sizeof(cf) * NP : 0;   // lo part of refined positions
  cdf* ulimb = (cdf*)p;          p += sizeof(cdf) * K;   // e^{2 pi i k / N_limb} as double-float
  // derivative mode: its state
  DerShared& ds = *(DerShared*)p;  p += DER ? sizeof(DerShared) : 0;
  p = (unsigned char*)(((uintptr_t)p + 15) & ~(uintptr_t)15);
  // the ray stage's tables take the place of the image-limb slots, which
  // nothing reads once the sectors stand (16-byte rows of the offset table)
  unsigned char* pr_ = p;
  float* tabf = (float*)pr_;     pr_ += sizeof(cf) * tabcap;        // group offsets (cos d - 1, sin d)
  AnchorF* anch = (AnchorF*)pr_; pr_ += sizeof(AnchorF) * MAXANCH;
  float2* spc = (float2*)pr_;    pr_ += sizeof(float2) * MAXANCH;  // spot centre in each anchor's frame
  int* wqueue = (int*)pr_;       pr_ += DER ? sizeof(int) * NW * DQ : sizeof(int2) * NW * FQ;  // boundary points, a queue per warp
  float* rowp = (float*)pr_;     pr_ += sizeof(float) * 32 * tcap;    // forward: the tasks' terms
  float* pterm = (float*)pr_;    pr_ += sizeof(float) * PCAP * tcap;
  int* pcnt = (int*)pr_;         pr_ += sizeof(int) * tcap;
  float* r32 = (float*)p;        p += sizeof(float) * NP;
  float* rl32 = (float*)p;       p += sizeof(float) * NP;   // r = r32 + rl32 (double-float)
  float* t32 = (float*)p;        p += sizeof(float) * NP;
  float* e32 = (float*)p;        p += sizeof(float) * NP;
  double* pr = (double*)p;       p += sizeof(double) * PMAX;
  double* pt = (double*)p;       p += sizeof(double) * PMAX;
  int* queue = (int*)p;          p += sizeof(int) * QMAX;
  short* pidx = (short*)p;       p += sizeof(short) * ((NP + 7) & ~7);
  uint8_t* meta = (uint8_t*)p;   p += (NP + 15) & ~15;
  uint8_t* tb = (uint8_t*)p;     p += (NP + 15) & ~15;
  uint8_t* rb = (uint8_t*)p;     p += (NP + 15) & ~15;
  DualD* cdual = ds.cx;
  BoxT<DualD>* bdual = ds.box;

  if (tid == 0) {
    sh.cur_set = -1;
    sh.warm = 0;
    sh.ht = 2.0 * kPi / BT;
    sh.htf = (float)sh.ht;
    if constexpr (DER) {
      float4* aA = (float4*)pr_;
      float2* acs = (float2*)(aA + MAXANCH);
      double* sums = (double*)(acs + MAXANCH), *ws = sums + NW * DSUM * 32;
      der_sh = {acs, aA, sums, ws, ccap ? (double2*)(ws + 5 * DSUM * TASK_WARPS) : nullptr};
    }
    rays_sh.P = {anch, spc, tabf, wqueue, rowp, pterm, pcnt, DER ? 1 << 30 : tcap, tabcap, ccap, g.n_r, g.n_theta, g.uniform, g.ld_split && !g.uniform ? 1 : 0,
                 diag_cnt ? 1 : 0, 1.0f, (float)g.s_fac, g.grad_rule, g.delta_c};
  }
  for (int k = tid; k < K; k += NT) {
    double sn, cs;
    sincospi(2.0 * (double)k / (double)K, &sn, &cs);
    ulimb[k].x = df_from_double(cs);
    ulimb[k].y = df_from_double(sn);
  }
  __syncthreads();

  // tiles: all (set, epoch) pairs, or the listed indices s * E + e
  const long long ntiles = items ? (long long)n_items : (long long)S * E;
  const long long t_begin = (long long)blockIdx.x * tiles_per_block;
  int law_set = -1;
  bool law_gen = false;
  for (long long tile = t_begin; tile < t_begin + tiles_per_block && tile < ntiles; ++tile) {
    long long q = items ? (long long)items[tile] : tile;
    if (q < 0 || q >= (long long)S * E) continue;  // block-uniform: skips the whole tile
    const int s = (int)(q / E), e = (int)(q % E);
    if constexpr (LAW != 2) {
      // the other instantiation takes this set (block-uniform)
      if (s != law_set) { law_set = s; law_gen = generic_law(P[s], g); }
      if (law_gen != (LAW == 1)) continue;
    }
    // ------------------------------------------------ set and epoch set-up
    if (tid == 0) {
      if (s != sh.cur_set) {
        icrs_params prm = P[s];
        sh.L = make_lens(prm);
        sh.rho = prm.rho;
        sh.u1 = prm.u1;
        sh.u2 = prm.u2;
        sh.pa[0] = prm.a1; sh.pa[1] = prm.a2; sh.pa[2] = prm.a3; sh.pa[3] = prm.a4;
        {
          // limb darkening I = I0 [1 - u1 (1 - mu) - u2 (1 - mu)^2 - sum_k a_k
          // (1 - mu^(k/2))], mu = sqrt(1 - d^2/rho^2), I0 = 1 / (pi (1 - u1/3 -
          // u2/6 - sum_k a_k k/(k+4))) (the linear law of Appendix A.2 when
          // the others are 0); uniform: I = 1/pi.  As a polynomial in s =
          // mu^(1/2):
          //   I = c0f + c1f mu + c2f mu^2 + s (c1h + c3h mu),
          //   c0f = I0 (1 - u1 - u2 - sum a) (the limb value), c1f = I0 (u1 +
          //   2 u2 + a2), c2f = I0 (a4 - u2), c1h = I0 a1, c3h = I0 a3.
          // Formed once per set by one thread: every thread forming them for
          // every epoch cost 38k of the 239k cycles that the ray stage of a
          // 64 x 256 epoch took (an FP64 instruction occupies the SM for
          // about 16 cycles, whatever its warp's active lanes).
          const double sa_ = sh.pa[0] / 5.0 + sh.pa[1] * (2.0 / 6.0) + sh.pa[2] * (3.0 / 7.0) + sh.pa[3] * 0.5;
          const double I0d = 1.0 / (kPi * (1.0 - sh.u1 / 3.0 - sh.u2 / 6.0 - sa_));
          sh.I0 = g.uniform ? (float)(1.0 / kPi) : (float)I0d;
          sh.c0f = g.uniform ? sh.I0
                             : (float)(I0d * (1.0 - sh.u1 - sh.u2 - sh.pa[0] - sh.pa[1] - sh.pa[2] - sh.pa[3]));
          sh.c1f = g.uniform ? 0.f : (float)(I0d * (sh.u1 + 2.0 * sh.u2 + sh.pa[1]));
          sh.c2f = g.uniform ? 0.f : (float)(I0d * (sh.pa[3] - sh.u2));
          sh.c1h = g.uniform ? 0.f : (float)(I0d * sh.pa[0]);
          sh.c3h = g.uniform ? 0.f : (float)(I0d * sh.pa[2]);
          sh.half = (sh.c1h != 0.f || sh.c3h != 0.f) ? 1 : 0;
        }
        sh.spot = prm.spot_c != 0.0;
        sh.generic = sh.half || sh.spot;
        sh.spot_x = prm.spot_x; sh.spot_y = prm.spot_y; sh.spot_r = prm.spot_r; sh.spot_c = prm.spot_c;
        sh.spot_rr32 = (float)(sh.rho * prm.spot_r);
        sh.spot_f32 = (float)(1.0 - prm.spot_c);
        sh.spot_bad = sh.spot && !(prm.spot_r >= 0.0 && prm.spot_c < 1.0 &&
                                   hypot(prm.spot_x, prm.spot_y) + prm.spot_r <= 1.0);
        sh.spot_new = sh.spot && !sh.spot_bad;
        sh.spot_norm = 1.0;
        sh.spot_gu = 0.0;
        sh.spot_acc[0] = sh.spot_acc[1] = 0.0;
        for (int j = 0; j < NL; ++j) {
          sh.eps32[j] = (float)sh.L.eps[j];
          double eps[NL];
          cd a[NL], D[NL + 1], Ee[NL];
          for (int i = 0; i < NL; ++i) { eps[i] = sh.L.eps[i]; a[i] = sh.L.a[i] - sh.L.a[j]; sh.aj32[j][i] = tof(a[i]); }
          poly_DE<NL, double>(eps, a, D, Ee);
          for (int i = 0; i <= NL; ++i) { sh.D32[j][i] = tof(D[i]); sh.D64[j][i] = D[i]; }
          for (int i = 0; i < NL; ++i) { sh.E32[j][i] = tof(Ee[i]); sh.E64[j][i] = Ee[i]; }
          for (int i = 0; i < NL; ++i) { sh.adf[j][i][0] = df_from_double(a[i].x); sh.adf[j][i][1] = df_from_double(a[i].y); }
          sh.epsdf[j] = df_from_double(sh.L.eps[j]);
        }
        sh.l2 = -1;
        if (NL == 3) {
          int c2 = -1;
          for (int i = 0; i < 3; ++i) {
            if (i == sh.L.ll) continue;
            if (c2 < 0 || sh.L.eps[i] < sh.L.eps[c2]) c2 = i;
          }
          sh.l2 = c2;
        }
        sh.adf_ll[0] = df_from_double(sh.L.a[sh.L.ll].x);
        sh.adf_ll[1] = df_from_double(sh.L.a[sh.L.ll].y);
        sh.rhodf = df_from_double(prm.rho);
        sh.warm = 0;
        sh.cur_set = s;
      } else {
        sh.warm = 1;  // previous tile of this block was the previous epoch of this set
        sh.spot_new = 0;
      }
      sh.wc = source_centre(P[s], T_[(size_t)s * E + e]);
      if (DER) {
        // d w_c / d(t0, tE, u0, alpha) and d(a_j, eps_j) / d(s, q) (binary):
        // w_c = tau (cos a, sin a) + u0 (-sin a, cos a), tau = (t - t0) / tE;
        // a_1 = -q s / (1 + q), a_2 = s / (1 + q), eps_1 = 1 / (1 + q),
        // eps_2 = q / (1 + q)
        const icrs_params& pp = P[s];
        double tau = (T_[(size_t)s * E + e] - pp.t0) / pp.tE;
        double sa, ca;
        sincos(pp.alpha, &sa, &ca);
        ds.dwc[0] = mk(-ca / pp.tE, -sa / pp.tE);
        ds.dwc[1] = mk(-tau * ca / pp.tE, -tau * sa / pp.tE);
        ds.dwc[2] = mk(-sa, ca);
        ds.dwc[3] = mk(-tau * sa - pp.u0 * ca, tau * ca - pp.u0 * sa);
        double oq = 1.0 + pp.q;
        ds.dadp[0][0] = -pp.q / oq;  ds.dadp[0][1] = -pp.s / (oq * oq);
        ds.dadp[1][0] = 1.0 / oq;    ds.dadp[1][1] = -pp.s / (oq * oq);
        ds.depsq[0] = -1.0 / (oq * oq);
        ds.depsq[1] = 1.0 / (oq * oq);
      }
      for (int j = 0; j < NL; ++j) {
        cd d = sh.wc - sh.L.a[j];
        sh.wcj32[j] = tof(d);
        sh.wcdf[j][0] = df_from_double(d.x);
        sh.wcdf[j][1] = df_from_double(d.y);
      }
      sh.status = 0u;
      sh.qn = 0;
      sh.pn = 0;
      for (int c = 0; c < 16; ++c) sh.cnt[c] = 0;
      sh.clk0 = clock64();
      sh.tocc[0] = sh.tocc[1] = sh.tocc[2] = sh.tocc[3] = 0u;
    }
    __syncthreads();
    const int ll = sh.L.ll;
    const float rho32 = (float)sh.rho;
    if (LAW != 0 && sh.spot_new) {
      // the spot's share of the unspotted flux F_spot = int_spot I dA (rho
      // units, the disk's flux is 1) and dF_spot/du1, once per set: polar
      // quadrature about the spot centre, the periodic trapezoid rule in the
      // angle (64 nodes), 8-point Gauss-Legendre in the radius on 16 panels
      // graded geometrically toward the spot's edge
      double gx[8], gw[8];
      for (int i = 0; i < 8; ++i) {
        double z = cos(kPi * (i + 0.75) / 8.5), dp = 1.0;
        for (int it = 0; it < 60; ++it) {
          double p0 = 1.0, p1 = z;
          for (int k = 2; k <= 8; ++k) { const double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k; p0 = p1; p1 = p2; }
          dp = 8.0 * (z * p1 - p0) / (z * z - 1.0);
          const double dz = p1 / dp;
          z -= dz;
          if (fabs(dz) < 1e-15) break;
        }
        gx[i] = z;
        gw[i] = 2.0 / ((1.0 - z * z) * dp * dp);
      }
      const double sa = sh.pa[0] / 5.0 + sh.pa[1] * (2.0 / 6.0) + sh.pa[2] * (3.0 / 7.0) + sh.pa[3] * 0.5;
      const double I0d = g.uniform ? 1.0 / kPi : 1.0 / (kPi * (1.0 - sh.u1 / 3.0 - sh.u2 / 6.0 - sa));
      double f = 0.0, fu = 0.0;
      for (int idx = tid; idx < 16 * 8 * 64; idx += NT) {
        const int b = idx / 512, i = (idx / 64) & 7, j = idx & 63;
        const double lo = b == 0 ? 0.0 : sh.spot_r * (1.0 - ldexp(1.0, -b));
        const double hi = b == 15 ? sh.spot_r : sh.spot_r * (1.0 - ldexp(1.0, -(b + 1)));
        const double rr = 0.5 * (hi - lo) * gx[i] + 0.5 * (hi + lo);
        const double w_ = 0.5 * (hi - lo) * gw[i] * rr * (2.0 * kPi / 64.0);
        double sn_, cs_;
        sincospi(2.0 * j / 64.0, &sn_, &cs_);
        const double x = sh.spot_x + rr * cs_, y = sh.spot_y + rr * sn_;
        const double mu = sqrt(fmax(1.0 - (x * x + y * y), 0.0));
        double I = 1.0, Iu = 0.0;
        if (!g.uniform) {
          const double om = 1.0 - mu, sq = sqrt(mu);
          I = 1.0 - sh.u1 * om - sh.u2 * om * om - sh.pa[0] * (1.0 - sq) - sh.pa[1] * (1.0 - mu) -
              sh.pa[2] * (1.0 - sq * mu) - sh.pa[3] * (1.0 - mu * mu);
          // dI/du1 = (pi/3) I0 I - I0 (1 - mu), with I = I0 x the bracket
          Iu = (kPi / 3.0) * I0d * I0d * I - I0d * om;
        }
        f += w_ * I0d * I;
        fu += w_ * Iu;
      }
      for (int o = 16; o > 0; o >>= 1) {
        f += __shfl_xor_sync(0xffffffffu, f, o);
        fu += __shfl_xor_sync(0xffffffffu, fu, o);
      }
      if (lane == 0) { atomicAdd(&sh.spot_acc[0], f); atomicAdd(&sh.spot_acc[1], fu); }
      __syncthreads();
      if (tid == 0) {
        // A = N S / rho^2, N = 1 / (1 - c F_spot): dN/du1 = N^2 c dF/du1,
        // so dA/du1 gains A N c dF/du1 (spot_gu)
        sh.spot_norm = 1.0 / (1.0 - sh.spot_c * sh.spot_acc[0]);
        sh.spot_gu = sh.spot_norm * sh.spot_c * sh.spot_acc[1];
      }
      __syncthreads();
    }

    // ------------------------------------------------ 1. limb roots (FP32 EA)
    // Cold start: 32 anchor limb points from the Cauchy circle, then every
    // limb point from its nearest anchor; warm start: from the same limb
    // point of the previous epoch.
    const bool warm = sh.warm;
    const int nanc = K < 32 ? K : 32;
    if (!warm) {
      if (warp == 0 && lane < nanc) {
        int k = (int)(((long long)lane * K) / nanc);
        float sp, cp;
        sincospif(2.0f * (float)k / (float)K, &sp, &cp);
        cf w = mk(sh.wcj32[ll].x + rho32 * cp, sh.wcj32[ll].y + rho32 * sp);
        cf b[N + 1];
        lens_poly<NL, float>(sh.eps32, sh.aj32[ll], sh.D32[ll], sh.E32[ll], w, b);
        cf z[N];
        float last[N];
        cauchy_start<N>(b, z);
        int it = ehrlich_aberth_f32<N>(b, z, g.max_iter, 4.0f * EPS32, last);
        if (it < 0) atomicOr(&sh.status, ICRS_ST_NONCONV);
        for (int j = 0; j < N; ++j) sh.anc[lane][j] = z[j];
      }
      __syncthreads();
    }
    for (int k = tid; k < K; k += NT) {
      float sp = ulimb[k].y.hi, cp = ulimb[k].x.hi;
      cf w = mk(sh.wcj32[ll].x + rho32 * cp, sh.wcj32[ll].y + rho32 * sp);
      cf b[N + 1];
      lens_poly<NL, float>(sh.eps32, sh.aj32[ll], sh.D32[ll], sh.E32[ll], w, b);
      cf z[N];
      if (warm) {
        for (int j = 0; j < N; ++j) z[j] = phi[k * N + j];
      } else {
        int a = (int)(((long long)k * nanc + K / 2) / K);
        if (a >= nanc) a = nanc - 1;
        for (int j = 0; j < N; ++j) z[j] = sh.anc[a][j];
      }
      // separate coincident starts
      for (int j = 1; j < N; ++j)
        for (int i = 0; i < j; ++i)
          if (abs2(z[j] - z[i]) < 1e-24f) z[j] = z[j] + mk(1e-6f * (j + 1), 1e-6f * j);
      float last[N];
      int it = ehrlich_aberth_f32<N>(b, z, g.max_iter, 4.0f * EPS32, last);
      if (it < 0) {
        // fall back to a cold start
        cauchy_start<N>(b, z);
        it = ehrlich_aberth_f32<N>(b, z, g.max_iter, 4.0f * EPS32, last);
        if (it < 0) atomicOr(&sh.status, ICRS_ST_NONCONV);
      }
      // Candidate roots (frame f, position in that frame).  Triple lens: the
      // polynomial about the lightest lens cannot resolve the cluster of
      // roots beside the second light lens in FP32, so a second EA about
      // that lens (warm-started from the first) supplies the roots nearest
      // to it.
      cf cz[2 * N];
      signed char cfm[2 * N];
      int nc = 0;
      const int l2 = sh.l2;
      cf z2[N];
      if (NL == 3) {
        cf w2 = w - sh.aj32[ll][l2];
        cf b2[N + 1];
        lens_poly<NL, float>(sh.eps32, sh.aj32[l2], sh.D32[l2], sh.E32[l2], w2, b2);
        for (int j = 0; j < N; ++j) z2[j] = z[j] - sh.aj32[ll][l2];
        float last2[N];
        if (ehrlich_aberth_f32<N>(b2, z2, g.max_iter, 4.0f * EPS32, last2) < 0) atomicOr(&sh.status, ICRS_ST_NONCONV);
      }
      for (int j = 0; j < N; ++j) {
        int nj = ll;
        float best = abs2(z[j]);
        for (int i = 0; i < NL; ++i) {
          if (i == ll) continue;
          float d = abs2(z[j] - sh.aj32[ll][i]);
          if (d < best) { best = d; nj = i; }
        }
        if (NL == 3 && nj == l2) continue;
        cz[nc] = z[j]; cfm[nc] = (signed char)ll; ++nc;
      }
      int n1 = nc;  // candidates from the first frame
      if (NL == 3) {
        for (int j = 0; j < N; ++j) {
          int nj = l2;
          float best = abs2(z2[j]);
          for (int i = 0; i < NL; ++i) {
            if (i == l2) continue;
            float d = abs2(z2[j] - sh.aj32[l2][i]);
            if (d < best) { best = d; nj = i; }
          }
          if (nj != l2) continue;
          cz[nc] = z2[j]; cfm[nc] = (signed char)l2; ++nc;
        }
      }
      // The two frames can disagree about which roots lie nearest the
      // second light lens (a root by a cell boundary, kept from both): drop
      // the first-frame candidate closest to a second-frame one, which
      // resolves that cluster better, until N remain.
      while (NL == 3 && nc > N && n1 > 0) {
        int bi = 0;
        float bd = __int_as_float(0x7f800000);
        for (int i = 0; i < n1; ++i)
          for (int j = n1; j < nc; ++j) {
            const float d = abs2(cz[i] - (cz[j] + sh.aj32[ll][l2]));
            if (d < bd) { bd = d; bi = i; }
          }
        for (int i = bi; i < nc - 1; ++i) { cz[i] = cz[i + 1]; cfm[i] = cfm[i + 1]; }
        --nc;
        --n1;
      }
      if (nc > N) { atomicOr(&sh.status, ICRS_ST_OVERFLOW); nc = N; }
      const float img_tol = (float)g.img_tol;
      for (int j = 0; j < N; ++j) {
        int pslot = k * N + j;
        meta[pslot] = 0;
        pidx[pslot] = -1;
        e32[pslot] = 0.f;
        if (j >= nc) {
          // unused slot (triple, fewer candidates): keep a warm start
          phi[pslot] = z[j];
          continue;
        }
        const int f = cfm[j];
        const cf zf = cz[j];
        // position in the lightest lens's frame (warm start for the next epoch)
        phi[pslot] = (f == ll) ? zf : zf + sh.aj32[ll][f];
        // nearest lens, offset x in its frame
        int nj = f;
        float best = abs2(zf);
        for (int i = 0; i < NL; ++i) {
          if (i == f) continue;
          float d = abs2(zf - sh.aj32[f][i]);
          if (d < best) { best = d; nj = i; }
        }
        cf x = (nj == f) ? zf : zf - sh.aj32[f][nj];
        cf wj = w - sh.aj32[ll][nj];
        // FP32 screen: roots whose residual is far above img_tol are not images
        cf F32 = lens_map<NL, float>(sh.eps32, sh.aj32[nj], x) - wj;
        float noise = 0.f;
        for (int i = 0; i < NL; ++i) noise += sh.eps32[i] * rsqrtf(fmaxf(abs2(x - sh.aj32[nj][i]), 1e-37f));
        noise = 16.0f * EPS32 * (noise + sqrtf(abs2(x)) + sqrtf(abs2(wj)) + 1.0f);
        float res32 = sqrtf(abs2(F32));
        if (res32 == res32 && res32 - noise > 4.0f * img_tol) continue;
        // compensated residual F = x - sum eps_i (x - a_i)/|x - a_i|^2 - w in
        // double-float (frame of lens nj), then one Newton step in FP32
        df wx = df_add(sh.wcdf[nj][0], df_mul(sh.rhodf, ulimb[k].x));
        df wy = df_add(sh.wcdf[nj][1], df_mul(sh.rhodf, ulimb[k].y));
        df Fx = df_make(x.x, 0.f), Fy = df_make(x.y, 0.f);
        for (int i = 0; i < NL; ++i) {
          df dx = df_sub(df_make(x.x, 0.f), sh.adf[nj][i][0]);
          df dy = df_sub(df_make(x.y, 0.f), sh.adf[nj][i][1]);
          df nn = df_add(df_mul(dx, dx), df_mul(dy, dy));
          df tt = df_div(sh.epsdf[i], nn);
          Fx = df_sub(Fx, df_mul(dx, tt));
          Fy = df_sub(Fy, df_mul(dy, tt));
        }
        Fx = df_sub(Fx, wx);
        Fy = df_sub(Fy, wy);
        cf F = mk(Fx.hi + Fx.lo, Fy.hi + Fy.lo);
        float res = sqrtf(abs2(F));
        // position kept for an FP64 decision if needed
        // position of this root in the lightest lens's frame, double-float:
        // x (exact float) + (a_nj - a_ll) (double-float)
        df px = df_add(df_make(x.x, 0.f), sh.adf[ll][nj][0]);
        df py = df_add(df_make(x.y, 0.f), sh.adf[ll][nj][1]);
        if (!(res == res) || res > 0.25f * img_tol) {
          if (!(res >= 4.0f * img_tol)) {  // FP64 decides
            meta[pslot] = M_UNSURE;
            phi[pslot] = mk(px.hi, py.hi);
          }
          continue;
        }
        cf gm = shear<NL, float>(sh.eps32, sh.aj32[nj], x);
        float ag2 = abs2(gm), ag = sqrtf(ag2);
        float det = 1.0f - ag2;
        float jinv = (1.0f + ag) / fmaxf(fabsf(det), 1e-30f);
        cf dz = scl(cj(gm) * cj(F) - F, 1.0f / det);
        // second-derivative scale |dgamma/dz| = |sum 2 eps_i/(x - a_i)^3|
        cf g3 = mk(0.f, 0.f);
        for (int i = 0; i < NL; ++i) { cf id = inv(x - sh.aj32[nj][i]); g3 = g3 + scl(id * id * id, 2.0f * sh.eps32[i]); }
        float adz2 = abs2(dz);
        // refined position: a_nj + x + dz (lightest frame: aj32[ll][nj] + x + dz)
        px = df_add(px, df_make(dz.x, 0.f));
        py = df_add(py, df_make(dz.y, 0.f));
        df zx = df_add(px, sh.adf_ll[0]);
        df zy = df_add(py, sh.adf_ll[1]);
        float zxf = zx.hi + zx.lo, zyf = zy.hi + zy.lo;
        // r = |z| as a double-float: r^2 in double-float, then one Newton
        // correction of the float square root
        df r2 = df_add(df_mul(zx, zx), df_mul(zy, zy));
        float rr = sqrtf(r2.hi);
        df rsq = two_prod(rr, rr);
        float rlo = ((r2.hi - rsq.hi) - rsq.lo + r2.lo) / (2.0f * rr);
        float th = atan2f(zyf, zxf);
        // error bound of the double-float r after the step: second-order Newton
        // term plus the double-float residual's rounding
        float ee = 4.0f * sqrtf(abs2(g3)) * adz2 * jinv + jinv * 1e-12f * (1.0f + noise / (16.0f * EPS32)) +
                   1e-12f * rr;
        if (!(rr == rr) || !(th == th) || !(ee == ee) || isinf(ee)) {
          meta[pslot] = M_UNSURE;
          phi[pslot] = mk(px.hi, py.hi);
          continue;
        }
        meta[pslot] = M_VALID;
        phi[pslot] = mk(px.hi, py.hi);
        if (has_plo) plo[pslot] = mk(px.lo, py.lo);
        r32[pslot] = rr;
        rl32[pslot] = rlo;
        t32[pslot] = th;
        e32[pslot] = ee;
      }
    }
    __syncthreads();

    if (diag_cnt && tid == 0) { long long c_ = clock64(); sh.cnt[4] = (int)min(c_ - sh.clk0, 2000000000LL); sh.clk0 = c_; }
    // ------------------------------------------------ 1b. ambiguous roots in FP64
    for (int ps = tid; ps < NP; ps += NT)
      if (meta[ps] & M_UNSURE) q_push(sh, queue, ps);
    __syncthreads();
    {
      int qn = min(sh.qn, QMAX);
      for (int qi = tid; qi < qn; qi += NT) {
        int ps = queue[qi];
        int k = ps / N;
        atomicAdd(&sh.cnt[1], 1);
        cd w = limb_point64(sh, k, K);
        cd z0 = tod(phi[ps]) + sh.L.a[ll];
        double r, th;
        int conv = 1;
        int ok = validate_root64<NL>(sh, z0, w, g.img_tol, &r, &th, &conv);
        uint8_t m = 0;
        if (ok && NL == 2 && !conv) {
          // not converged: kept as an image with an infinite error bound, so
          // that the limb point goes to the FP64 re-solve below
          m = M_VALID;
          const float rh = (float)r;
          r32[ps] = rh; rl32[ps] = (float)(r - (double)rh); t32[ps] = (float)th;
          e32[ps] = __int_as_float(0x7f800000);
        } else if (ok) {
          int pi = atomicAdd(&sh.pn, 1);
          float rh = (float)r;
          if (pi < PMAX) { pr[pi] = r; pt[pi] = th; pidx[ps] = (short)pi; m = M_VALID | M_EXACT; r32[ps] = rh; rl32[ps] = (float)(r - (double)rh); t32[ps] = (float)th; e32[ps] = 0.f; }
          else { m = M_VALID; atomicOr(&sh.status, ICRS_ST_OVERFLOW); r32[ps] = rh; rl32[ps] = (float)(r - (double)rh); t32[ps] = (float)th; e32[ps] = 1e-12f; }
        }
        meta[ps] = m;
      }
    }
    __syncthreads();
    if (tid == 0) sh.qn = 0;
    __syncthreads();
    // image counts per limb point; an illegal count sends the limb point to
    // an FP64 root solve (warm-started from its FP32 roots) and FP64
    // validation of every root
    auto legal_count = [&](int m) -> bool {
      return (NL == 2) ? (m == 3 || m == 5) : (m == 4 || m == 6 || m == 8 || m == 10);
    };
    // Binary lens: the same FP64 re-solve takes limb points whose FP32 image
    // set is not trustworthy although its count is legal: an image whose
    // refining Newton step left a large error bound (an approximation next to
    // a critical curve, where det J ~ 0 sends the step far away), two slots
    // holding the same image (two approximations that met at one root while
    // another image was missed), or two non-image roots within PAIR_TOL of
    // each other (a close image pair that the FP32 polynomial rounded into a
    // pair of false roots; seen at separations up to 5.5e-3).  Without this check the image set, and
    // so the sectors, could depend on where the iteration started.  (Triple
    // lens: images beside the small lenses have large second derivatives and
    // so large bounds, and the FP64 re-solve in the lightest lens's frame is
    // less accurate there than the two-frame FP32 solve; only illegal counts
    // are re-solved.)
    for (int k = tid; k < K; k += NT) {
      int m = 0;
      bool suspect = false;
      float zx[N], zy[N];
      if (NL == 2) {
        // two roots that are not images, close together: the FP32
        // coefficients may have turned a close image pair (a limb point just
        // inside a fold caustic) into a pair of false roots
        for (int j = 0; j < N; ++j) {
          if (meta[k * N + j] & M_VALID) continue;
          const cf a_ = phi[k * N + j];
          for (int i2 = 0; i2 < j; ++i2) {
            if (meta[k * N + i2] & M_VALID) continue;
            const float tol = PAIR_TOL * fmaxf(1.0f, sqrtf(abs2(a_) + 1e-30f));
            if (abs2(a_ - phi[k * N + i2]) <= tol * tol) suspect = true;
          }
        }
      }
      for (int j = 0; j < N; ++j) {
        const int ps = k * N + j;
        if (!(meta[ps] & M_VALID)) continue;
        const bool ex = meta[ps] & M_EXACT;
        const float r = ex ? (float)pr[pidx[ps]] : r32[ps];
        const float th = ex ? (float)pt[pidx[ps]] : t32[ps];
        if (!ex && !(e32[ps] <= EE_SUSPECT * fmaxf(1.0f, r))) suspect = true;
        // (the refined position itself; a polished or validated root's is r e^{i th})
        float x, y;
        if (ex) {
          float sn, cs;
          sincosf(th, &sn, &cs);
          x = r * cs - (float)sh.L.a[ll].x;
          y = r * sn - (float)sh.L.a[ll].y;
        } else {
          x = phi[ps].x;
          y = phi[ps].y;
        }
        for (int i2 = 0; i2 < m; ++i2) {
          const float dx = x - zx[i2], dy = y - zy[i2];
          const float tol = DUP_TOL * fmaxf(1.0f, r);
          if (dx * dx + dy * dy <= tol * tol) suspect = true;
        }
        zx[m] = x; zy[m] = y;
        ++m;
      }
      if (!legal_count(m) || (NL == 2 && suspect)) q_push(sh, queue, k);
    }
    __syncthreads();
    {
      const int qn = min(sh.qn, QMAX);
      // a few points: one per warp; more: as many as a warp has lanes for;
      // beyond one round of those: one per thread, since a warp's FP64
      // instruction occupies the SM for 16 cycles however many lanes are
      // active (64 sets, always by warps: 32,000 epochs at 64 x 256 55.5 ms
      // against 48.4; always by threads: 6,400 at 512 x 1024 27.5 against 26.9,
      // and one epoch alone waits up to 400k cycles)
      const int np = qn <= NW ? 1 : 32 / N;
      if (qn <= NW * (32 / N)) {
        for (int qi = warp * np; qi < qn; qi += NW * np) {
          if (lane == 0) atomicAdd(&sh.cnt[1], min(np, qn - qi));
          resolve_limb_points64<NL>(sh, queue + qi, min(np, qn - qi), K, g.max_iter, g.img_tol, PMAX, phi, r32, rl32,
                                    t32, e32, pidx, meta, pr, pt);
        }
      } else {
        for (int qi = tid; qi < qn; qi += NT) {
          atomicAdd(&sh.cnt[1], 1);
          const int m = resolve_limb_point64<NL>(sh, queue[qi], K, g.max_iter, g.img_tol, PMAX, phi, r32, rl32, t32, e32,
                                                 pidx, meta, pr, pt);
          if (!legal_count(m)) atomicOr(&sh.status, ICRS_ST_IMGCOUNT);
        }
      }
    }
    __syncthreads();
    if (tid == 0) sh.qn = 0;
    __syncthreads();

    // polish helper: process the queue (points not yet exact)
    auto run_polish = [&]() {
      __syncthreads();
      int qn = min(sh.qn, QMAX);
      for (int qi = tid; qi < qn; qi += NT) {
        int ps = queue[qi];
        if (meta[ps] & M_EXACT) continue;
        int k = ps / N;
        atomicAdd(&sh.cnt[0], 1);
        double r, th;
        if (has_plo && e32[ps] <= 1e-11f) {
          // the double-float position is already accurate to ~1e-12
          cd z0 = mk((double)phi[ps].x + (double)plo[ps].x, (double)phi[ps].y + (double)plo[ps].y) + sh.L.a[ll];
          r = sqrt(z0.x * z0.x + z0.y * z0.y);
          th = atan2(z0.y, z0.x);
        } else {
          cd w = limb_point64(sh, k, K);
          cd z0 = tod(phi[ps]) + sh.L.a[ll];
          polish_image64<NL>(sh, z0, w, &r, &th);
        }
        int pi = atomicAdd(&sh.pn, 1);
        if (pi < PMAX) {
          pr[pi] = r; pt[pi] = th; pidx[ps] = (short)pi;
          float rh = (float)r;
          r32[ps] = rh; rl32[ps] = (float)(r - (double)rh); t32[ps] = (float)th; e32[ps] = 0.f;
          meta[ps] |= M_EXACT;
        } else {
          atomicOr(&sh.status, ICRS_ST_OVERFLOW);
        }
      }
      __syncthreads();
      if (tid == 0) sh.qn = 0;
      __syncthreads();
    };
    // r of a slot: FP64 if polished, else the double-float (r32 + rl32)
    auto rv = [&](int ps) -> double { return (meta[ps] & M_EXACT) ? pr[pidx[ps]] : (double)r32[ps] + (double)rl32[ps]; };
    auto tv = [&](int ps) -> double { return (meta[ps] & M_EXACT) ? pt[pidx[ps]] : (double)t32[ps]; };

    if (diag_pts) {
      size_t o = ((size_t)s * E + e) * (size_t)NP;
      for (int ps = tid; ps < NP; ps += NT) {
        float* d = diag_pts + (o + ps) * 4;
        bool ex = meta[ps] & M_EXACT;
        if (meta[ps] & M_VALID) {
          d[0] = ex ? (float)pr[pidx[ps]] : r32[ps];
          d[1] = ex ? (float)pt[pidx[ps]] : t32[ps];
        } else {
          // a root that is not an image: its position (r, theta)
          const cd z_ = tod(phi[ps]) + sh.L.a[ll];
          d[0] = (float)sqrt(abs2(z_));
          d[1] = (float)atan2(z_.y, z_.x);
        }
        d[2] = (float)meta[ps];
        d[3] = e32[ps];
      }
    }
    if (diag_cnt && tid == 0) { long long c_ = clock64(); sh.cnt[5] = (int)min(c_ - sh.clk0, 2000000000LL); sh.clk0 = c_; }
    // ------------------------------------------------ 2. theta bins
    // The binning phases (2 to 7) walk the image-limb slots root by root (a
    // warp takes 32 neighbouring limb points of one root, which mostly belong
    // to one image): what they collect per angular interval or cell is then
    // reduced over the warp before one shared-memory atomic per interval,
    // instead of 32 atomics that queue on one word.
    const double ht = sh.ht;
    const float htf = sh.htf;
    const int KW = (K + 31) & ~31;  // limb points of one root, padded to whole warps
    // calls f(ps, valid) for every slot, all 32 lanes of a warp together
    auto for_slots = [&](auto f) {
      for (int idx = tid; idx < KW * N; idx += NT) {
        const int j = idx / KW, k = idx - j * KW;
        const int ps = k * N + j;
        const bool ok = k < K && (meta[k < K ? ps : 0] & M_VALID);
        f(ok ? ps : 0, ok);
      }
    };
    // calls f(in, id) once for every distinct id of the warp's lanes with
    // `has` set (in: this lane has that id), all lanes together
    auto by_id = [&](bool has, int id, auto f) {
      unsigned todo = __ballot_sync(0xffffffffu, has);
      while (todo) {
        const int id0 = __shfl_sync(0xffffffffu, id, __ffs(todo) - 1);
        const bool in = has && id == id0;
        f(in, id0);
        todo &= ~__ballot_sync(0xffffffffu, in);
      }
    };
    for (int ps = tid; ps < NP; ps += NT) {
      if (!(meta[ps] & M_VALID) || (meta[ps] & M_EXACT)) continue;
      // distance of the FP32 angle from the nearest bin edge, against the
      // error of that FP32 evaluation: the point's own bound e32 / r, atan2f
      // (<= 2 ulp of pi, 4.8e-7), the float pi (8.7e-8), the sum (2.4e-7),
      // and the division by the float bin width (<= 128 bins x 1.2e-7 bin
      // widths, 7.5e-7 rad): 1.6e-6 rad in all; 64 EPS32 = 3.8e-6 leaves a
      // factor of two.  Closer points get an FP64 angle.
      float u = (t32[ps] + kPiF) / htf;
      float fr = u - floorf(u);
      float d = fminf(fr, 1.0f - fr) * htf;
      float eth = e32[ps] / fmaxf(r32[ps], 1e-30f) + 64.0f * EPS32;
      if (d <= eth) q_push(sh, queue, ps);
    }
    run_polish();
    for_slots([&](int ps, bool ok) {
      int t = 0;
      if (ok) {
        if (meta[ps] & M_EXACT) t = (int)floor((pt[pidx[ps]] + kPi) / ht);
        else t = (int)floorf((t32[ps] + kPiF) / htf);
        t = min(max(t, 0), BT - 1);
        tb[ps] = (uint8_t)t;
      }
      unsigned w_ = 0u;  // lane i (< 4): word i of the warp's bins
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const unsigned o = __reduce_or_sync(0xffffffffu, ok && (t >> 5) == i ? 1u << (t & 31) : 0u);
        if (lane == i) w_ = o;
      }
      if (w_) atomicOr(&sh.tocc[lane], w_);
    });
    for (int i = tid; i < MAXT * MAXRB; i += NT) {
      const int T = i / MAXRB, b = i - T * MAXRB;
      sh.tmask[T][b][0] = sh.tmask[T][b][1] = sh.tmask[T][b][2] = sh.tmask[T][b][3] = 0u;
      sh.rrun[T][b] = -1;
      if (b == 0) {
        sh.t_rlo_u[T] = 0xffffffffu; sh.t_rhi_l[T] = 0u;
        sh.t_rlo[T] = ~0ull; sh.t_rhi[T] = 0ull;
        sh.t_s[T][0] = 0xffffffffu; sh.t_s[T][1] = 0u;
        sh.rocc[T] = 0u;
      }
    }
    __syncthreads();

    if (diag_cnt && tid == 0) { long long c_ = clock64(); sh.cnt[6] = (int)min(c_ - sh.clk0, 2000000000LL); sh.clk0 = c_; }
    if (diag_cnt && tid == 0) sh.cnt[13] = sh.cnt[0];
    // ------------------------------------------------ 3. theta runs (cyclic)
    // One warp, lane i the bins 32 i .. 32 i + 31 where words are formed and
    // one lane per bin where runs are numbered: a run starts at an occupied
    // bin whose predecessor (cyclic) is empty, and runs are numbered in cyclic
    // order from the first empty bin t0.
    if (warp == 0) {
      auto occb = [&](int t) -> bool { return (sh.tocc[t >> 5] >> (t & 31)) & 1u; };
      int nfree = BT, t0 = BT;  // empty bins, first empty bin
      nfree = BT - (__popc(sh.tocc[0]) + __popc(sh.tocc[1]) + __popc(sh.tocc[2]) + __popc(sh.tocc[3]));
      const bool full = nfree == 0;
      int nT = 0;
      if (nfree == BT) {
        for (int t = lane; t < 128; t += 32) sh.runT[t] = -1;
      } else if (full) {
        for (int t = lane; t < 128; t += 32) sh.runT[t] = t < BT ? 0 : -1;
        if (lane == 0) sh.startT[0] = 0;
        nT = 1;
      } else {
        for (int i = 3; i >= 0; --i) {
          const unsigned fr = ~sh.tocc[i];
          if (fr && 32 * i + __ffs(fr) - 1 < BT) t0 = 32 * i + __ffs(fr) - 1;
        }
        for (int t = lane; t < 128; t += 32) if (t >= BT || !occb(t)) sh.runT[t] = -1;
        // bins in cyclic order kk = 1 .. BT from t0: the run's number is the
        // count of run starts up to the bin, less one
        bool over = false;
        for (int k0 = 1; k0 <= BT; k0 += 32) {
          const int kk = k0 + lane;
          int t = t0 + kk;
          t = t >= BT ? t - BT : t;
          const bool oc = kk <= BT && occb(t);
          const bool st_ = oc && !occb(t == 0 ? BT - 1 : t - 1);
          const unsigned sb = __ballot_sync(0xffffffffu, st_);
          const int r = nT + __popc(sb & (0xffffffffu >> (31 - lane))) - 1;
          if (oc) {
            sh.runT[t] = (signed char)min(r, MAXT - 1);
            if (st_ && r < MAXT) sh.startT[r] = t;
          }
          if (oc && r >= MAXT) over = true;
          nT += __popc(sb);
        }
        nT = min(nT, MAXT);
        if (over) atomicOr(&sh.status, ICRS_ST_OVERFLOW);
      }
      if (lane == 0) { sh.nT = nT; sh.full = full ? 1 : 0; }
    }
    __syncthreads();
    const int nT = sh.nT;

    // ------------------------------------------------ 4. r range per theta run
    // Extremes in three narrowing passes: FP32 radii with their FP32 errors,
    // then the double-float radii of the points those leave (error e32,
    // mostly a few 1e-12), then FP64 polishes of the points still left whose
    // e32 is above 1e-11.  (Polishing every point that the FP32 pass leaves
    // took 255 polishes an epoch of the 64 x 256 batch; 54 are left, and phases
    // 2 to 7 went from 218k to 164k cycles.)
    for_slots([&](int ps, bool ok) {
      const int T = ok ? sh.runT[tb[ps]] : 0;
      const float r = r32[ps], er = (meta[ps] & M_EXACT) ? 4.0f * EPS32 * r : e32[ps] + 4.0f * EPS32 * r;
      by_id(ok, T, [&](bool in, int T0) {
        const unsigned lo = __reduce_min_sync(0xffffffffu, in ? fkey(r + er) : 0xffffffffu);
        const unsigned hi = __reduce_max_sync(0xffffffffu, in ? fkey(r - er) : 0u);
        if (lane == 0) { atomicMin(&sh.t_rlo_u[T0], lo); atomicMax(&sh.t_rhi_l[T0], hi); }
      });
    });
    __syncthreads();
    const float tiny = TINY_EXTENT * rho32;
    // r of a slot (the double-float r32 + rl32, which a polish sets too) less a
    // nearby float, and its error bound: the difference of the high parts is
    // exact, so the sum keeps 1e-7 of the difference
    auto r_from = [&](int ps, float ref, float* err) -> float {
      const float d = (r32[ps] - ref) + rl32[ps];
      *err = ((meta[ps] & M_EXACT) ? 0.f : e32[ps]) + 2e-7f * fabsf(d) + 1e-14f * r32[ps];
      return d;
    };
    for (int ps = tid; ps < NP; ps += NT) {
      if (!(meta[ps] & M_VALID)) continue;
      int T = sh.runT[tb[ps]];
      float r = r32[ps], er = (meta[ps] & M_EXACT) ? 4.0f * EPS32 * r : e32[ps] + 4.0f * EPS32 * r;
      if (fkey(r - er) <= sh.t_rlo_u[T] || fkey(r + er) >= sh.t_rhi_l[T]) {
        meta[ps] |= M_CAND;
        float e_;
        const float lo = r_from(ps, fkey_inv(sh.t_rlo_u[T]), &e_);
        atomicMin(&sh.t_s[T][0], fkey(lo + e_));
        const float hi = r_from(ps, fkey_inv(sh.t_rhi_l[T]), &e_);
        atomicMax(&sh.t_s[T][1], fkey(hi - e_));
      }
    }
    __syncthreads();
    for (int ps = tid; ps < NP; ps += NT) {
      if (!(meta[ps] & M_CAND)) continue;
      int T = sh.runT[tb[ps]];
      float e_;
      const float lo = r_from(ps, fkey_inv(sh.t_rlo_u[T]), &e_);
      bool cand = fkey(lo - e_) <= sh.t_s[T][0];
      const float hi = r_from(ps, fkey_inv(sh.t_rhi_l[T]), &e_);
      cand = cand || fkey(hi + e_) >= sh.t_s[T][1];
      if (!cand) { meta[ps] &= (uint8_t)~M_CAND; continue; }
      // an image smaller than tiny contributes below the parity tolerance:
      // its decisions stay in FP32
      bool is_tiny = fkey_inv(sh.t_rhi_l[T]) - fkey_inv(sh.t_rlo_u[T]) < tiny;
      // the double-float r (error e32) is exact enough unless e32 is large
      if (!(meta[ps] & M_EXACT) && !is_tiny && !(e32[ps] <= 1e-11f)) q_push(sh, queue, ps);
    }
    run_polish();
    for (int ps = tid; ps < NP; ps += NT) {
      if (!(meta[ps] & M_CAND)) continue;
      meta[ps] &= (uint8_t)~M_CAND;
      int T = sh.runT[tb[ps]];
      double r = rv(ps);
      atomicMin(&sh.t_rlo[T], dkey(r));
      atomicMax(&sh.t_rhi[T], dkey(r));
    }
    __syncthreads();
    if (tid < nT) {
      double lo = dkey_inv(sh.t_rlo[tid]), hi = dkey_inv(sh.t_rhi[tid]);
      const double h = (hi - lo) / BR;
      sh.rlo[tid] = lo;
      sh.hr[tid] = h;
      sh.rlh[tid] = (float)lo;
      sh.rll[tid] = (float)(lo - (double)(float)lo);
      sh.ihr[tid] = (float)(1.0 / h);
      sh.rsmall[tid] = !(h > 0.0) ? 2 : (h * BR < (double)tiny ? 1 : 0);
    }
    __syncthreads();

    if (diag_cnt && tid == 0) { long long c_ = clock64(); sh.cnt[7] = (int)min(c_ - sh.clk0, 2000000000LL); sh.clk0 = c_; }
    if (diag_cnt && tid == 0) sh.cnt[14] = sh.cnt[0];
    // ------------------------------------------------ 5. r bins per theta run
    // Bin of r within its angular interval, floor((r - r_lo) / h_r): in FP32
    // from the double-float r where the bin edge is farther than the FP32
    // error, else in FP64 (after an FP64 polish if the double-float r itself
    // is uncertain).
    auto rbin_u = [&](int ps, int T, float* err) -> float {
      const float ihr = sh.ihr[T];
      float dr = (r32[ps] - sh.rlh[T]) + (rl32[ps] - sh.rll[T]);
      float u = dr * ihr;
      *err = 4.0f * EPS32 * fabsf(u) + e32[ps] * ihr + 1e-6f;
      return u;
    };
    for (int ps = tid; ps < NP; ps += NT) {
      if (!(meta[ps] & M_VALID) || (meta[ps] & M_EXACT)) continue;
      int T = sh.runT[tb[ps]];
      if (sh.rsmall[T] || e32[ps] <= 1e-11f) continue;
      float eu;
      float u = rbin_u(ps, T, &eu);
      float fr = u - floorf(u);
      if (fminf(fr, 1.0f - fr) <= eu && u > 0.5f && u < (float)BR - 0.5f) q_push(sh, queue, ps);
    }
    run_polish();
    for_slots([&](int ps, bool ok) {
      const int T = ok ? sh.runT[tb[ps]] : 0;
      int b = 0;
      if (ok && sh.rsmall[T] != 2) {
        float eu;
        float u = rbin_u(ps, T, &eu);
        float fr = u - floorf(u);
        if (fminf(fr, 1.0f - fr) > eu) b = (int)floorf(u);
        else b = (int)floor((rv(ps) - sh.rlo[T]) / sh.hr[T]);
        b = min(max(b, 0), BR - 1);
      }
      if (ok) {
        rb[ps] = (uint8_t)b;
        atomicOr(&sh.tmask[T][b][tb[ps] >> 5], 1u << (tb[ps] & 31));
      }
      by_id(ok, T, [&](bool in, int T0) {
        const unsigned o = __reduce_or_sync(0xffffffffu, in ? 1u << b : 0u);
        if (lane == 0) atomicOr(&sh.rocc[T0], o);
      });
    });
    for (int i = tid; i < MAXCELL * 4; i += NT) {
      const int c = i >> 2, k = i & 3;
      sh.c_u[c][k] = (k & 1) ? 0u : 0xffffffffu;
      sh.c_x[c][k] = (k & 1) ? 0ull : ~0ull;
      sh.c_s[c][k] = (k & 1) ? 0u : 0xffffffffu;
      if (k == 0) sh.c_cnt[c] = 0;
    }
    if constexpr (DER) {
      for (int i = tid; i < MAXCELL_D * 4; i += NT) ds.cell_arg[i >> 2][i & 3] = 0x7fffffff;
    }
    __syncthreads();

    if (diag_cnt && tid == 0) { long long c_ = clock64(); sh.cnt[8] = (int)min(c_ - sh.clk0, 2000000000LL); sh.clk0 = c_; }
    if (diag_cnt && tid == 0) sh.cnt[15] = sh.cnt[0];
    // ------------------------------------------------ 6. gap probes, r runs, origin
    // One warp per theta run (round robin): every empty gap with points of a
    // shared theta bin on both sides is probed at its middle radius (FP32 with
    // a guard band, FP64 when the guard cannot decide).  The last warp tests
    // the origin meanwhile.
    if (warp == NW - 1 && lane == 0) {
      cd w0 = lens_map<NL, double>(sh.L.eps, sh.L.a, mk(0.0, 0.0));
      sh.origin_in = sqrt(abs2(w0 - sh.wc)) < sh.rho;
    }
    for (int T = warp; T < nT; T += NW) {
      unsigned int occ = sh.rocc[T];
      unsigned int fill = 0u;
      // this lane's r bin: its theta bins
      unsigned mine[4];
#pragma unroll
      for (int h = 0; h < 4; ++h) mine[h] = lane < BR ? sh.tmask[T][lane < MAXRB ? lane : 0][h] : 0u;
      for (int b = 1; b < BR; ++b) {
        if (((occ >> b) & 1u) || !((occ >> (b - 1)) & 1u)) continue;
        int e2 = b;
        while (e2 < BR && !((occ >> e2) & 1u)) ++e2;
        if (e2 >= BR) break;
        unsigned shared_[4];
#pragma unroll
        for (int h = 0; h < 4; ++h)
          shared_[h] = __reduce_or_sync(0xffffffffu, lane < b ? mine[h] : 0u) &
                       __reduce_or_sync(0xffffffffu, lane >= e2 ? mine[h] : 0u);
        bool hit = false;
        if (shared_[0] | shared_[1] | shared_[2] | shared_[3]) {
          const double rg = sh.rlo[T] + sh.hr[T] * 0.5 * (double)(b + e2);
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            if (hit || !shared_[h]) continue;
            const int t = 32 * h + lane;
            bool in = false;
            if (t < BT && ((shared_[h] >> lane) & 1u)) {
              double th = -kPi + (t + 0.5) * ht;
              float sth, cth;
              sincosf((float)th, &sth, &cth);
              cf z = mk((float)rg * cth, (float)rg * sth);
              float eps[NL];
              cf a[NL];
              for (int i = 0; i < NL; ++i) { eps[i] = sh.eps32[i]; a[i] = tof(sh.L.a[i]); }
              cf w = lens_map<NL, float>(eps, a, z);
              cf dw = w - tof(sh.wc);
              float d2 = abs2(dw);
              float errb = 64.0f * EPS32 * (sqrtf(abs2(w)) + 2.0f);
              float d = sqrtf(d2);
              if (fabsf(d - rho32) <= errb) {
                double s64, c64;
                sincos(th, &s64, &c64);
                cd z64 = mk(rg * c64, rg * s64);
                cd w64 = lens_map<NL, double>(sh.L.eps, sh.L.a, z64);
                in = sqrt(abs2(w64 - sh.wc)) < sh.rho;
              } else {
                in = d < rho32;
              }
            }
            hit = __any_sync(0xffffffffu, in);
          }
        }
        if (hit) fill |= ((e2 < 32 ? 1u << e2 : 0u) - 1u) & ~((1u << b) - 1u);
      }
      occ |= fill;
      // r runs: numbered by their first bins
      const unsigned starts = occ & ~(occ << 1);
      if (lane < BR && ((occ >> lane) & 1u))
        sh.rrun[T][lane] = (signed char)(__popc(starts & (0xffffffffu >> (31 - lane))) - 1);
      if (lane == 0) { sh.rocc[T] = occ; sh.cellbase[T + 1] = __popc(starts); }
    }
    __syncthreads();
    if (tid == 0) {
      sh.cellbase[0] = 0;
      int tot = 0;
      for (int T = 0; T < nT; ++T) { int c = sh.cellbase[T + 1]; sh.cellbase[T] = tot; tot += c; }
      sh.cellbase[nT] = tot;
      if (tot > MAXCELL) { tot = MAXCELL; atomicOr(&sh.status, ICRS_ST_OVERFLOW); }
      sh.ncell = tot;
      if (DER && tot > MAXCELL_D) atomicOr(&sh.status, ICRS_ST_OVERFLOW);
    }
    __syncthreads();

    if (diag_cnt && tid == 0) { long long c_ = clock64(); sh.cnt[9] = (int)min(c_ - sh.clk0, 2000000000LL); sh.clk0 = c_; }
    // ------------------------------------------------ 7. cell extremes
    auto cell_of = [&](int ps) -> int {
      int T = sh.runT[tb[ps]];
      int c = sh.cellbase[T] + sh.rrun[T][rb[ps]];
      return c < MAXCELL ? c : MAXCELL - 1;
    };
    // A point lies past the wrap of its angular interval when its bin comes
    // before the interval's first bin.  The decision is taken on the bin, not
    // on the angle: a point binned in FP64 next to the interval's first edge
    // can have an FP32 angle on the other side of that edge, and the FP32
    // candidate pass and the FP64 extreme pass must unwrap it alike.
    auto past_wrap = [&](int ps) -> bool { return (int)tb[ps] < sh.startT[sh.runT[tb[ps]]]; };
    auto unwrap_t = [&](int ps, double th) -> double { return past_wrap(ps) ? th + 2.0 * kPi : th; };
    // the FP32 angle, unwrapped (2 pi and the sum rounded: 4.1e-7 more, inside
    // the 16 EPS32 of et together with atan2f's 4.8e-7)
    auto unwrap_f = [&](int ps) -> float { return past_wrap(ps) ? t32[ps] + 2.0f * kPiF : t32[ps]; };
    auto er_et = [&](int ps, float* er, float* et) {
      const float r = r32[ps];
      const bool ex = meta[ps] & M_EXACT;
      *er = ex ? 4.0f * EPS32 * r : e32[ps] + 4.0f * EPS32 * r;
      *et = ex ? 16.0f * EPS32 : e32[ps] / fmaxf(r, 1e-30f) + 16.0f * EPS32;
    };
    for_slots([&](int ps, bool ok) {
      const int c = ok ? cell_of(ps) : 0;
      const float r = r32[ps];
      float er, et;
      er_et(ps, &er, &et);
      const float th = ok ? unwrap_f(ps) : 0.f;
      by_id(ok, c, [&](bool in, int c0) {
        const unsigned k0 = __reduce_min_sync(0xffffffffu, in ? fkey(r + er) : 0xffffffffu);
        const unsigned k1 = __reduce_max_sync(0xffffffffu, in ? fkey(r - er) : 0u);
        const unsigned k2 = __reduce_min_sync(0xffffffffu, in ? fkey(th + et) : 0xffffffffu);
        const unsigned k3 = __reduce_max_sync(0xffffffffu, in ? fkey(th - et) : 0u);
        if (lane == 0) {
          sh.c_cnt[c0] = 1;
          atomicMin(&sh.c_u[c0][0], k0);
          atomicMax(&sh.c_u[c0][1], k1);
          atomicMin(&sh.c_u[c0][2], k2);
          atomicMax(&sh.c_u[c0][3], k3);
        }
      });
    });
    __syncthreads();
    // the same narrowing passes as for the r ranges.  Angles: the points that
    // the FP32 pass leaves are compared by the sine of their angle from the
    // FP32 extreme's direction X, cross(X, z) / |z| with z in double-float
    // (it differs by a few 1e-6 at most, so the sine keeps 1e-13)
    const bool refine = has_plo && !sh.full;
    if (refine) {
      for (int i = tid; i < sh.ncell * 2; i += NT) {
        float sn_, cs_;
        sincosf(fkey_inv(sh.c_u[i >> 1][2 + (i & 1)]), &sn_, &cs_);
        sh.c_ref[i >> 1][i & 1] = make_float2(cs_, sn_);
      }
      __syncthreads();
    }
    auto sine_from = [&](int ps, int c, int k, float* err) -> float {
      const float r = r32[ps];
      if (meta[ps] & M_EXACT) {
        *err = 4e-13f;
        return sine_from64(sh.c_ref[c][k], pt[pidx[ps]]);
      }
      const float2 X = sh.c_ref[c][k];
      const df zx = df_add(df_make(phi[ps].x, plo[ps].x), sh.adf_ll[0]);
      const df zy = df_add(df_make(phi[ps].y, plo[ps].y), sh.adf_ll[1]);
      const df cr = df_sub(df_mul(df_make(X.x, 0.f), zy), df_mul(df_make(X.y, 0.f), zx));
      const float s_ = (cr.hi + cr.lo) / r;
      *err = 1.01f * e32[ps] / r + 4e-13f + 4e-7f * fabsf(s_);
      return s_;
    };
    // FP32 extents of a point's cell below tiny: its decisions stay in FP32
    auto tiny_cell = [&](int c, float r) -> bool {
      return fkey_inv(sh.c_u[c][1]) - fkey_inv(sh.c_u[c][0]) < tiny &&
             (fkey_inv(sh.c_u[c][3]) - fkey_inv(sh.c_u[c][2])) * r < tiny;
    };
    for (int ps = tid; ps < NP; ps += NT) {
      if (!(meta[ps] & M_VALID)) continue;
      const int c = cell_of(ps);
      const float r = r32[ps], th = unwrap_f(ps);
      float er, et;
      er_et(ps, &er, &et);
      if (fkey(r - er) <= sh.c_u[c][0] || fkey(r + er) >= sh.c_u[c][1]) {
        meta[ps] |= M_CAND;
        float e_;
        const float lo = r_from(ps, fkey_inv(sh.c_u[c][0]), &e_);
        atomicMin(&sh.c_s[c][0], fkey(lo + e_));
        const float hi = r_from(ps, fkey_inv(sh.c_u[c][1]), &e_);
        atomicMax(&sh.c_s[c][1], fkey(hi - e_));
      }
      const bool lo = fkey(th - et) <= sh.c_u[c][2], hi = fkey(th + et) >= sh.c_u[c][3];
      if (lo || hi) {
        meta[ps] |= M_CANDT;
        if (refine && !tiny_cell(c, r)) {
          float e_;
          if (lo) { const float s_ = sine_from(ps, c, 0, &e_); atomicMin(&sh.c_s[c][2], fkey(s_ + e_)); }
          if (hi) { const float s_ = sine_from(ps, c, 1, &e_); atomicMax(&sh.c_s[c][3], fkey(s_ - e_)); }
        }
      }
    }
    __syncthreads();
    for (int ps = tid; ps < NP; ps += NT) {
      const uint8_t m_ = meta[ps];
      if (!(m_ & (M_CAND | M_CANDT))) continue;
      const int c = cell_of(ps);
      const float r = r32[ps];
      const bool is_tiny = tiny_cell(c, r);
      bool cand_r = m_ & M_CAND, cand_t = m_ & M_CANDT;
      if (cand_r) {
        float e_;
        const float lo = r_from(ps, fkey_inv(sh.c_u[c][0]), &e_);
        cand_r = fkey(lo - e_) <= sh.c_s[c][0];
        const float hi = r_from(ps, fkey_inv(sh.c_u[c][1]), &e_);
        cand_r = cand_r || fkey(hi + e_) >= sh.c_s[c][1];
      }
      if (cand_t && refine && !is_tiny) {
        const float th = unwrap_f(ps);
        float er, et, e_;
        er_et(ps, &er, &et);
        cand_t = false;
        if (fkey(th - et) <= sh.c_u[c][2]) { const float s_ = sine_from(ps, c, 0, &e_); cand_t = fkey(s_ - e_) <= sh.c_s[c][2]; }
        if (fkey(th + et) >= sh.c_u[c][3]) { const float s_ = sine_from(ps, c, 1, &e_); cand_t = cand_t || fkey(s_ + e_) >= sh.c_s[c][3]; }
      }
      meta[ps] = (uint8_t)((m_ & ~(M_CAND | M_CANDT)) | (cand_r ? M_CAND : 0) | (cand_t ? M_CANDT : 0));
      // theta extremes need an FP64 angle; r extremes only if the
      // double-float r is uncertain
      const bool need = (cand_t && !sh.full) || ((cand_r || cand_t) && !(e32[ps] <= 1e-11f));
      if (need && !(m_ & M_EXACT) && !is_tiny) q_push(sh, queue, ps);
    }
    run_polish();
    for (int ps = tid; ps < NP; ps += NT) {
      const uint8_t m_ = meta[ps];
      if (!(m_ & (M_CAND | M_CANDT))) continue;
      meta[ps] = (uint8_t)(m_ & ~(M_CAND | M_CANDT));
      int c = cell_of(ps);
      if (m_ & M_CAND) {
        const double r = rv(ps);
        atomicMin(&sh.c_x[c][0], dkey(r));
        atomicMax(&sh.c_x[c][1], dkey(r));
      }
      if (m_ & M_CANDT) {
        const double th = unwrap_t(ps, tv(ps));
        atomicMin(&sh.c_x[c][2], dkey(th));
        atomicMax(&sh.c_x[c][3], dkey(th));
      }
    }
    __syncthreads();
    if (DER) {
      // the point that sets each cell extreme (lowest slot on ties), then
      // the extremes as dual numbers carrying that point's tangents
      for (int ps = tid; ps < NP; ps += NT) {
        if (!(meta[ps] & M_VALID)) continue;
        int c = cell_of(ps);
        if (c >= MAXCELL_D) continue;
        unsigned long long kr = dkey(rv(ps)), kt = dkey(unwrap_t(ps, tv(ps)));
        if (kr == sh.c_x[c][0]) atomicMin(&ds.cell_arg[c][0], ps);
        if (kr == sh.c_x[c][1]) atomicMin(&ds.cell_arg[c][1], ps);
        if (kt == sh.c_x[c][2]) atomicMin(&ds.cell_arg[c][2], ps);
        if (kt == sh.c_x[c][3]) atomicMin(&ds.cell_arg[c][3], ps);
      }
      __syncthreads();
      const int nd = min(sh.ncell, MAXCELL_D) * 4;
      for (int idx = tid; idx < nd; idx += NT) {
        const int c = idx >> 2, k = idx & 3;
        DualD v = dconst(dkey_inv(sh.c_x[c][k]));
        const int ps = ds.cell_arg[c][k];
        if (sh.c_cnt[c] && ps < NP) {
          const int kl = ps / N;
          cd u = mk((double)ulimb[kl].x.hi + (double)ulimb[kl].x.lo, (double)ulimb[kl].y.hi + (double)ulimb[kl].y.lo);
          // tangents at the FP64 position (the value stays the extreme the
          // sectors were built from)
          double r_ = rv(ps), t_ = tv(ps);
          if (!(meta[ps] & M_EXACT)) {
            cd z0 = tod(phi[ps]);
            if (has_plo) z0 = z0 + tod(plo[ps]);
            polish_image64<NL>(sh, z0 + sh.L.a[ll], limb_point64(sh, kl, K), &r_, &t_);
          }
          double dr_[NPAR], dt_[NPAR];
          point_tangents(sh, ds, r_, t_, u, dr_, dt_);
          for (int q = 0; q < NPAR; ++q) v.d[q] = k < 2 ? dr_[q] : dt_[q];
        }
        cdual[idx] = v;
      }
      __syncthreads();
    }

    if (diag_cnt && tid == 0) { long long c_ = clock64(); sh.cnt[10] = (int)min(c_ - sh.clk0, 2000000000LL); sh.clk0 = c_; }
    // ------------------------------------------------ 8. sectors (FP64, one thread)
    if (tid == 0 && !DER) {
      int nb = 0;
      for (int T = 0; T < nT; ++T) {
        int c0 = sh.cellbase[T], c1 = sh.cellbase[T + 1];
        for (int c = c0; c < c1 && c < MAXCELL; ++c) {
          if (!sh.c_cnt[c]) continue;
          Box B = cell_box<double>(dkey_inv(sh.c_x[c][0]), dkey_inv(sh.c_x[c][1]), dkey_inv(sh.c_x[c][2]),
                                   dkey_inv(sh.c_x[c][3]), g.margin, sh.full != 0, sh.origin_in && c == c0);
          if (nb < MAXBOX) sh.box[nb++] = B;
          else sh.status |= ICRS_ST_OVERFLOW;
        }
      }
      bool capped = false;
      nb = merge_boxes<double>(sh.box, nb, N, &capped);
      if (capped) sh.status |= ICRS_ST_SECTCAP;
      sh.nbox = nb;
    }
    if (tid == 0 && DER) {
      // the same rules on dual numbers: the sector bounds and their tangents
      int nb = 0;
      for (int T = 0; T < nT; ++T) {
        int c0 = sh.cellbase[T], c1 = sh.cellbase[T + 1];
        for (int c = c0; c < c1 && c < MAXCELL; ++c) {
          if (!sh.c_cnt[c]) continue;
          if (c >= MAXCELL_D || nb >= MAXBOX_D) { sh.status |= ICRS_ST_OVERFLOW; continue; }
          bdual[nb++] = cell_box<DualD>(cdual[c * 4 + 0], cdual[c * 4 + 1], cdual[c * 4 + 2], cdual[c * 4 + 3],
                                        g.margin, sh.full != 0, sh.origin_in && c == c0);
        }
      }
      bool capped = false;
      nb = merge_boxes<DualD>(bdual, nb, N, &capped);
      if (capped) sh.status |= ICRS_ST_SECTCAP;
      for (int b = 0; b < nb; ++b) {
        sh.box[b].r_lo = bdual[b].r_lo.v;
        sh.box[b].r_hi = bdual[b].r_hi.v;
        sh.box[b].th_lo = bdual[b].th_lo.v;
        sh.box[b].width = bdual[b].width.v;
        sh.box[b].periodic = bdual[b].periodic;
      }
      sh.nbox = nb;
    }
    __syncthreads();

    if (diag_cnt && tid == 0) { long long c_ = clock64(); sh.cnt[11] = (int)min(c_ - sh.clk0, 2000000000LL); sh.clk0 = c_; }
    // ------------------------------------------------ 9. rays
    double raysum = 0.0;  // this thread's share
    if constexpr (!DER) {
      raysum = ray_stage<NL, LAW>(sh, rays_sh);
    } else {
      raysum = der_stage(sh, rays_sh, der_sh);
      der_sums(rays_sh, der_sh, sh.nbox, ds.Gb, ds.H);
    }
    if (diag_cnt && tid == 0) { long long c_ = clock64(); sh.cnt[12] = (int)min(c_ - sh.clk0, 2000000000LL); sh.clk0 = c_; }
    // ------------------------------------------------ 10. reduction
    double v = raysum;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) sh.red[warp] = v;
    __syncthreads();
    if (warp == 0) {
      double tot = lane < NW ? sh.red[lane] : 0.0;
      for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
      // unspotted normalisation A0 = S / rho^2; a spot divides by the
      // unlensed flux 1 - c F_spot (N = spot_norm); an invalid spot gives NaN
      const double A0 = tot / (sh.rho * sh.rho);
      double A = A0 * sh.spot_norm;
      if (LAW != 0 && sh.spot_bad) A = __longlong_as_double(0x7ff8000000000000LL);
      bool nan_ = !(A == A) || isinf(A);
      size_t o = (size_t)s * E + e;
      if (DER) {
        // dA/dp = (sum_b G_b . d bounds_b/dp + H . d(w_c, rho, u1, a, eps)/dp) / rho^2
        //         - 2 S / rho^3 [p = rho], one parameter per lane
        const int q = lane & 7;
        double dS = 0.0;
        for (int b = 0; b < sh.nbox; ++b)
          dS += ds.Gb[b][0] * bdual[b].r_lo.d[q] + ds.Gb[b][1] * bdual[b].r_hi.d[q] +
                ds.Gb[b][2] * bdual[b].th_lo.d[q] + ds.Gb[b][3] * bdual[b].width.d[q];
        if (q < 4) dS += ds.H[0] * ds.dwc[q].x + ds.H[1] * ds.dwc[q].y;
        else if (q == 4) dS += ds.H[4] * ds.dadp[0][0] + ds.H[5] * ds.dadp[1][0];
        else if (q == 5)
          dS += ds.H[4] * ds.dadp[0][1] + ds.H[5] * ds.dadp[1][1] + ds.H[6] * ds.depsq[0] + ds.H[7] * ds.depsq[1];
        else if (q == 6) dS += ds.H[2];
        else dS += ds.H[3];
        double dA = dS * (1.0 / (sh.rho * sh.rho));
        if (q == 6) dA -= 2.0 * A0 / sh.rho;
        // the spot's normalisation: dA = N dA0 + A0 dN, dN/du1 = N^2 c dF/du1
        dA *= sh.spot_norm;
        if (q == 7) dA += A * sh.spot_gu;
        nan_ = __any_sync(0xffffffffu, nan_ || !(dA == dA) || isinf(dA));
        if (lane < NPAR) {
          if (dout.dA) dout.dA[o * NPAR + q] = dA;
          double wgt = 0.0;
          if (dout.gA) wgt = dout.gA[o];
          if (dout.yobs) {
            // chi^2 = sum_e ((y_e - A_e) / sigma_e)^2 with the flux F = A
            const double r_ = (dout.yobs[o] - A) / dout.sig[o];
            wgt = -2.0 * r_ / dout.sig[o];
            if (dout.chi2 && lane == 0) atomicAdd(&dout.chi2[s], r_ * r_);
          }
          if (dout.grad) atomicAdd(&dout.grad[(size_t)s * NPAR + q], wgt * dA);
        }
      }
      if (nan_ && lane == 0) sh.status |= ICRS_ST_NAN;
      if (lane == 0) {
      if (A_out) A_out[o] = A;
      if (st_out) st_out[o] = (sh.status & 0xffu) | ((uint32_t)min(sh.nbox, 255) << 8);
      if (diag_cnt)
        for (int c = 0; c < 16; ++c) diag_cnt[o * 16 + c] = sh.cnt[c];
      if (diag_sect)
        for (int b = 0; b < 10; ++b) {
          double* d = diag_sect + (o * 10 + b) * 5;
          if (b < sh.nbox) { d[0] = sh.box[b].r_lo; d[1] = sh.box[b].r_hi; d[2] = sh.box[b].th_lo; d[3] = sh.box[b].width; d[4] = sh.box[b].periodic; }
          else { d[0] = d[1] = d[2] = d[3] = d[4] = 0.0; }
        }
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------- point source
// One thread per source position: images and magnification of a point source
// (point_source_solve, shared with the surrogate's feature kernel).
template <int NL>
__global__ void point_source_kernel(const icrs_params* __restrict__ P, int S, const double* __restrict__ W, int n,
                                    icrs_grid g, double* __restrict__ A, double* __restrict__ images,
                                    int32_t* __restrict__ n_img, uint32_t* __restrict__ status) {
  constexpr int N = NL * NL + 1;
  long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)S * n) return;
  const int s = (int)(idx / n);
  PsLens<NL> L;
  ps_lens<NL>(make_lens(P[s]), L);
  const cd w = mk(W[2 * idx], W[2 * idx + 1]);
  const PointSource<NL> r = point_source_solve<NL>(L, w, g.max_iter, g.img_tol, images ? images + idx * N * 2 : nullptr);
  A[idx] = r.A;
  if (n_img) n_img[idx] = r.m;
  if (status) status[idx] = r.st;
}

// ---------------------------------------------------------------- likelihood
// Linear-flux marginalised NLL of one light curve per block (Appendix B,
// Eq. NLL, Woodbury form), and optionally its gradient sum_e dnll/dA_e dA_e/dp
// from the per-epoch derivatives dA [S][E][8].  Fixed-order FP64 sums.
constexpr int NLL_THREADS = 256;

__device__ inline double block_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double s = 0.0;
  for (int w = 0; w < NLL_THREADS / 32; ++w) s += red[w];
  return s;
}

__global__ void __launch_bounds__(NLL_THREADS)
marginal_nll_kernel(const double* __restrict__ A, const double* __restrict__ F, const double* __restrict__ sig,
                    const double* __restrict__ prior, int E, const double* __restrict__ dA,
                    double* __restrict__ nll, double* __restrict__ grad, double* __restrict__ fluxes) {
  __shared__ double red[NLL_THREADS / 32];
  const int s = blockIdx.x;
  const size_t o = (size_t)s * E;
  const double mu0 = prior[4 * s + 0], mu1 = prior[4 * s + 1];
  const double l0 = prior[4 * s + 2], l1 = prior[4 * s + 3];
  // sums over the epochs: M^T C^-1 M, M^T C^-1 r, r^T C^-1 r, ln|C|
  // (r = F - M mu, m_e = (A_e - 1, 1), c_e = 1 / sigma_e^2)
  double saa = 0, sa1 = 0, s11 = 0, sar = 0, s1r = 0, srr = 0, slc = 0, nbad = 0;
  for (int e = threadIdx.x; e < E; e += NLL_THREADS) {
    const double a = A[o + e] - 1.0, sg = sig[o + e];
    const double c = 1.0 / (sg * sg);
    const double r = F[o + e] - mu0 * a - mu1;
    saa += c * a * a; sa1 += c * a; s11 += c;
    sar += c * a * r; s1r += c * r; srr += c * r * r;
    slc += log(sg * sg);
    if (!(sg > 0.0)) nbad += 1.0;
  }
  saa = block_sum(saa, red); sa1 = block_sum(sa1, red); s11 = block_sum(s11, red);
  sar = block_sum(sar, red); s1r = block_sum(s1r, red); srr = block_sum(srr, red);
  slc = block_sum(slc, red); nbad = block_sum(nbad, red);
  // K = Lambda^-1 + M^T C^-1 M and its inverse
  const double k00 = 1.0 / l0 + saa, k01 = sa1, k11 = 1.0 / l1 + s11;
  const double det = k00 * k11 - k01 * k01;
  const double i00 = k11 / det, i01 = -k01 / det, i11 = k00 / det;
  const double kv0 = i00 * sar + i01 * s1r, kv1 = i01 * sar + i11 * s1r;  // K^-1 v
  const double a0 = mu0 + kv0, a1 = mu1 + kv1;                              // posterior mean
  const bool bad = nbad > 0.0 || !(l0 > 0.0) || !(l1 > 0.0) || !(det > 0.0);
  if (threadIdx.x == 0) {
    const double quad = srr - (sar * kv0 + s1r * kv1);
    const double logdet = slc + log(l0) + log(l1) + log(det);
    nll[s] = bad ? __longlong_as_double(0x7ff8000000000000LL) : 0.5 * (quad + logdet);
    if (fluxes) { fluxes[2 * s] = a0; fluxes[2 * s + 1] = a1; }
  }
  if (!grad) return;
  double gq[NPAR];
  for (int q = 0; q < NPAR; ++q) gq[q] = 0.0;
  for (int e = threadIdx.x; e < E; e += NLL_THREADS) {
    const double a = A[o + e] - 1.0, sg = sig[o + e];
    const double c = 1.0 / (sg * sg);
    const double ge = c * ((i00 * a + i01) - (F[o + e] - a * a0 - a1) * a0);
    const double* d = dA + (o + e) * NPAR;
    for (int q = 0; q < NPAR; ++q) gq[q] += ge * d[q];
  }
  for (int q = 0; q < NPAR; ++q) {
    const double v = block_sum(gq[q], red);
    if (threadIdx.x == 0) grad[(size_t)s * NPAR + q] = v;
  }
}

// ---------------------------------------------------------------- host side
// Columns of the ray stage's offset tables: every sector of an epoch at once
// (forward), about three (derivative, where shared memory is shorter).
static int mag_tabcap(int NL, bool der) { return (der ? 3 : NL * NL + 1) * (GTH_MAX + 2); }

static size_t mag_smem_bytes(int NL, const icrs_grid& g, int pmax, int has_plo, bool der, int nt, int ccap, int tcap) {
  const int N = NL * NL + 1;
  const size_t NP = (size_t)g.n_limb * N;
  size_t b = sizeof(cf) * NP * (has_plo ? 2 : 1) + sizeof(cdf) * g.n_limb + 16;
  if (der) b += sizeof(DerShared);               // derivative state
  // image-limb slots; the ray stage's tables take their place
  size_t slots = 4 * sizeof(float) * NP + sizeof(short) * ((NP + 7) & ~(size_t)7) + 3 * ((NP + 15) & ~(size_t)15);
  slots += 2 * sizeof(double) * pmax + sizeof(int) * QMAX;
  const size_t rays = sizeof(cf) * mag_tabcap(NL, der) + (sizeof(AnchorF) + sizeof(float2)) * MAXANCH +
                      (der ? sizeof(int) * (nt / 32) * DQ + der_rays_bytes(nt / 32) : sizeof(int2) * (nt / 32) * FQ) +
                      sizeof(double2) * ccap + (size_t)tcap * (sizeof(float) * (32 + PCAP) + sizeof(int));
  return b + (slots > rays ? slots : rays);
}

static int check_grid(const icrs_grid* g) {
  if (!g) return ICRS_EINVAL;
  if (g->n_r < 1 || g->n_r > 4096) return ICRS_EINVAL;
  if (g->n_theta < 8 || g->n_theta > 8192) return ICRS_EINVAL;
  if (g->n_limb < 16 || g->n_limb > 1024) return ICRS_EINVAL;
  if (g->n_bins_r < 2 || g->n_bins_r > MAXRB) return ICRS_EINVAL;
  if (g->n_bins_theta < 2 || g->n_bins_theta > 128) return ICRS_EINVAL;
  if (!(g->delta_c > 0.0) || !(g->margin >= 0.0) || !(g->img_tol > 0.0)) return ICRS_EINVAL;
  if (g->max_iter < 1 || g->max_iter > 10000) return ICRS_EINVAL;
  if (g->ld_split != 0 && g->ld_split != 1) return ICRS_EINVAL;
  if (g->grad_rule != 0 && g->grad_rule != 1) return ICRS_EINVAL;
  if (g->grad_rule && !(g->s_fac > 0.0)) return ICRS_EINVAL;
  return ICRS_OK;
}

// Reads n_lens of the first parameter set from the device (the ABI requires
// all sets of one call to share it).
static int first_n_lens(const icrs_params* p, cudaStream_t st, int* nl) {
  int32_t v = 0;
  cudaError_t e = cudaMemcpyAsync(&v, (const char*)p + offsetof(icrs_params, n_lens), sizeof(int32_t),
                                  cudaMemcpyDeviceToHost, st);
  if (e != cudaSuccess) return ICRS_ECUDA;
  e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return ICRS_ECUDA;
  if (v != 2 && v != 3) return ICRS_EINVAL;
  *nl = v;
  return ICRS_OK;
}

// Launch of one instantiation at NTB threads per block, with its shared
// memory, point-table size and flags already chosen: occupancy, contiguous
// chunks of epochs per block (warm starts along the light curve).
template <int NL, bool DER, int NTB, int LAW>
static int launch_nt(const icrs_params* p, int S, const double* t, int E, const icrs_grid* g, double* A,
                     uint32_t* status, double* dsect, int32_t* dcnt, float* dpts, const DerOut& dout,
                     cudaStream_t st, const int32_t* items, int n_items, int nsm, size_t smem, int pmax,
                     int has_plo, int ccap, int tcap) {
  if (cudaFuncSetAttribute(mag_kernel<NL, DER, NTB, LAW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
      cudaSuccess)
    return ICRS_ECUDA;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, mag_kernel<NL, DER, NTB, LAW>, NTB, smem) != cudaSuccess)
    return ICRS_ECUDA;
  if (per_sm < 1) return ICRS_EUNSUPPORTED;
  long long tiles = items ? (long long)n_items : (long long)S * E;
  long long slots = (long long)nsm * per_sm;
  long long per_block = (tiles + slots - 1) / slots;
  if (per_block < 1) per_block = 1;
  long long blocks = (tiles + per_block - 1) / per_block;
  mag_kernel<NL, DER, NTB, LAW><<<(unsigned)blocks, NTB, smem, st>>>(p, S, t, E, *g, (int)per_block, A, status,
                                                                      dsect, dcnt, dpts, pmax, has_plo,
                                                                      mag_tabcap(NL, DER), ccap, tcap, dout, items, n_items);
  return cudaGetLastError() == cudaSuccess ? ICRS_OK : ICRS_ECUDA;
}

// Shared-memory sizing of one (NL, DER) launch: forward, the FP64 point table
// grows (up to one entry per image-limb slot) before the lo parts of image
// positions are added; derivative mode takes the lo parts first (fewer FP64
// polishes).
template <int NL, bool DER, int LAW>
static int launch_inst(const icrs_params* p, int S, const double* t, int E, const icrs_grid* g, double* A,
                       uint32_t* status, double* dsect, int32_t* dcnt, float* dpts, const DerOut& dout,
                       cudaStream_t st, const int32_t* items = nullptr, int n_items = 0) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return ICRS_ECUDA;
  int optin = 0, nsm = 0;
  if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) return ICRS_ECUDA;
  if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return ICRS_ECUDA;
  // shared memory beside the dynamic part
  cudaFuncAttributes fa;
  if (cudaFuncGetAttributes(&fa, mag_kernel<NL, DER, NT_BASE, LAW>) != cudaSuccess) return ICRS_ECUDA;
  // forward: the tasks of one sector at least, of as many as fit once the rest
  // is chosen
  const int nt1 = DER ? 0 : sector_tasks(g->n_r, g->n_theta);
  int tcap = nt1;
  auto fits = [&](int pm, int plo) {
    return mag_smem_bytes(NL, *g, pm, plo, DER, NT_BASE, 0, tcap) + fa.sharedSizeBytes <= (size_t)optin;
  };
  int pmax = PMAX_MIN;
  if (!fits(pmax, 0)) return ICRS_EUNSUPPORTED;
  int has_plo = (DER && fits(pmax, 1)) ? 1 : 0;
  const int np_all = g->n_limb * (NL * NL + 1);
  // the FP64 point table takes the remaining room (16 bytes per entry), up to
  // one entry per image-limb slot
  pmax = np_all < PMAX_MIN ? PMAX_MIN : np_all;
  while (pmax > PMAX_MIN && !fits(pmax, has_plo)) pmax = pmax - 64 > PMAX_MIN ? pmax - 64 : PMAX_MIN;
  if (!DER) has_plo = fits(pmax, 1) ? 1 : 0;
  // derivative: the cosine table of the columns, for all sectors at once or as
  // many as fit
  int ccap = 0;
  if (DER)
    for (int k = NL * NL + 1; k > 0 && !ccap; --k)
      if (mag_smem_bytes(NL, *g, pmax, has_plo, DER, NT_BASE, k * g->n_theta, 0) + fa.sharedSizeBytes <= (size_t)optin)
        ccap = k * g->n_theta;
  for (int k = NL * NL + 1; k > 1 && !DER && tcap == nt1; --k) {
    tcap = k * nt1;
    if (!fits(pmax, has_plo)) tcap = nt1;
  }
  const size_t smem = mag_smem_bytes(NL, *g, pmax, has_plo, DER, NT_BASE, ccap, tcap);
  return launch_nt<NL, DER, NT_BASE, LAW>(p, S, t, E, g, A, status, dsect, dcnt, dpts, dout, st, items, n_items, nsm,
                                          smem, pmax, has_plo, ccap, tcap);
}

// Binary forward: the linear instantiation, then the generic one (each takes
// its own sets and skips the others; same stream, so they run in order).
static int launch_binary_fwd(const icrs_params* p, int S, const double* t, int E, const icrs_grid* g, double* A,
                             uint32_t* status, double* dsect, int32_t* dcnt, float* dpts, cudaStream_t st,
                             const int32_t* items = nullptr, int n_items = 0) {
  DerOut none = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
  int rc = launch_inst<2, false, 0>(p, S, t, E, g, A, status, dsect, dcnt, dpts, none, st, items, n_items);
  if (rc) return rc;
  return launch_inst<2, false, 1>(p, S, t, E, g, A, status, dsect, dcnt, dpts, none, st, items, n_items);
}

static int launch_mag(const icrs_params* p, int S, const double* t, int E, const icrs_grid* g,
                      double* A, uint32_t* status, double* dsect, int32_t* dcnt, float* dpts, void* stream) {
  if (S < 0 || E < 0) return ICRS_EINVAL;
  if (S == 0 || E == 0) return check_grid(g);
  if (!p || !t || !A) return ICRS_EINVAL;
  int rc = check_grid(g);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  int nl = g->n_lens;
  if (nl == 0) { rc = first_n_lens(p, st, &nl); if (rc) return rc; }
  if (nl != 2 && nl != 3) return ICRS_EINVAL;
  DerOut none = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
  if (nl == 2) return launch_binary_fwd(p, S, t, E, g, A, status, dsect, dcnt, dpts, st);
  return launch_inst<3, false, 2>(p, S, t, E, g, A, status, dsect, dcnt, dpts, none, st);
}

// Derivative launch (binary lens only): zeroes the accumulated outputs on the
// stream, then runs the derivative instantiation.
static int launch_der(const icrs_params* p, int S, const double* t, int E, const icrs_grid* g, DerOut d,
                      double* A, uint32_t* status, void* stream) {
  if (S < 0 || E < 0) return ICRS_EINVAL;
  int rc = check_grid(g);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  if (S > 0) {
    if (d.grad && cudaMemsetAsync(d.grad, 0, sizeof(double) * NPAR * (size_t)S, st) != cudaSuccess) return ICRS_ECUDA;
    if (d.chi2 && cudaMemsetAsync(d.chi2, 0, sizeof(double) * (size_t)S, st) != cudaSuccess) return ICRS_ECUDA;
  }
  if (S == 0 || E == 0) return ICRS_OK;
  if (!p || !t) return ICRS_EINVAL;
  int nl = g->n_lens;
  if (nl == 0) { rc = first_n_lens(p, st, &nl); if (rc) return rc; }
  if (nl == 3 || g->ld_split) return ICRS_EUNSUPPORTED;
  if (nl != 2) return ICRS_EINVAL;
  return launch_inst<2, true, 2>(p, S, t, E, g, A, status, nullptr, nullptr, nullptr, d, st);
}

}  // namespace icrs

using namespace icrs;

extern "C" {

int icrs_abi_version(void) { return 3; }

void icrs_grid_default(icrs_grid* g) {
  if (!g) return;
  memset(g, 0, sizeof(*g));
  g->n_r = 64; g->n_theta = 256; g->n_limb = 500;
  g->n_bins_r = 32; g->n_bins_theta = 128; g->max_iter = 100; g->uniform = 0;
  g->n_lens = 2;
  g->delta_c = 0.02; g->margin = 0.05; g->img_tol = 1e-3;
  g->s_fac = 100.0;
}

const char* icrs_strerror(int code) {
  switch (code) {
    case ICRS_OK: return "ok";
    case ICRS_EINVAL: return "invalid argument";
    case ICRS_ECUDA: return "CUDA runtime error";
    case ICRS_ETIMEOUT: return "device wait timed out";
    case ICRS_EUNSUPPORTED: return "unsupported configuration (shared memory or sizes)";
    default: return "unknown error";
  }
}

int icrs_point_source(const icrs_params* p, int S, const double* w, int n, const icrs_grid* g,
                      double* A, double* images, int32_t* n_img, uint32_t* status, void* stream) {
  if (S < 0 || n < 0) return ICRS_EINVAL;
  if (S == 0 || n == 0) return check_grid(g);
  if (!p || !w || !A) return ICRS_EINVAL;
  int rc = check_grid(g);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  int nl = g->n_lens;
  if (nl == 0) { rc = first_n_lens(p, st, &nl); if (rc) return rc; }
  if (nl != 2 && nl != 3) return ICRS_EINVAL;
  long long total = (long long)S * n;
  int threads = 128;
  long long blocks = (total + threads - 1) / threads;
  if (blocks > 2147483647LL) return ICRS_EUNSUPPORTED;
  if (nl == 2) point_source_kernel<2><<<(unsigned)blocks, threads, 0, st>>>(p, S, w, n, *g, A, images, n_img, status);
  else point_source_kernel<3><<<(unsigned)blocks, threads, 0, st>>>(p, S, w, n, *g, A, images, n_img, status);
  return cudaGetLastError() == cudaSuccess ? ICRS_OK : ICRS_ECUDA;
}

int icrs_magnification(const icrs_params* p, int S, const double* t, int E, const icrs_grid* g,
                       double* A, uint32_t* status, void* stream) {
  return launch_mag(p, S, t, E, g, A, status, nullptr, nullptr, nullptr, stream);
}

int icrs_magnification_diag(const icrs_params* p, int S, const double* t, int E, const icrs_grid* g,
                            double* A, uint32_t* status, double* sectors, int32_t* counters,
                            float* points, void* stream) {
  return launch_mag(p, S, t, E, g, A, status, sectors, counters, points, stream);
}

size_t icrs_marginal_nll_workspace_bytes(int S, int E) {
  if (S <= 0 || E <= 0) return 0;
  return sizeof(double) * (size_t)S * (size_t)E * (NPAR + 1);
}

int icrs_marginal_nll_grad(const icrs_params* p, int S, const double* t, int E, const icrs_grid* g, const double* F,
                           const double* sigma, const double* prior, double* nll, double* grad, double* fluxes,
                           double* A, uint32_t* status, void* workspace, size_t workspace_bytes, void* stream) {
  if (S < 0 || E < 0) return ICRS_EINVAL;
  int rc = check_grid(g);
  if (rc) return rc;
  if (S == 0) return ICRS_OK;
  if (!p || !prior || !nll || (E > 0 && (!t || !F || !sigma))) return ICRS_EINVAL;
  const size_t need = icrs_marginal_nll_workspace_bytes(S, E);
  if (E > 0 && (!workspace || workspace_bytes < need || ((uintptr_t)workspace & 7u))) return ICRS_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  double* dA = (double*)workspace;
  double* Aw = A ? A : (E > 0 ? dA + (size_t)S * E * NPAR : nullptr);
  if (E > 0) {
    if (grad) {
      DerOut d = {nullptr, nullptr, nullptr, dA, nullptr, nullptr};
      rc = launch_der(p, S, t, E, g, d, Aw, status, stream);
    } else {
      rc = launch_mag(p, S, t, E, g, Aw, status, nullptr, nullptr, nullptr, stream);
    }
    if (rc) return rc;
  }
  marginal_nll_kernel<<<S, NLL_THREADS, 0, st>>>(Aw, F, sigma, prior, E, dA, nll, grad, fluxes);
  return cudaGetLastError() == cudaSuccess ? ICRS_OK : ICRS_ECUDA;
}

int icrs_magnification_indexed(const icrs_params* p, int S, const double* t, int E, const int32_t* items, int n,
                               const icrs_grid* g, double* A, uint32_t* status, void* stream) {
  if (S < 0 || E < 0 || n < 0) return ICRS_EINVAL;
  int rc = check_grid(g);
  if (rc) return rc;
  if (S == 0 || E == 0 || n == 0) return ICRS_OK;
  if (!p || !t || !items || !A) return ICRS_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  int nl = g->n_lens;
  if (nl == 0) { rc = first_n_lens(p, st, &nl); if (rc) return rc; }
  if (nl != 2 && nl != 3) return ICRS_EINVAL;
  DerOut none = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
  if (nl == 2) return launch_binary_fwd(p, S, t, E, g, A, status, nullptr, nullptr, nullptr, st, items, n);
  return launch_inst<3, false, 2>(p, S, t, E, g, A, status, nullptr, nullptr, nullptr, none, st, items, n);
}

int icrs_magnification_vjp(const icrs_params* p, int S, const double* t, int E, const icrs_grid* g,
                           const double* gA, double* grad, double* dA, double* A, uint32_t* status, void* stream) {
  if (S > 0 && E > 0 && !gA && grad) return ICRS_EINVAL;
  if (S > 0 && !grad && !dA) return ICRS_EINVAL;
  DerOut d = {gA, nullptr, nullptr, dA, grad, nullptr};
  return launch_der(p, S, t, E, g, d, A, status, stream);
}

int icrs_chi2_grad(const icrs_params* p, int S, const double* t, int E, const icrs_grid* g, const double* y,
                   const double* sigma, double* chi2, double* grad, double* A, uint32_t* status, void* stream) {
  if (S > 0 && E > 0 && (!y || !sigma)) return ICRS_EINVAL;
  if (S > 0 && (!chi2 || !grad)) return ICRS_EINVAL;
  DerOut d = {nullptr, y, sigma, nullptr, grad, chi2};
  return launch_der(p, S, t, E, g, d, A, status, stream);
}

}  // extern "C"
