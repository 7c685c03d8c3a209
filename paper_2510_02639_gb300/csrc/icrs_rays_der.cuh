// Derivative ray stage (binary lens): the rays of all sectors of one epoch,
// their value and, in reverse mode, its derivative with respect to the sector
// bounds and to (w_c, rho, u1, a_j, eps_j).
//
// The sweep is the forward stage's, one column at a time: every inside ray
// has a seed a = dRow/dd and adds a times the gradient of its distance d to
// its lane's FP32 sums over the task's columns.  Superblocks that lie outside
// the source on all 32 rows are skipped, those inside need no decisions (as in
// icrs_rays.cuh, with the same bits).
//
// Two things bounded the earlier form of this stage, both of them FP64 (one
// FP64 instruction occupies the SM for 16 cycles):
//   * the boundary points' stencil distances, five FP64 rays each, about 300
//     instructions a ray.  A crossing's slope is a difference of nearly equal
//     distances, so they stay FP64 (in double-float about the anchors the
//     gradient moved by 1e-8: the crossings are rounded to FP32 before f' and
//     the basis, which shows), but the columns' sines and cosines, more than
//     half of that, come from a table formed once per sector;
//   * a warp reduction of twelve FP64 row terms per task.  The rows' terms
//     are now added, still in FP64, to a column of sums per lane in shared
//     memory, and reduced once per sector.
// What bounds it now: at 64 x 256 the FP64 flush and the tangents, at 1024 x
// 2048 the sweep's issue rate (196 instructions a ray in which a gradient is
// formed, FMA pipe 42 % busy) and the wait for the slowest warp.  chi^2 and its
// gradient, 32 sets of 500 epochs at 64 x 256: 80.4 ms before, 44.0 now; 8 sets
// of 250 at 1024 x 2048: 99.1 ms and 67.2.
#pragma once

#include "icrs_rays.cuh"

namespace icrs {

constexpr int DSUM = 15;  // sums per lane, see row_add

struct DerRays {
  float2* acs;       // cos, sin of each anchor angle
  float4* aA;        // A_0, A_1 of each anchor (FP32)
  double* sums;      // [warp][DSUM][32], lane i of sum k at (i + k) & 31
  double* wsum;      // [sector][DSUM][warp]
  double2* ctab;     // cosine and sine of the batch's columns, or NULL (no room)

  __device__ void store(int an, const AnchorX<2>& x) const {
    acs[an] = make_float2((float)x.cs, (float)x.sn);
    aA[an] = make_float4((float)x.A[0].x, (float)x.A[0].y, (float)x.A[1].x, (float)x.A[1].y);
  }

  // cosines and sines of the columns of sectors b0 .. b1 - 1
  __device__ void columns(const RayShared& rs, int b0, int b1) const {
    if (!ctab) return;
    const int NTH = rs.P.NTH, n = (b1 - b0) * NTH;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const Sec& S = rs.sec[b0 + i / NTH];
      const int l = i % NTH;
      double c, sn;
      sincos(S.th_lo + (l + 0.5) * S.dth64, &sn, &c);
      ctab[i] = make_double2(c, sn);
    }
  }
};
// Shared memory of these tables (bytes), for nw warps.
constexpr size_t der_rays_bytes(int nw) {
  return MAXANCH * (sizeof(float2) + sizeof(float4)) + sizeof(double) * nw * DSUM * 32 +
         sizeof(double) * 5 * DSUM * TASK_WARPS;
}

// FP64 distance of a ray from the source centre, (c, sn) its column's cosine
// and sine.
__device__ __noinline__ double ray_distance_cs(const double* eps, const cd* a, cd wc, double r, double c, double sn) {
  const cd z = mk(r * c, r * sn);
  return sqrt(abs2(lens_map<2, double>(eps, a, z) - wc));
}

// A row's sums v (v[0] = sum of I W, v[1 + k] = pg[k]) into the lane's column
// of sums; S_b = sum_i K_i Row_i, K_i = r_i dr dth, r_i = r_lo + (i + 1/2) dr,
// dr = (r_hi - r_lo) / N_r, dth = width / N_theta, so that the derivatives of
// S_b with respect to the bounds and the rest (bounds_of) are combinations of
//   sum Row, sum Row (i + 1/2), sum Row r_i, sum r_i v1, sum r_i v1 (i + 1/2),
//   sum r_i v2, sum r_i v3, sum r_i v4 .. sum r_i v11.
// (The products of two floats are exact in FP64, so each addition rounds once.)
struct RowTerms { float v[12]; };
__device__ __forceinline__ void row_add(double* sums, int lane, int irow, float r, const RowTerms& t) {
  auto add = [&](int k, double a, double b) {
    double* const s = sums + k * 32 + ((lane + k) & 31);
    *s = fma(a, b, *s);
  };
  const double h = irow + 0.5, rd = (double)r, v0 = (double)t.v[0], v1 = (double)t.v[1];
  add(0, v0, 1.0);
  add(1, v0, h);
  add(2, v0, rd);
  add(3, v1, rd);
  add(4, v1 * rd, h);
#pragma unroll
  for (int k = 2; k < 12; ++k) add(3 + k, (double)t.v[k], rd);
}

// What the law and the gradient rule need per ray.
struct DerLaw {
  float c0f, c1f, c2f, I0, irho2, irho, rho32, sfac, eps0, eps1;
  int uniform, gradrule, half;
  float c1h, c3h;
};

// I and dI/dd, dI/drho, dI/du1 at squared distance d2:
//   dI/dx = c1/(2 mu) + c2, dx/dd = -2 d/rho^2, dx/drho = 2 d^2/rho^3,
//   dI/du1 = I (pi/3) I0 - I0 (1 - mu)   (dI0/du1 = (pi/3) I0^2)
// (hc: std::true_type for the generic law: half-integer powers of mu checked
// at run time)
template <class HC>
__device__ __forceinline__ float brightness_der(const DerLaw& w, float d2, float* Id, float* Ir, float* Iu, HC) {
  if (w.uniform) { *Id = 0.f; *Ir = 0.f; *Iu = 0.f; return w.I0; }
  // (hardware reciprocal square roots: 2^-22.9 relative, far inside the
  // derivative's tolerance)
  float x = fmaxf(0.f, 1.0f - d2 * w.irho2);
  const float rs = x > 0.f ? rsqrt_fast(x) : 0.f;  // 1 / mu
  float sx = x * rs;
  float I = w.c0f + w.c1f * sx + w.c2f * x;
  float d = d2 * rsqrt_fast(fmaxf(d2, 1e-37f));
  // k = (dI/dmu) / mu / rho^2
  float k = x > 0.f ? (w.c1f * rs + 2.0f * w.c2f) * w.irho2 : 0.f;
  if constexpr (HC::value) {
    if (w.half && x > 0.f) {
      // s (c1h + c3h mu): dI/dmu = c1h / (2 s) + 1.5 c3h s, s = mu^(1/2)
      const float c1h = w.c1h, c3h = w.c3h;
      const float s_ = sqrtf(sx);
      I += s_ * (c1h + c3h * sx);
      k += (0.5f * c1h / s_ + 1.5f * c3h * s_) * rs * w.irho2;
    }
  }
  *Id = -k * d;
  *Ir = k * d2 * w.irho;
  *Iu = I * (float)(kPi / 3.0) * w.I0 + w.I0 * (sx - 1.0f);
  return I;
}

// Per ray with seed a = dRow/dd (dI/dd inside; the paper's sigmoid rule adds
// its own), the row's sums pg[k] += a dd/dq_k are taken from the ray's FP32
// geometry (rotated frame R = e^{-i th_m}: Q_j = A_j + dz, u = Delta w' / d,
// gamma = sum eps_j / Q_j^2):
//   dd/dz = J u, J = [[1 + g.x, -g.y], [-g.y, 1 - g.x]]
//   dd/dr_i = (J u) . e^{i phi},  dd/dth_l = (J u) . (i z)
//   dd/dw_c = -conj(R) u,  dd/da_j.x = -eps_j Re(conj(u) conj(R) Q_j^2) / |Q_j|^4
//   dd/deps_j = -(u . Q_j) / |Q_j|^2
// pg: sum a dd/dr_i, sum a dd/dth_l, sum a dd/dth_l (l + 1/2), then d/d(w_c.x,
// w_c.y, rho, u1, a1.x, a2.x, eps1, eps2).
__device__ __forceinline__ void grad_core(const DerLaw& w, const cf dz, const cf dw, float tx, float ty, float ri_,
                                          float lwf, const float4 A01, const float2 cs_, float a, float* pgx) {
  const float eps0 = w.eps0, eps1 = w.eps1;
  const cf Q0 = mk(A01.x + dz.x, A01.y + dz.y), Q1 = mk(A01.z + dz.x, A01.w + dz.y);
  const float i0 = rcp_fast(abs2(Q0)), i1 = rcp_fast(abs2(Q1));
  const float id = rsqrt_fast(fmaxf(abs2(dw), 1e-37f));
  const float ux = dw.x * id, uy = dw.y * id;
  const cf q0 = Q0 * Q0, q1 = Q1 * Q1;
  const cf gm = scl(cj(q0), eps0 * i0 * i0) + scl(cj(q1), eps1 * i1 * i1);
  const float gzx = (1.0f + gm.x) * ux - gm.y * uy;
  const float gzy = -gm.y * ux + (1.0f - gm.x) * uy;
  const float ex = 1.0f + tx, ey = ty;
  const float gr_ = gzx * ex + gzy * ey;
  const float gt_ = ri_ * (gzy * ex - gzx * ey);
  pgx[0] += a * gr_;
  pgx[1] += a * gt_;
  pgx[2] += a * gt_ * lwf;
  const float ct = cs_.x, st = cs_.y;
  pgx[3] -= a * (ct * ux - st * uy);
  pgx[4] -= a * (st * ux + ct * uy);
  // conj(R) Q_j^2 with conj(R) = (ct, st)
  const cf P0 = mk(ct, st) * q0, P1 = mk(ct, st) * q1;
  pgx[7] -= a * eps0 * (ux * P0.x + uy * P0.y) * i0 * i0;
  pgx[8] -= a * eps1 * (ux * P1.x + uy * P1.y) * i1 * i1;
  pgx[9] -= a * (ux * Q0.x + uy * Q0.y) * i0;
  pgx[10] -= a * (ux * Q1.x + uy * Q1.y) * i1;
}

// A ray's seed, its value I (inside) into racc and the brightness derivatives
// into pgx[5], pgx[6]; the paper's gradient rule (Sec. 3.5) gives the
// indicator chi = Theta(x), x = (rho - d) / rho, the sigmoid derivative S s (1
// - s), s = 1 / (1 + e^{-S x}), with the interior weight: seed -I S s (1 - s)
// / rho on d and I S s (1 - s) d / rho^2 on rho (tangents only)
// (fs: the ray's spot factor, which scales its brightness)
template <class HC>
__device__ __forceinline__ float seed_of(const DerLaw& w, bool in, float d2, float* pgx, float& racc, HC hc, float fs) {
  float a = 0.f;
  if (in) {
    float Id, Ir, Iu;
    racc += fs * brightness_der(w, d2, &Id, &Ir, &Iu, hc);
    a = fs * Id;
    pgx[5] += fs * Ir;
    pgx[6] += fs * Iu;
  }
  if (w.gradrule) {
    const float dd_ = sqrtf(d2);
    const float sx = w.sfac * (1.0f - dd_ / w.rho32);
    if (fabsf(sx) < 40.0f) {
      const float sg = 1.0f / (1.0f + __expf(-sx));
      const float x = fmaxf(fmaf(-d2, w.irho2, 1.0f), 1e-30f);
      const float mu = x * rsqrtf(x);
      float I = fmaf(w.c2f, x, fmaf(w.c1f, mu, w.c0f));
      if (w.half) I = fmaf(sqrtf(mu), fmaf(w.c3h, mu, w.c1h), I);
      const float c = fs * I * w.sfac * sg * (1.0f - sg);
      a -= c / w.rho32;
      pgx[5] += c * dd_ / (w.rho32 * w.rho32);
    }
  }
  return a;
}

template <class SH>
__device__ __forceinline__ DerLaw der_law(const SH& sh, const RayArgs& P) {
  DerLaw w;
  w.rho32 = (float)sh.rho;
  w.irho2 = 1.0f / (w.rho32 * w.rho32);
  w.irho = 1.0f / w.rho32;
  w.c0f = sh.c0f; w.c1f = sh.c1f; w.c2f = sh.c2f; w.I0 = sh.I0;
  w.sfac = P.sfac;
  w.eps0 = sh.eps32[0]; w.eps1 = sh.eps32[1];
  w.uniform = P.uniform; w.gradrule = P.gradrule; w.half = sh.half;
  w.c1h = sh.c1h; w.c3h = sh.c3h;
  return w;
}

// A lane's sums over a task's columns.
struct RowSums {
  float racc;      // sum of I over the inside rays
  float pg[11];    // sums of the gradients, see grad_core
};

// The undecided rays of a lane's block, as undecided_rays: decided ones' flags
// come back in *bits, the rest in the row's sums.  (These rays lie at the
// limb, where dI/dd grows like 1/mu: they are added to the same FP32 sums, in
// the same order, as before, since their rounding shows.)
template <class SH>
__device__ __noinline__ RowSums der_undecided(SH& sh, const RayShared& rs, const DerRays& dr, int b, int aidx, int gbase,
                                              float ri, float dri, int irow, int l0, int nb, unsigned* bits, RowSums r) {
  const Sec& S = rs.sec[b];
  const AnchorF& an = rs.P.anch[aidx];
  const DerLaw w = der_law(sh, rs.P);
  unsigned out = 0u;
#pragma unroll 1
  for (int k = 0; k < nb; ++k) {
    const cf t = tab_at(rs.P.tabf + 2 * S.tbase, l0 + k - gbase);
    float eb;
    cf dz, dw;
    float d2 = ray_eval<2>(an, t.x, t.y, ri, dri, &eb, &dw, &dz);
    if (d2 < an.lo2 || d2 > an.hi2) continue;
    const bool in = ray_decide<2>(sh, rs, S, d2, eb, irow, l0 + k);
    if (in) out |= 1u << (nb - 1 - k);
    const float fs = in ? spot_factor<2, 2>(sh, rs, S, aidx, dw, eb, irow, l0 + k) : 1.f;
    const float a = seed_of(w, in, d2, r.pg, r.racc, std::true_type{}, fs);
    if (a != 0.f) grad_core(w, dz, dw, t.x, t.y, ri, (float)(l0 + k) + 0.5f, dr.aA[aidx], dr.acs[aidx], a, r.pg);
  }
  *bits = out;
  return r;
}

// n <= 32 queued boundary points, one per lane.  The stencil's flags come from
// the FP32 distances (as in the forward stage), the crossing and its
// derivative from the FP64 ones: the point's value I (W - 1) beyond
// the I that the sweep added, its seed (W - 1) dI/dd, and the crossing seeds
// -I f'(delta) l_m(x) / p'(x) on the stencil rays (p the cubic through the
// stencil distances, x its crossing).
template <class SH>
__device__ __noinline__ float2 der_flush(SH& sh, RayShared& rs, const DerRays& dr, const int* q, int n, float2 acc) {
  const RayArgs& P = rs.P;
  const int lane = threadIdx.x & 31, NTH = P.NTH;
  __syncwarp();
  if (lane < n) {
    const int v_ = q[lane];
    const Sec& S = rs.sec[v_ >> 25];
    const int irow = (v_ >> 13) & 4095, m = v_ & 8191;
    const int gi_ = irow / S.gr;
    const float dri_ = ((float)(irow - gi_ * S.gr) + 0.5f - 0.5f * (float)S.gr) * S.dr32;
    const float ri_ = __fadd_rn(S.rc[gi_], dri_);
    const double r64 = S.r_lo + (irow + 0.5) * S.dr64;
    const float inf = __int_as_float(0x7f800000);
    float sv[5] = {0.f, 0.f, 0.f, 0.f, 0.f}, fsc = 1.f;
    double dist[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) dist[k] = (double)inf;
#pragma unroll 1
    for (int k = 0; k < 5; ++k) {  // (rolled: sv and dist move up one place per ray)
      const int l = m - 2 + k;
      float d2, fs;
      const bool in = ray_classify<2, 2>(sh, rs, S, gi_, ri_, dri_, irow, l, &d2, &fs);
      double D = (double)inf;
      if (S.periodic || (l >= 0 && l < NTH)) {
        const int lw = l < 0 ? l + NTH : (l >= NTH ? l - NTH : l);
        double c, sn;
        if (dr.ctab) { const double2 t = dr.ctab[S.cbase + lw]; c = t.x; sn = t.y; }
        else sincos(S.th_lo + (lw + 0.5) * S.dth64, &sn, &c);
        D = ray_distance_cs(sh.L.eps, sh.L.a, sh.wc, r64, c, sn);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) { sv[i] = sv[i + 1]; dist[i] = dist[i + 1]; }
      sv[4] = in ? __int_as_float(__float_as_int(d2) | 0x80000000) : d2;
      dist[4] = D;
      if (k == 2) fsc = fs;
    }
    if (signbit(sv[2])) {
      const DerLaw w = der_law(sh, P);
      float Id, Ir, Iu;
      float I = sh.generic ? brightness_der(w, -sv[2], &Id, &Ir, &Iu, std::true_type{})
                           : brightness_der(w, -sv[2], &Id, &Ir, &Iu, std::false_type{});
      // a spot scales the point's brightness and its derivatives
      I *= fsc; Id *= fsc; Ir *= fsc; Iu *= fsc;
      const bool Lin = signbit(sv[1]), Rin = signbit(sv[3]);
      float f_[2] = {0.f, 0.f}, sdc[2] = {0.f, 0.f}, xs_[2] = {0.f, 0.f};
      int nds[2] = {0, 0}, b0s[2] = {0, 0};
#pragma unroll 1
      for (int side = 0; side < 2; ++side) {
        const bool isL = side == 0;
        if (isL ? Lin : Rin) continue;
        float fv = 0.f, sc = 0.f, xt = 0.f;
        int nd = 0, xb = isL ? -2 : -1;
        if (isinf(isL ? sv[1] : sv[3])) {
          atomicOr(&sh.status, ICRS_ST_EDGE);
          fv = fdelta<float>(0.5f, (float)P.delta_c, P.uniform);
        } else {
          // stencil nodes xb, xb + 1, ... (an edge cuts one outer node off);
          // the crossing in FP32, then two Newton steps on the FP64 cubic
          // (Newton's forward differences)
          double y[4];
          float yf[4];
#pragma unroll
          for (int c = 0; c < 4; ++c) y[c] = isL ? dist[c] : dist[c + 1];
          nd = 4;
          if (isinf(y[3])) nd = 3;
          if (isinf(y[0])) { y[0] = y[1]; y[1] = y[2]; y[2] = y[3]; ++xb; --nd; }
          if (nd < 4) atomicOr(&sh.status, ICRS_ST_EDGE);
#pragma unroll
          for (int c = 0; c < 4; ++c) yf[c] = (float)y[c];
          const double yin = dist[2], yout = isL ? dist[1] : dist[3];
          const double dd1 = y[1] - y[0];
          const double dd2 = nd > 2 ? 0.5 * (y[2] - 2.0 * y[1] + y[0]) : 0.0;
          const double dd3 = nd > 3 ? (y[3] - 3.0 * y[2] + 3.0 * y[1] - y[0]) * (1.0 / 6.0) : 0.0;
          double xd = crossing_solve<float>(yf, (float)xb, nd, (float)yin, (float)yout, isL ? -1.0f : 1.0f, w.rho32, 1e-5f, 12);
          bool ok = true;
#pragma unroll 1
          for (int it = 0; it < 2; ++it) {
            const double tt = xd - xb;
            const double pv = y[0] + tt * (dd1 + (tt - 1.0) * (dd2 + (tt - 2.0) * dd3)) - sh.rho;
            const double pd = dd1 + (2.0 * tt - 1.0) * dd2 + ((3.0 * tt - 6.0) * tt + 2.0) * dd3;
            if (!(pd != 0.0)) { ok = false; break; }
            xd -= pv / pd;
          }
          if (!ok || !(isL ? (xd >= -1.0 && xd <= 0.0) : (xd >= 0.0 && xd <= 1.0)))
            xd = crossing_solve<double>(y, (double)xb, nd, yin, yout, isL ? -1.0 : 1.0, sh.rho, 1e-14, 60);
          const double dd = isL ? -xd : xd;
          const float dl = (float)dd;
          float fp;
          if (P.uniform) { fv = dl + 0.5f; fp = 1.0f; }
          else if (dd >= P.delta_c) {
            const float sq = sqrtf(1.0f + 0.5f / dl);
            fv = (0.5f + dl) * (2.0f / 3.0f) * sq;
            fp = (2.0f / 3.0f) * sq - (0.5f + dl) / (6.0f * dl * dl * sq);
          } else { fv = (2.0f / 3.0f) * dl + 0.5f; fp = 2.0f / 3.0f; }
          // the paper's gradient rule: the fixed derivative of the
          // second-order branch on both branches
          if (w.gradrule && !P.uniform) fp = 2.0f / 3.0f;
          const double tt = xd - xb;
          const double slope = dd1 + (2.0 * tt - 1.0) * dd2 + ((3.0 * tt - 6.0) * tt + 2.0) * dd3;
          xt = (float)tt;
          sc = (float)((isL ? -fp : fp) / slope);
        }
        f_[side] = fv; sdc[side] = sc; xs_[side] = xt; nds[side] = nd; b0s[side] = m + xb;
      }
      float W;
      if (Lin) W = f_[1];
      else if (Rin) W = f_[0];
      else {
        W = fmaxf(0.f, f_[0] + f_[1] - 1.0f);
        if (!(f_[0] + f_[1] - 1.0f > 0.f)) nds[0] = nds[1] = 0;
      }
      float v[12];
#pragma unroll
      for (int k = 0; k < 12; ++k) v[k] = 0.f;
      v[0] = I * (W - 1.0f);
      v[1 + 5] += (W - 1.0f) * Ir;
      v[1 + 6] += (W - 1.0f) * Iu;
      // the gradients of the rays' distances times their seeds: the point's
      // own (k = 0), then the crossings' on four stencil nodes a side
#pragma unroll 1
      for (int k = 0; k < 9; ++k) {
        int l = m;
        float a = (W - 1.0f) * Id;
        if (k > 0) {
          const int sd = k <= 4 ? 0 : 1, c = (k - 1) & 3;
          const int nd = sd ? nds[1] : nds[0];
          if (c >= nd) continue;
          const float sd_ = sd ? sdc[1] : sdc[0], sc = I * sd_, t = sd ? xs_[1] : xs_[0];
          if (c == 0) v[1 + 5] = __fadd_rn(v[1 + 5], __fmul_rn(I, sd_));
          // Lagrange basis of the nodes 0 .. nd - 1 at t
          const float t1 = t - 1.0f, t2 = t - 2.0f, t3 = t - 3.0f;
          float lc;
          if (nd == 4)
            lc = c == 0 ? -t1 * t2 * t3 * (1.0f / 6.0f)
                        : c == 1 ? 0.5f * t * t2 * t3 : c == 2 ? -0.5f * t * t1 * t3 : t * t1 * t2 * (1.0f / 6.0f);
          else if (nd == 3) lc = c == 0 ? 0.5f * t1 * t2 : c == 1 ? -t * t2 : 0.5f * t * t1;
          else lc = c == 0 ? -t1 : t;
          l = (sd ? b0s[1] : b0s[0]) + c;
          a = -sc * lc;
        }
        if (a == 0.f || (!S.periodic && (l < 0 || l >= NTH))) continue;
        const int lw = l < 0 ? l + NTH : (l >= NTH ? l - NTH : l);
        const int mgrp = (int)__umulhi((unsigned int)lw, S.gmagic);
        const int ai = S.abase + gi_ * S.mth + mgrp;
        const cf t = tab_at(P.tabf + 2 * S.tbase, lw - mgrp * S.gth);
        cf dz, dw;
        (void)ray_eval<2>(P.anch[ai], t.x, t.y, ri_, dri_, nullptr, &dw, &dz);
        grad_core(w, dz, dw, t.x, t.y, ri_, (float)lw + 0.5f, dr.aA[ai], dr.acs[ai], a, v + 1);
      }
      RowTerms t;
#pragma unroll
      for (int k = 0; k < 12; ++k) t.v[k] = v[k];
      row_add(dr.sums + (threadIdx.x >> 5) * DSUM * 32, lane, irow, ri_, t);
      kahan_add(acc, ri_ * v[0] * S.bxw);
    }
  }
  __syncwarp();
  return acc;
}

// Sum over the epoch's sectors of this thread's share (FP64); the sectors'
// derivative sums into dr.wsum, ICRS_ST_* bits into sh.status.
template <class SH>
__device__ __noinline__ double der_stage(SH& sh, RayShared& rs, const DerRays& dr) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int NT = blockDim.x, NW = NT >> 5;
  // (The launch's arguments, the anchors, the queue and the lane sums are read
  // through shared memory where they are used: kept in registers they pushed
  // the sweep's own values into local memory, a spotted set's gradient at 1024
  // x 2048 54 ms against 43.7.)
  const RayArgs& P = rs.P;
  const int NR = P.NR, NTH = P.NTH;
  const DerLaw w = der_law(sh, P);
  float2 acc = make_float2(0.f, 0.f);  // Kahan sum of this thread
  const unsigned lt_mask = (1u << lane) - 1u;
  // Tasks are dealt out in a fixed order (this thread's tasks tw, tw + NW, ...:
  // a compensated sum's order shows in A).  Their column chunks repeat with a
  // period of 4, 8 or 16, and an SM's four schedulers take the warps by their
  // number modulo 4, so tw = warp would leave one scheduler with the chunks
  // across the image and another with empty ones; turned by one place every
  // four warps, each has all of them (1024 x 2048 chi^2 gradient, 2,000 epochs:
  // 78 ms before, 72.5 with it; 64 x 256 the same).  The sums are the same bits.
  const int tw = (warp & ~3) | ((warp + (warp >> 2)) & 3);
  int dq_n = 0;
  const int nbox = sh.nbox;
  const bool generic = sh.generic, spot = sh.spot;

  if (tid < nbox) sec_setup(rs.sec[tid], sh.box[tid], NR, NTH);
  if (tid == 0) rs.b1 = 0;
  __syncthreads();

  for (;;) {
    ray_tables<2, 2>(sh, rs, dr);
    const int b0 = rs.b0, b1 = rs.b1;
    if (b0 >= b1) break;
    for (int b = b0; b < b1; ++b) {
      const Sec& S = rs.sec[b];
#pragma unroll
      for (int k = 0; k < DSUM; ++k) dr.sums[(warp * DSUM + k) * 32 + lane] = 0.0;
      __syncwarp();
      for (int tk = tw; tk < S.ntask; tk += NW) {
        const int rbk = tk / S.nch, chk = tk - rbk * S.nch;
        const int i = rbk * 32 + lane;
        const bool rowok = i < NR;
        const int ii = rowok ? i : NR - 1;
        const int gi = ii / S.gr;
        const float fri = (float)(ii - gi * S.gr) + 0.5f - 0.5f * (float)S.gr;
        const float dri = __fmul_rn(fri, S.dr32), ri = __fmaf_rn(fri, S.dr32, S.rc[gi]);
        const int c0 = chk * S.ch, c1 = min(c0 + S.ch, NTH);
        const int gth = S.gth, sb = w.gradrule ? 0 : S.sb;
        const float* const tps = P.tabf + 2 * S.tbase;
        float rowacc = 0.f;  // sum of I over the row's inside rays
        float pg[11];
#pragma unroll
        for (int k = 0; k < 11; ++k) pg[k] = 0.f;
        unsigned win = halo_flag<2, 2>(sh, rs, b, gi, ri, dri, ii, c0 - 1);
        AnchorF ar;  // the current group's anchor, A_j and angle
        int aidx = 0;
        float4 A01 = make_float4(0.f, 0.f, 0.f, 0.f);
        float2 cs = make_float2(1.f, 0.f);
        int gbase = 0;
        float spx = 0.f;  // its spot band's width
        auto push_bits = [&](unsigned bm, int base) {
          while (__any_sync(0xffffffffu, bm != 0u)) {
            const bool has = bm != 0u;
            const int m = base - (has ? __ffs(bm) - 1 : 0);
            bm &= bm - 1u;
            unsigned rem = __ballot_sync(0xffffffffu, has);
            while (rem) {
              if (dq_n == DQ) { acc = der_flush(sh, rs, dr, P.wqueue + warp * DQ, DQ, acc); dq_n = 0; }
              const int at = dq_n + __popc(rem & lt_mask);
              const bool take = ((rem >> lane) & 1u) && at < DQ;
              if (take) P.wqueue[warp * DQ + at] = pack_point(b, i, m);
              const unsigned tk_ = __ballot_sync(0xffffffffu, take);
              dq_n += __popc(tk_);
              rem &= ~tk_;
            }
          }
        };
        auto centres = [&](int nb, bool first) -> unsigned {
          unsigned bm = ((win & ~((win << 1) & (win >> 1))) >> 1) & ((1u << nb) - 1u);
          if (first) bm &= ~(1u << (nb - 1));
          return rowok ? bm : 0u;
        };
        // one column: value, flag and, for a decided ray, its seed and
        // gradient; an undecided ray waits for the block end.  sure: every
        // ray of the warp's column is known to be inside.
        auto colD = [&](int l, const cf t, bool& unc, auto hc, auto sure) {
          cf dz, dw;
          const float d2 = ray_eval<2>(ar, t.x, t.y, ri, dri, nullptr, &dw, &dz);
          bool in = true, u_ = false;
          if constexpr (!decltype(sure)::value) {
            in = d2 < ar.lo2;
            u_ = !(in || d2 > ar.hi2);
            unc = unc || u_;
            win = (win << 1) | (in ? 1u : 0u);
          }
          if (!u_) {
            float fs = 1.f;
            if constexpr (decltype(hc)::value)
              fs = in && spot ? spot_sweep<2, 2>(sh, rs, S, aidx, SpotBand{P.spc[aidx], spx}, dw, t.x, t.y, ri, dri, ii, l) : 1.f;
            const float a = seed_of(w, in, d2, pg, rowacc, hc, fs);
            if (a != 0.f) grad_core(w, dz, dw, t.x, t.y, ri, (float)l + 0.5f, A01, cs, a, pg);
          }
        };
        int l = c0;
        bool first = true;
        while (l < c1) {
          const int mgrp = (int)__umulhi((unsigned int)l, S.gmagic);
          aidx = S.abase + gi * S.mth + mgrp;
          ar = P.anch[aidx];
          A01 = dr.aA[aidx];
          cs = dr.acs[aidx];
          if (spot) spx = spot_band(sh, rs, ar, aidx).X;
          gbase = mgrp * gth;
          const int lend = min(gbase + gth, c1);
          const bool test = __any_sync(0xffffffffu, sb && ar.rout < __int_as_float(0x7f800000));
          cf wa = mk(0.f, 0.f);
          if (test) {
            const cf t = tab_at(tps, l - gbase);
            (void)ray_eval<2>(ar, t.x, t.y, ri, dri, nullptr, &wa);
          }
          while (l < lend) {
            const int ls = test ? min(l + sb, lend) : lend;  // end of the superblock
            bool all_in = false;
            if (test) {
              cf wb;
              const cf t = tab_at(tps, ls - gbase);
              const float db2 = ray_eval<2>(ar, t.x, t.y, ri, dri, nullptr, &wb);
              bool out, inn;
              chord_test(ar, wa, wb, db2, out, inn);
              wa = wb;
              const bool all_out = __all_sync(0xffffffffu, out);
              all_in = !generic && ls - l >= 2 && __all_sync(0xffffffffu, inn);
              if (all_out || all_in) {
                if (all_in) {
                  win = (win << 2) | 3u;
                  unsigned bm = ((win & ~((win << 1) & (win >> 1))) >> 1) & (first ? 1u : 3u);
                  if (!rowok) bm = 0u;
                  if (__any_sync(0xffffffffu, bm != 0u)) push_bits(bm, l);
                } else {
                  const unsigned bm = (rowok && !first) ? win & 1u : 0u;
                  if (__any_sync(0xffffffffu, bm != 0u)) push_bits(bm, l - 1);
                }
                first = false;
                win = all_in ? 0xffffffffu : 0u;
                if (all_out) { l = ls; continue; }
              }
            }
            if (all_in) {
              bool unc = false;
#pragma unroll 1
              for (; l < ls; ++l) colD(l, tab_at(tps, l - gbase), unc, std::false_type{}, std::true_type{});
              continue;
            }
            while (l < ls) {
              const int nb = min(KB, ls - l);
              bool unc = false;
              if (generic) {
#pragma unroll 1
                for (int k = 0; k < nb; ++k)
                  colD(l + k, tab_at(tps, l + k - gbase), unc, std::true_type{}, std::false_type{});
              } else {
#pragma unroll 1
                for (int k = 0; k < nb; ++k)
                  colD(l + k, tab_at(tps, l + k - gbase), unc, std::false_type{}, std::false_type{});
              }
              unsigned bm = centres(nb, first);
              if (__any_sync(0xffffffffu, unc || bm != 0u)) {
                if (unc) {
                  RowSums r;
                  r.racc = rowacc;
#pragma unroll
                  for (int k = 0; k < 11; ++k) r.pg[k] = pg[k];
                  unsigned bits;
                  r = der_undecided(sh, rs, dr, b, aidx, gbase, ri, dri, ii, l, nb, &bits, r);
                  win |= bits;
                  rowacc = r.racc;
#pragma unroll
                  for (int k = 0; k < 11; ++k) pg[k] = r.pg[k];
                  bm = centres(nb, first);
                }
                push_bits(bm, l + nb - 2);
              }
              first = false;
              l += nb;
            }
          }
        }
        // right halo column c1: finalizes column c1 - 1
        win = (win << 1) | halo_flag<2, 2>(sh, rs, b, gi, ri, dri, ii, c1);
        push_bits(rowok ? (((win & ~((win << 1) & (win >> 1))) >> 1) & 1u) : 0u, c1 - 1);
        if (rowok) {
          RowTerms t;
          t.v[0] = rowacc;
#pragma unroll
          for (int k = 0; k < 11; ++k) t.v[k + 1] = pg[k];
          // (a chunk beside the image adds nothing; FP64 instructions are what
          // the rows' terms cost)
          unsigned nz = 0u;
#pragma unroll
          for (int k = 0; k < 12; ++k) nz |= __float_as_uint(t.v[k]) << 1;
          if (nz) row_add(dr.sums + warp * DSUM * 32, lane, ii, ri, t);
          kahan_add(acc, ri * rowacc * S.bxw);
        }
      }
      if (dq_n) acc = der_flush(sh, rs, dr, P.wqueue + warp * DQ, dq_n, acc);
      dq_n = 0;
      // the warp's sums of this sector, lane k sum k over the 32 columns
      __syncwarp();
      if (lane < DSUM) {
        double t = 0.0;
#pragma unroll 4
        for (int j = 0; j < 32; ++j) t += dr.sums[(warp * DSUM + lane) * 32 + ((j + lane) & 31)];
        dr.wsum[(b * DSUM + lane) * TASK_WARPS + warp] = t;
      }
      __syncwarp();
    }
    __syncthreads();
  }
  return (double)acc.x - (double)acc.y;
}

// dS / d(r_lo, r_hi, th_lo, width) of each sector into Gb and dS / d(w_c.x,
// w_c.y, rho, u1, a1.x, a2.x, eps1, eps2) into H (after a barrier; every
// thread calls it).
__device__ inline void der_sums(const RayShared& rs, const DerRays& dr, int nbox, double (*Gb)[4], double* H) {
  const int tid = threadIdx.x;
  auto total = [&](int b, int k) -> double {
    double s = 0.0;
    for (int w = 0; w < TASK_WARPS; ++w) s += dr.wsum[(b * DSUM + k) * TASK_WARPS + w];
    return s;
  };
  // one thread per sum, the totals in place of warp 0's
  for (int i = tid; i < nbox * DSUM; i += blockDim.x) {
    const double t = total(i / DSUM, i % DSUM);
    dr.wsum[i * TASK_WARPS] = t;
  }
  __syncthreads();
  auto at = [&](int b, int k) -> double { return dr.wsum[(b * DSUM + k) * TASK_WARPS]; };
  if (tid < nbox) {
    const Sec& S = rs.sec[tid];
    const double NR = rs.P.NR, NTH = rs.P.NTH, K = S.dr64 * S.dth64;
    const double r0 = at(tid, 0), r1 = at(tid, 1) / NR, rr = at(tid, 2), v1 = at(tid, 3), v1f = at(tid, 4) / NR;
    Gb[tid][0] = K * (v1 - v1f) + K * (r0 - r1) - rr * S.dth64 / NR;
    Gb[tid][1] = K * v1f + K * r1 + rr * S.dth64 / NR;
    Gb[tid][2] = K * at(tid, 5);
    Gb[tid][3] = K * at(tid, 6) / NTH + rr * S.dr64 / NTH;
  }
  if (tid >= 32 && tid < 40) {
    double h = 0.0;
    for (int b = 0; b < nbox; ++b) h += rs.sec[b].dr64 * rs.sec[b].dth64 * at(b, 7 + tid - 32);
    H[tid - 32] = h;
  }
  __syncthreads();
}

}  // namespace icrs
