// Forward ray stage of the magnification kernel: all sectors of one epoch,
// their polar grids, the quadrature of Appendix A (Miyazaki & Kawahara,
// arXiv:2510.02639, Sec. 3.3) and the per-thread sums.
//
// The sectors are taken together (in batches when their tables do not fit):
// their anchors are formed at once, their tasks share one queue of work and
// the rare FP64 crossings are solved at the end, one ray per lane.  One sector
// after another, each with its own FP64 chains (an FP64 operation takes 66
// cycles from operand to result here, a division 570, a sine 1750) and its
// own barriers, took 70k cycles a sector at 64 x 256, five times the rays'.
//
// A warp takes a task of 32 rows (lane = row) and a chunk of theta columns.
// Columns are taken in superblocks: the source-plane offsets of a row at a
// superblock's two ends bound the offsets between them (chord plus sagitta, see
// AnchorF::rout), so a superblock that lies outside the source on all 32 rows
// is skipped and one that lies inside on all rows needs no per-ray decisions.
// What is skipped would have added exactly zero and what is summed is summed
// in the same order as without the test, so the results are the same bits.
//
// Bounded by the FP32 pipes and the latency of a ray's chain at fine grids (FMA
// pipe 58 % busy at 1024 x 2048, nine tenths of an epoch's time) and by the
// FP64 chains of the other phases at coarse ones.  The magnification kernel,
// 64 sets: 25,600 epochs at 1024 x 2048 328 ms before and 205 with this stage;
// 32,000 at 64 x 256 65 ms and 49 (with the binning and re-solve phases).
#pragma once

#include "icrs_common.cuh"
#include "icrs_df64.cuh"
#include "icrs_sectors.cuh"

namespace icrs {

using Box = BoxT<double>;

constexpr int MAXANCH = 128;     // FP64 anchors of a batch of sectors
constexpr int GTH_MAX = 256;     // columns per theta group (at most)
constexpr int MAXSEC = 10;       // sectors of an epoch (N_deg of the triple lens)
constexpr int TASK_WARPS = 16;   // the theta chunks are cut for this many warps
constexpr int DQ = 32;           // deferred boundary points per warp (derivative): one per lane at a flush
constexpr int FQ = 64;           // the same, forward: flushed 32 at a time
constexpr int PCAP = 64;         // places for a task's boundary points (forward; more are gathered, see gather_points)
constexpr int XQ = 8;            // boundary points per warp whose crossing needs FP64
constexpr float EPS32 = 5.9604645e-8f;  // 2^-24
constexpr int KB = 8;            // columns per block (even: column pairs load as 16 bytes)

// Anchor of a (theta group, r group) of a sector: the rays' squared distance
// is evaluated about it in FP32 with U = sum_j K_j / Q_j (A_j = e^{-i th_m}
// (z_m - a_j), K_j = eps_j / A_j, Q_j = A_j + dz, dz the ray's offset from the
// anchor z_m in the anchor's rotated frame) as one quotient N / P of
// polynomials in dz, with N = sum_j K_j prod_{k != j} Q_k and P = prod_j Q_j:
//   binary:  N = n0 + n1 dz,             P = p0 + dz (p1 + dz)
//   triple:  N = n0 + dz (n1 + dz n2),   P = p0 + dz (p1 + dz (p2 + dz))
// (coefficients formed in FP64 and rounded once).
struct AnchorF {
  cf ws;        // e^{-i th_m} (f(z_m) - w_c)
  cf n[3];      // numerator coefficients
  cf p[3];      // denominator coefficients (monic)
  float e0;     // error bound constant part
  float lo2;    // below: every ray of the group is inside the source (FP32 certain)
  float hi2;    // above: every ray of the group is outside (FP32 certain)
  // superblocks: with both ends' squared offsets below in2 every ray between
  // them has a squared distance below lo2; with the chord between the ends
  // farther than rout from the centre, every ray's is above hi2
  float in2;
  float rout;
};

// One sector of the current batch.
struct Sec {
  double r_lo, r_hi, th_lo, dr64, dth64;
  float dr32, dth32, bxw;
  float rc[4];           // radius of each r group's anchors
  unsigned int gmagic;   // l / gth = umulhi(l, gmagic)
  int periodic;
  int gth, gr, mth, nanch;  // columns and rows per group, theta groups, anchors
  int abase, tbase;      // first anchor, first offset-table column
  int cbase;             // first column of the cosine table (derivative)
  int ch, nch;           // columns per chunk, chunks
  int ntask;
  int sb;                // columns per superblock
  int task0;             // its first task in the batch
  float sag;             // (sb dth)^2 / 8
};

// A boundary point: sector of the batch (4 bits), row (12), column (13).
__device__ __forceinline__ int pack_point(int b, int row, int col) { return (b << 25) | (row << 13) | col; }

// Offset of ray (i, l) from the source centre in FP64.
template <int NL>
__device__ __noinline__ cd sec_offset64(const double* eps, const cd* a, cd wc, const Sec& S, int i, int l) {
  double r = S.r_lo + (i + 0.5) * S.dr64;
  double th = S.th_lo + (l + 0.5) * S.dth64;
  double s, c;
  sincos(th, &s, &c);
  cd z = mk(r * c, r * s);
  return lens_map<NL, double>(eps, a, z) - wc;
}

// Columns per theta chunk of a sector, and its number of tasks: 32 rows (one
// per lane) x a chunk of an even number of columns, about 8 tasks per warp.
__host__ __device__ inline int chunk_columns(int NR, int NTH) {
  const int nrb = (NR + 31) >> 5, nch = (8 * TASK_WARPS + nrb - 1) / nrb;
  const int c = 2 * ((NTH + 2 * nch - 1) / (2 * nch));
  return NTH < 16 ? NTH : (c < 16 ? 16 : (c < NTH ? c : NTH));
}
__host__ __device__ inline int sector_tasks(int NR, int NTH) {
  const int c = chunk_columns(NR, NTH);
  return ((NR + 31) >> 5) * ((NTH + c - 1) / c);
}

// Group layout of sector B (one thread).
__device__ inline void sec_setup(Sec& S, const Box& B, int NR, int NTH) {
  S.r_lo = B.r_lo; S.r_hi = B.r_hi; S.th_lo = B.th_lo; S.periodic = B.periodic;
  S.dr64 = (B.r_hi - B.r_lo) / NR;
  S.dth64 = B.width / NTH;
  S.dr32 = (float)S.dr64;
  S.dth32 = (float)S.dth64;
  S.bxw = (float)(S.dr64 * S.dth64);
  // anchors: enough groups that an anchor is within ~0.025 of its rays
  const double LMAX = 0.05;
  int mth = (int)ceil(B.r_hi * B.width / LMAX);
  int mr = (int)ceil((B.r_hi - B.r_lo) / LMAX);
  mth = min(max(mth, 1), min(64, NTH));
  // groups of at most GTH_MAX columns (the offset table's size; for
  // n_theta <= 8192 this needs at most 32 groups)
  mth = max(mth, (NTH + GTH_MAX - 1) / GTH_MAX);
  mr = min(max(mr, 1), min(4, NR));
  mth = min(mth, MAXANCH / mr);  // the anchor table holds MAXANCH entries
  // theta groups of an even width: column pairs (l, l + 1), l even, share
  // their group
  S.gth = 2 * ((NTH + 2 * mth - 1) / (2 * mth));
  S.gr = (NR + mr - 1) / mr;
  S.mth = (NTH + S.gth - 1) / S.gth;
  mr = (NR + S.gr - 1) / S.gr;
  S.nanch = S.mth * mr;
  // l / gth as a multiply-high by ceil(2^32 / gth), exact for l, gth < 2^16
  // (here both <= 8192)
  S.gmagic = (unsigned int)((0xFFFFFFFFull / (unsigned long long)S.gth) + 1ull);
  for (int gi = 0; gi < mr; ++gi) S.rc[gi] = (float)(B.r_lo + (gi * S.gr + 0.5 * S.gr) * S.dr64);
  S.ch = chunk_columns(NR, NTH);
  S.nch = (NTH + S.ch - 1) / S.ch;
  S.ntask = ((NR + 31) >> 5) * S.nch;
  // A superblock's test costs about two ray evaluations a row, and what it
  // saves grows with the number of superblocks across the image: 16 columns, 32
  // from 1024 a sector, 64 from 2048, which makes at most 64 of them up to 4096
  // columns; none when a chunk holds only two blocks.  The optimum
  // is flat: 64 sets, without and with 16, 32, 64 columns, 12,800 epochs at 256
  // x 1024 44.6 and 41.8, 40.4, 40.5 ms; 6,400 at 512 x 1024 31.1 and 28.1, 27.0,
  // 26.8; 6,400 at 1024 x 2048 80.2 and 60.6, 55.2, 53.5 ms.
  S.sb = S.ch <= 2 * KB ? 0 : (NTH >= 2048 ? 64 : (NTH >= 1024 ? 32 : 16));
  const float ls = (float)S.sb * S.dth32;
  S.sag = 0.125f * ls * ls;
}

// Half-width X of a group's band on squared distances, as in make_anchor but in
// FP64.
template <int NL>
__device__ __noinline__ double band64(const cd* A64, const cd* K64, const cd* nc, const cd* pc, double half, float e0,
                                      float rho32) {
  double um = 0.0, pmin = 1.0;
  for (int j = 0; j < NL; ++j) {
    const double aa = sqrt(abs2(A64[j]));
    um += sqrt(abs2(K64[j])) / (aa - half);
    pmin *= aa - half;
  }
  const double mn = sqrt(abs2(nc[0])) + half * (sqrt(abs2(nc[1])) + half * sqrt(abs2(nc[2])));
  const double mp = NL == 2 ? sqrt(abs2(pc[0])) + half * (sqrt(abs2(pc[1])) + half)
                            : sqrt(abs2(pc[0])) + half * (sqrt(abs2(pc[1])) + half * (sqrt(abs2(pc[2])) + half));
  constexpr double cN = NL == 2 ? 4.0 : 9.0, cP = NL == 2 ? 6.0 : 13.0;
  const double du = EPS32 * (cN * mn + (cP + 9.0) * um * mp) / pmin;
  const double eb = (double)e0 + 2.0 * half * (du + 3.0 * EPS32 * um);
  return 1.01 * (2.0 * (double)rho32 * eb + eb * eb) + 8.0 * EPS32 * ((double)rho32 * (double)rho32);
}

// An anchor's quantities in FP64.
template <int NL>
struct AnchorX {
  double cs, sn;  // of the anchor's angle
  cd ws, A[NL], n[3], p[3];
};

// Anchor an of sector S (one thread).
template <int NL>
__device__ inline AnchorF make_anchor(const Sec& S, const double* eps, const cd* a, cd wc, float rho32, int an,
                                      AnchorX<NL>& ax) {
  cd* const A64 = ax.A;
  cd* const nc = ax.n;
  cd* const pc = ax.p;
  const int gi = an / S.mth, mi = an % S.mth;
  const double rc = S.r_lo + (gi * S.gr + 0.5 * S.gr) * S.dr64;
  const double thc = S.th_lo + (mi * S.gth + 0.5 * S.gth) * S.dth64;
  double sn, cs;
  sincos(thc, &sn, &cs);
  ax.cs = cs; ax.sn = sn;
  const cd R = mk(cs, -sn);  // e^{-i th_c}
  const cd zc = mk(rc * cs, rc * sn);
  const cd w = lens_map<NL, double>(eps, a, zc) - wc;
  AnchorF af;
  ax.ws = R * w;
  af.ws = tof(ax.ws);
  cd K64[NL];
  float aa[NL], kk[NL];
  for (int j = 0; j < NL; ++j) {
    A64[j] = R * (zc - a[j]);
    K64[j] = scl(inv(A64[j]), eps[j]);
    aa[j] = sqrtf(abs2(tof(A64[j])));
    kk[j] = fabsf((float)eps[j]) / aa[j];  // (|K_j|: a mass can be negative, see g1)
  }
  nc[2] = pc[2] = mk(0.0, 0.0);
  if constexpr (NL == 2) {
    nc[0] = K64[0] * A64[1] + K64[1] * A64[0];
    nc[1] = K64[0] + K64[1];
    pc[0] = A64[0] * A64[1];
    pc[1] = A64[0] + A64[1];
  } else {
    nc[0] = K64[0] * (A64[1] * A64[2]) + K64[1] * (A64[0] * A64[2]) + K64[2] * (A64[0] * A64[1]);
    nc[1] = K64[0] * (A64[1] + A64[2]) + K64[1] * (A64[0] + A64[2]) + K64[2] * (A64[0] + A64[1]);
    nc[2] = K64[0] + K64[1] + K64[2];
    pc[0] = A64[0] * A64[1] * A64[2];
    pc[1] = A64[0] * A64[1] + A64[0] * A64[2] + A64[1] * A64[2];
    pc[2] = A64[0] + A64[1] + A64[2];
  }
  for (int k = 0; k < 3; ++k) { af.n[k] = tof(nc[k]); af.p[k] = tof(pc[k]); }
  // error bound of |Delta w'|: anchor term plus rounding of the ray's offset
  // (at most the group half-diagonal) and of its image term.  (The bounds are
  // formed in FP32: their factors 2 and 1.01 leave room for the 1e-5 by which
  // that rounds them, aa - half cancelling to a seventeenth of aa at the nearest
  // lens admitted included; 400,000 random anchors a lens count, up to that
  // edge, were off by 8e-6 at most.  The FP64 form took ten square roots and
  // divisions of 600 cycles each.)
  const float half = 0.5f * (float)S.gr * S.dr32 + (float)S.r_hi * 0.5f * (float)S.gth * S.dth32;
  af.e0 = 16.0f * EPS32 * (fabsf(af.ws.x) + fabsf(af.ws.y) + 2.0f * half);
  // the group's band: every ray has |dz| <= half, so |Q_j| >= |A_j| - half,
  // |P| >= prod_j (|A_j| - half) and |U| <= sum_j |K_j| / (|A_j| - half); the
  // rounding error of the FP32 quotient is bounded by u (cN M_N + (cP + 9)
  // |U| M_P) / |P| (M_N, M_P: the polynomials with coefficient moduli, at
  // |dz| = half) and that of dz U by |dz| (that + 3 u |U|), times 2 for the
  // FP32 evaluation of the bound itself (see ray_eval)
  const double rr64 = (double)rho32 * (double)rho32;
  const float rr = (float)rr64, inf = __int_as_float(0x7f800000);
  af.lo2 = -1.0f; af.hi2 = inf;
  af.in2 = -1.0f; af.rout = inf;
  bool bounded = true, near_ = false;
  float um = 0.f, pmin = 1.f, g1 = 0.f, g2 = 0.f;
  const float hx = 1.0001f * half + 1.001f * (float)S.r_hi * S.dth32;  // one column past the group
  for (int j = 0; j < NL; ++j) {
    if (!(aa[j] > 1.0625f * half)) bounded = false;
    if (!(aa[j] > 1.0626f * hx)) near_ = true;
    const float m_ = aa[j] - half, ih = 1.0f / (aa[j] - hx);
    um += kk[j] / m_;
    pmin *= m_;
    // (moduli: q2 + q3 > 1 or q < 0 make a mass negative, and the method has a value there too)
    g1 += fabsf((float)eps[j]) * ih * ih;
    g2 += 2.0f * fabsf((float)eps[j]) * ih * ih * ih;
  }
  if (bounded) {
    float mn = 0.f, mp = 1.f;
    for (int k = NL - 1; k >= 0; --k) { mn = mn * half + sqrtf(abs2(af.n[k])); mp = mp * half + sqrtf(abs2(af.p[k])); }
    constexpr float cN = NL == 2 ? 4.0f : 9.0f, cP = NL == 2 ? 6.0f : 13.0f;
    const float du = EPS32 * (cN * mn + (cP + 9.0f) * um * mp) / pmin;
    const float eb = af.e0 + 2.0f * half * (du + 3.0f * EPS32 * um);
    const float X = 1.01f * (2.0f * rho32 * eb + eb * eb) + 8.0f * EPS32 * rr;
    // (a wide band's 1e-6 would be many units of lo2 and hi2, and move rays
    // between the FP32 and the FP64 decision: FP64)
    double X64 = (double)X;
    if (X > 1e-3f * rr)
      X64 = band64<NL>(A64, K64, nc, pc, 0.5 * S.gr * S.dr64 + S.r_hi * 0.5 * S.gth * S.dth64, af.e0, rho32);
    if (X64 < 0.5 * rr64) {
      af.lo2 = __double2float_rd(rr64 - X64);
      af.hi2 = __double2float_ru(rr64 + X64);
      // superblocks: along a row w(theta) deviates from the chord between a
      // superblock's ends by at most max |w''| l^2 / 8, with z'' = -z, w = z -
      // conj(sum_j eps_j / (z - a_j)): |w''| <= r (1 + |gamma|) + r^2
      // |gamma'|, |gamma| <= sum eps_j / (|A_j| - h)^2, |gamma'| <= 2 sum
      // |eps_j| / (|A_j| - h)^3; plus the ends' own errors.  No test when that
      // is more than half the source radius.
      const float rm = (float)S.r_hi;
      const float e = 1.001f * S.sag * (rm * (1.0f + g1) + rm * rm * g2) + 4.0f * eb + 4e-6f * rho32;
      if (S.sb && !near_ && e < 0.5f * rho32) {
        const float si = sqrtf(af.lo2) - e;
        if (si > 0.f) af.in2 = si * si * (1.0f - 1e-6f);
        af.rout = sqrtf(af.hi2) + e;
      }
    }
  }
  return af;
}


// ---------------------------------------------------------------- quadrature
// Crossing of the interpolated distance with rho.  The stencil nodes are
// consecutive integers x0, x0+1, ... (npt = 2..4), so the interpolant is
// written in Newton's forward-difference form (the same polynomial as the
// Lagrange form of Appendix A, without divisions).  The root on the bracket
// between the inside sample (offset 0, p < rho) and the outside sample
// (x_out = +-1, p >= rho) is found by the Illinois variant of regula falsi,
// which keeps the bracket and converges superlinearly.
template <class T>
__device__ inline T crossing_solve(const T* y, T x0, int npt, T yin, T yout, T x_out, T rho, T tol, int iters) {
  const T d1 = y[1] - y[0];
  const T d2 = npt > 2 ? T(0.5) * (y[2] - T(2) * y[1] + y[0]) : T(0);
  const T d3 = npt > 3 ? (y[3] - T(3) * y[2] + T(3) * y[1] - y[0]) * T(1.0 / 6.0) : T(0);
  T a = T(0), ga = yin - rho;      // inside end  (g < 0)
  T b = x_out, gb = yout - rho;    // outside end (g >= 0)
  int side = 0;
  for (int it = 0; it < iters; ++it) {
    T den = gb - ga;
    T c = (den != T(0)) ? b - gb * (b - a) / den : T(0.5) * (a + b);
    T t = c - x0;
    T gc = y[0] + t * (d1 + (t - T(1)) * (d2 + (t - T(2)) * d3)) - rho;
    if (gc == T(0)) return c;
    if ((gc < T(0)) == (gb < T(0))) {
      b = c; gb = gc;
      if (side == -1) ga *= T(0.5);
      side = -1;
    } else {
      a = b; ga = gb;
      b = c; gb = gc;
      side = 1;
    }
    if (fabs(b - a) < tol) break;
  }
  return b;
}

// LD correction f(delta) (Appendix A.2) or the uniform rule delta + 1/2.
template <class T>
__device__ __forceinline__ T fdelta(T d, T delta_c, int uniform) {
  if (uniform) return d + T(0.5);
  if (d >= delta_c) return (T(0.5) + d) * (T(2.0 / 3.0) * sqrt(T(1) + T(1) / (T(2) * d)));
  return T(2.0 / 3.0) * d + T(0.5);
}

// Crossing on the FP64 stencil ys (nodes xs0, xs0 + 1, ...): two Newton steps
// on the cubic from the FP32 crossing, the Illinois solve if they leave the
// bracket.
__device__ __noinline__ double crossing64(const double* ys, double xs0, int nd, double yin, double yout, bool isL,
                                          float x32, double rho) {
  const double d1 = ys[1] - ys[0];
  const double d2 = nd > 2 ? 0.5 * (ys[2] - 2.0 * ys[1] + ys[0]) : 0.0;
  const double d3 = nd > 3 ? (ys[3] - 3.0 * ys[2] + 3.0 * ys[1] - ys[0]) * (1.0 / 6.0) : 0.0;
  double x = (double)x32, st = 1.0;
  for (int it = 0; it < 3; ++it) {
    const double t = x - xs0;
    const double pv = ys[0] + t * (d1 + (t - 1.0) * (d2 + (t - 2.0) * d3)) - rho;
    const double pd = d1 + (2.0 * t - 1.0) * d2 + ((3.0 * t - 6.0) * t + 2.0) * d3;
    if (!(pd != 0.0)) break;
    st = pv / pd;
    x -= st;
    if (fabs(st) < 1e-9) break;  // quadratic: the next step would be ~1e-18
  }
  if (!(fabs(st) < 1e-7) || !(isL ? (x >= -1.0 && x <= 0.0) : (x >= 0.0 && x <= 1.0)))
    x = crossing_solve<double>(ys, xs0, nd, yin, yout, isL ? -1.0 : 1.0, rho, 1e-14, 60);
  return x;
}

// What the ray stage takes from the launch and the set; its out-of-line parts
// read it from shared memory.
struct RayArgs {
  AnchorF* anch;
  float2* spc;      // spot centre in each anchor's frame
  float* tabf;      // group offsets (cos d - 1, sin d) of the batch's sectors
  int* wqueue;      // boundary points per warp: forward FQ (point, place) pairs, derivative DQ points
  float* rowp;      // [task][32] the rows' r_i x sum (forward)
  float* pterm;     // [task][PCAP] the boundary points' terms
  int* pcnt;        // [task] the places they take
  int tcap;         // tasks of a batch
  int tabcap;       // columns that tabf holds
  int ccap;         // columns that the derivative's cosine table holds (0: none)
  int NR, NTH, uniform, split, diag;
  float one;        // 1
  float sfac;       // sigmoid steepness of the paper's gradient rule
  int gradrule;
  double delta_c;
};

struct RayShared {
  RayArgs P;
  Sec sec[MAXSEC];
  int b0, b1, nanch, ncol, ntask, next;
  int2 xq[TASK_WARPS][XQ];   // boundary points whose crossing needs FP64, per warp
};

// c + a b in FP32, each operation rounded as written.
__device__ __forceinline__ cf cfma_rn(const cf a, const cf b, const cf c) {
  return mk(__fmaf_rn(a.x, b.x, __fmaf_rn(-a.y, b.y, c.x)), __fmaf_rn(a.x, b.y, __fmaf_rn(a.y, b.x, c.y)));
}

// Squared distance |Delta w'|^2 of the ray at group offset (tx, ty) in the row
// (ri_, dri_) of anchor an: Delta w' = ws + dz + conj(dz N / P), dz = (ri_ tx +
// dri_, ri_ ty).  Every operation is rounded as written, so each evaluation of
// a ray gives the same bits.  With eb: the ray's own bound on the error of
// |Delta w'|, e0 + 2 |dz| u (cN M_N + cU |U| M_P) / |P|, from |dN| <= cN u
// M_N, |dP| <= cP u M_P (Horner in complex FMAs, plus the rounded
// coefficients) and cU = 3 cP + 10 (the quotient, |P|^2, the reciprocal and
// the products), times 2 for the FP32 evaluation of the bound.  dwo: Delta w'
// itself, dzo: dz.
template <int NL>
__device__ __forceinline__ float ray_eval(const AnchorF& an, float tx, float ty, float ri_, float dri_, float* eb,
                                          cf* dwo, cf* dzo = nullptr) {
  const cf dz = mk(__fmaf_rn(ri_, tx, dri_), __fmul_rn(ri_, ty));
  cf Pq, Nq;
  if constexpr (NL == 2) {
    const cf F = mk(__fadd_rn(an.p[1].x, dz.x), __fadd_rn(an.p[1].y, dz.y));
    Pq = cfma_rn(dz, F, an.p[0]);
    Nq = cfma_rn(an.n[1], dz, an.n[0]);
  } else {
    const cf F2 = mk(__fadd_rn(an.p[2].x, dz.x), __fadd_rn(an.p[2].y, dz.y));
    Pq = cfma_rn(dz, cfma_rn(dz, F2, an.p[1]), an.p[0]);
    Nq = cfma_rn(dz, cfma_rn(an.n[2], dz, an.n[1]), an.n[0]);
  }
  const float q = __fmaf_rn(Pq.x, Pq.x, __fmul_rn(Pq.y, Pq.y));
  const float ip = rcp_fast(q);  // <= 1 ulp
  // V = N conj(P), pv = dz V, Delta w' = (ws + dz) + conj(pv) / |P|^2
  const cf V = mk(__fmaf_rn(Nq.x, Pq.x, __fmul_rn(Nq.y, Pq.y)), __fmaf_rn(Nq.y, Pq.x, -__fmul_rn(Nq.x, Pq.y)));
  const cf pv = mk(__fmaf_rn(dz.x, V.x, -__fmul_rn(dz.y, V.y)), __fmaf_rn(dz.x, V.y, __fmul_rn(dz.y, V.x)));
  const cf dw = mk(__fmaf_rn(pv.x, ip, __fadd_rn(an.ws.x, dz.x)), __fmaf_rn(-pv.y, ip, __fadd_rn(an.ws.y, dz.y)));
  if (dwo) *dwo = dw;
  if (dzo) *dzo = dz;
  if (eb) {
    const float md = sqrtf(abs2(dz)), aP = sqrtf(q), aU = sqrtf(abs2(V)) * ip;
    const float mn = sqrtf(abs2(an.n[0])) + md * (sqrtf(abs2(an.n[1])) + md * sqrtf(abs2(an.n[2])));
    const float mp = NL == 2 ? sqrtf(abs2(an.p[0])) + md * (sqrtf(abs2(an.p[1])) + md)
                             : sqrtf(abs2(an.p[0])) + md * (sqrtf(abs2(an.p[1])) + md * (sqrtf(abs2(an.p[2])) + md));
    constexpr float cN = NL == 2 ? 4.0f : 9.0f, cU = NL == 2 ? 28.0f : 49.0f;
    *eb = an.e0 + 2.0f * md * EPS32 * (cN * mn + cU * aU * mp) / aP;
  }
  return __fmaf_rn(dw.x, dw.x, __fmul_rn(dw.y, dw.y));
}

__device__ __forceinline__ cf tab_at(const float* tp, int o) {
  const float* t_ = tp + 4 * (o >> 1) + (o & 1);
  return mk(t_[0], t_[2]);
}

// A superblock of one row from the offsets wa, wb of its ends (db2 = |wb|^2):
// out: every ray between them is outside, inn: inside.  The distance of the
// chord from the source centre counts; its rounding, a few u of the
// coordinates, is added to rout.
__device__ __forceinline__ void chord_test(const AnchorF& an, const cf wa, const cf wb, float db2, bool& out, bool& inn) {
  const cf d = wb - wa;
  const float da2 = abs2(wa);
  const float tt = __saturatef(-(wa.x * d.x + wa.y * d.y) * rcp_fast(fmaxf(abs2(d), 1e-37f)));
  const cf cl = mk(fmaf(tt, d.x, wa.x), fmaf(tt, d.y, wa.y));
  const float ro = an.rout + 1e-6f * (fabsf(wa.x) + fabsf(wa.y) + fabsf(d.x) + fabsf(d.y));
  out = abs2(cl) > ro * ro;
  inn = fmaxf(da2, db2) < an.in2;
}

// A ray the group band left open: its own bound decides in FP32 where it can,
// else the FP64 distance (d2 is then replaced by its square).
template <int NL, class SH>
__device__ __forceinline__ bool ray_decide(SH& sh, const RayShared& rs, const Sec& S, float& d2, float eb, int irow,
                                           int lw) {
  const float rho32 = (float)sh.rho, rr32 = rho32 * rho32;
  const float X = 1.01f * (2.0f * rho32 * eb + eb * eb) + 8.0f * EPS32 * rr32;
  if (fabsf(d2 - rr32) > X) return d2 < rr32;
  const double d64 = sqrt(abs2(sec_offset64<NL>(sh.L.eps, sh.L.a, sh.wc, S, irow, lw)));
  if (rs.P.diag) atomicAdd(&sh.cnt[2], 1);
  d2 = (float)(d64 * d64);
  return d64 < sh.rho;
}

// A ray's spot factor: 1 - c inside the spot, else 1.  dw: the ray's offset
// from the source centre in the frame of anchor ai, with error bound eb; the
// spot centre's FP32 rounding adds 4 u rho.  Decided in FP32 outside the band,
// else from the FP64 offset as the oracle decides it.
template <int NL, int LAW, class SH>
__device__ __forceinline__ float spot_factor(SH& sh, const RayShared& rs, const Sec& S, int ai, const cf dw, float eb,
                                             int irow, int lw) {
  if (LAW == 0 || !sh.spot) return 1.f;
  const float spot_rr = sh.spot_rr32;
  const float spot_r2 = spot_rr * spot_rr;
  const float spot_f = sh.spot_f32;
  const float2 c = rs.P.spc[ai];
  const float ex = dw.x - c.x, ey = dw.y - c.y;
  const float q = fmaf(ex, ex, ey * ey);
  const float e = eb + 4.0f * EPS32 * (float)sh.rho;
  const float X = 1.01f * (2.0f * spot_rr * e + e * e) + 8.0f * EPS32 * spot_r2;
  if (fabsf(q - spot_r2) > X) return q < spot_r2 ? spot_f : 1.f;
  const cd d64 = sec_offset64<NL>(sh.L.eps, sh.L.a, sh.wc, S, irow, lw);
  const double fx = d64.x / sh.rho - sh.spot_x, fy = d64.y / sh.rho - sh.spot_y;
  return fx * fx + fy * fy < sh.spot_r * sh.spot_r ? spot_f : 1.f;
}

// One ray that the band left open, and one ray's spot factor: both need the
// ray's own error bound (ten square roots), so they are evaluated again out of
// line.
template <int NL, class SH>
__device__ __noinline__ bool ray_undecided(SH& sh, const RayShared& rs, const Sec& S, int ai, float tx, float ty,
                                           float ri_, float dri_, int irow, int lw, float* d2o) {
  float eb;
  float d2 = ray_eval<NL>(rs.P.anch[ai], tx, ty, ri_, dri_, &eb, nullptr);
  const bool in = ray_decide<NL>(sh, rs, S, d2, eb, irow, lw);
  *d2o = d2;
  return in;
}
template <int NL, int LAW, class SH>
__device__ __noinline__ float ray_spot(SH& sh, const RayShared& rs, const Sec& S, int ai, float tx, float ty, float ri_,
                                       float dri_, int irow, int lw) {
  float eb;
  cf dw;
  (void)ray_eval<NL>(rs.P.anch[ai], tx, ty, ri_, dri_, &eb, &dw);
  return spot_factor<NL, LAW>(sh, rs, S, ai, dw, eb, irow, lw);
}

// A sweep's spot test, for a group of rays (anchor ai): outside the band of X
// about the spot's edge the FP32 squared distance from the spot's centre
// decides, with the group's error bound in place of the ray's: the half-width
// hi2 - rho^2 of the group's band on d^2 exceeds 2 rho times that bound, whose
// coefficients are up to 2.3 times smaller than those of a ray's own (15 against
// 28, triple 22 against 49), so 2.5 times it is at least the ray's.  Inside the
// band ray_spot decides, so the factors are the same as a ray's own.  (With each ray's bound, ten square roots, and the set's
// constants converted from FP64 at every ray, a spotted set's sweep ran at a
// fifth of a plain one's speed.)
struct SpotBand { float2 c; float X; };
template <class SH>
__device__ __forceinline__ SpotBand spot_band(const SH& sh, const RayShared& rs, const AnchorF& an, int ai) {
  const float rho32 = (float)sh.rho;
  const float e = 1.25f * (an.hi2 - rho32 * rho32) / rho32 + 4.0f * EPS32 * rho32;
  const float rr = sh.spot_rr32;
  return {rs.P.spc[ai], an.lo2 < 0.f ? __int_as_float(0x7f800000)
                                     : 1.02f * (2.0f * rr * e + e * e) + 8.0f * EPS32 * rr * rr};
}
template <int NL, int LAW, class SH>
__device__ __forceinline__ float spot_sweep(SH& sh, const RayShared& rs, const Sec& S, int ai, const SpotBand& sp,
                                            const cf dw, float tx, float ty, float ri_, float dri_, int irow, int lw) {
  const float ex = dw.x - sp.c.x, ey = dw.y - sp.c.y;
  const float r2 = sh.spot_rr32 * sh.spot_rr32, q = fmaf(ex, ex, ey * ey);
  if (fabsf(q - r2) > sp.X) return q < r2 ? sh.spot_f32 : 1.f;
  return ray_spot<NL, LAW>(sh, rs, S, ai, tx, ty, ri_, dri_, irow, lw);
}

// Any column l of row irow (wrapped; beyond a non-periodic edge: outside,
// +inf): inside or not, its squared distance d2o and (fso, optional) its spot
// factor.
template <int NL, int LAW, class SH>
__device__ __forceinline__ bool ray_classify(SH& sh, const RayShared& rs, const Sec& S, int gi_, float ri_, float dri_,
                                             int irow, int l, float* d2o, float* fso) {
  const int NTH = rs.P.NTH;
  if (!S.periodic && (l < 0 || l >= NTH)) { *d2o = __int_as_float(0x7f800000); if (fso) *fso = 1.f; return false; }
  const int lw = l < 0 ? l + NTH : (l >= NTH ? l - NTH : l);
  const int mgrp = (int)__umulhi((unsigned int)lw, S.gmagic);
  const int ai = S.abase + gi_ * S.mth + mgrp;
  const AnchorF& an = rs.P.anch[ai];
  const cf t = tab_at(rs.P.tabf + 2 * S.tbase, lw - mgrp * S.gth);
  float d2 = ray_eval<NL>(an, t.x, t.y, ri_, dri_, nullptr, nullptr);
  bool in = d2 < an.lo2;
  if (!in && !(d2 > an.hi2)) in = ray_undecided<NL>(sh, rs, S, ai, t.x, t.y, ri_, dri_, irow, lw, &d2);
  *d2o = d2;
  if (LAW != 0 && fso) *fso = sh.spot ? ray_spot<NL, LAW>(sh, rs, S, ai, t.x, t.y, ri_, dri_, irow, lw) : 1.f;
  return in;
}

// The out-of-line parts of the ray stage.  Inlined (the queue's flush at four
// places) they pushed the sweeps out of the instruction cache: a fifth of its
// requests missed and 1.5 of 9 stall cycles per instruction were fetches.
// A halo column's flag:
template <int NL, int LAW, class SH>
__device__ __noinline__ unsigned halo_flag(SH& sh, const RayShared& rs, int b, int gi, float ri, float dri, int irow,
                                           int l) {
  float d2;
  return ray_classify<NL, LAW>(sh, rs, rs.sec[b], gi, ri, dri, irow, l, &d2, nullptr) ? 1u : 0u;
}

// an inside ray's share of the row beyond c0f: mu (c1f + c2f mu), plus s (c1h
// + c3h mu), s = mu^(1/2), when h (half-integer powers); fs: the spot factor
// (the row's count adds c0f, so a spotted ray adds fs (c0f + J) - c0f here)
template <class SH>
__device__ __forceinline__ float ray_share(const SH& sh, float c0f, float c1f, float c2f, float mu, bool h, float fs) {
  float J = mu * fmaf(c2f, mu, c1f);
  if (h) J = fmaf(mu * rsqrt_fast(mu), fmaf(sh.c3h, mu, sh.c1h), J);
  return fmaf(fs, J, -c0f * (1.0f - fs));
}

// The undecided rays of a lane's block [l0, l0 + nb): decides each (bit nb - 1
// - k of the result: column l0 + k inside) and adds the inside ones' shares to
// *sj.
template <int NL, int LAW, class SH>
__device__ __noinline__ unsigned undecided_rays(SH& sh, const RayShared& rs, int b, int aidx, int gbase, float ri,
                                                float dri, int irow, int l0, int nb, float* sj) {
  const Sec& S = rs.sec[b];
  const AnchorF& an = rs.P.anch[aidx];
  const float rho32 = (float)sh.rho, irho2 = 1.0f / (rho32 * rho32);
  unsigned bits = 0u;
  float s_ = *sj;
#pragma unroll 1
  for (int k = 0; k < nb; ++k) {
    const cf t = tab_at(rs.P.tabf + 2 * S.tbase, l0 + k - gbase);
    float eb;
    cf dw;
    float d2 = ray_eval<NL>(an, t.x, t.y, ri, dri, &eb, &dw);
    if (d2 < an.lo2 || d2 > an.hi2) continue;
    if (ray_decide<NL>(sh, rs, S, d2, eb, irow, l0 + k)) {
      bits |= 1u << (nb - 1 - k);
      s_ = __fadd_rn(s_, ray_share(sh, sh.c0f, sh.c1f, sh.c2f, sqrtf(fmaxf(__fmaf_rn(-d2, irho2, 1.0f), 1e-30f)),
                                   LAW != 0 && sh.half != 0,
                                   spot_factor<NL, LAW>(sh, rs, S, aidx, dw, eb, irow, l0 + k)));
    }
  }
  *sj = s_;
  return bits;
}

__device__ __forceinline__ void kahan_add(float2& acc, float term) {
  const float y = term - acc.y;
  const float tt = acc.x + y;
  acc.y = (tt - acc.x) - y;
  acc.x = tt;
}

// The product a b, rounded with the compensation in one operation.
__device__ __forceinline__ void kahan_add(float2& acc, float a, float b) {
  const float y = __fmaf_rn(a, b, -acc.y);
  const float tt = __fadd_rn(acc.x, y);
  acc.y = __fsub_rn(__fsub_rn(tt, acc.x), y);
  acc.x = tt;
}

// The weight W of a boundary point (Appendix A) from the signed squared
// distances sv of the rays l - 2 .. l + 2 (sv[2] the point, negative inside),
// and its weight WU under the uniform rule.  A crossing too close to the
// branch of f(delta) for FP32 is taken from the FP64 distances dist if they
// are given (inf beyond a non-periodic edge); else false comes back.
template <class SH>
__device__ __forceinline__ bool boundary_weight(SH& sh, const RayArgs& P, const float* sv, const double* dist,
                                                float* Wo, float* WU) {
  const float rho32 = (float)sh.rho, dcf = (float)P.delta_c;
  const float d2 = -sv[2];
  const bool Lin = signbit(sv[1]), Rin = signbit(sv[3]);
  float W;
  float fL = 0.f, fR = 0.f, uL = 0.f, uR = 0.f;
#pragma unroll 1
  for (int side = 0; side < 2; ++side) {
    const bool isL = side == 0;
    if (isL ? Lin : Rin) continue;
    const float vo = isL ? sv[1] : sv[3];
    float delta, fv;
    bool done = false;
    if (isinf(vo)) {
      delta = 0.5f;
      atomicOr(&sh.status, ICRS_ST_EDGE);
    } else {
      // stencil: entering (-2,-1,0,+1), exiting (-1,0,+1,+2); a grid edge cuts
      // one outer node off
      float ys[4], x0 = isL ? -2.0f : -1.0f;
      int n = 4;
#pragma unroll
      for (int c = 0; c < 4; ++c) ys[c] = isL ? sv[c] : sv[c + 1];
      if (isinf(ys[3])) n = 3;
      if (isinf(ys[0])) { ys[0] = ys[1]; ys[1] = ys[2]; ys[2] = ys[3]; x0 += 1.0f; --n; }
      if (n < 4) atomicOr(&sh.status, ICRS_ST_EDGE);
#pragma unroll
      for (int c = 0; c < 4; ++c) ys[c] = sqrtf(fabsf(ys[c]));
      const float x = crossing_solve<float>(ys, x0, n, sqrtf(d2), sqrtf(fabsf(vo)), isL ? -1.0f : 1.0f, rho32, 1e-5f,
                                            12);
      delta = isL ? -x : x;
      if (!P.uniform && fabsf(delta - dcf) < 2e-3f) {
        // branch of f(delta) too close to call in FP32
        if (!dist) return false;
        double ysd[4], x0d = isL ? -2.0 : -1.0;
        int nd = 4;
#pragma unroll
        for (int c = 0; c < 4; ++c) ysd[c] = isL ? dist[c] : dist[c + 1];
        if (isinf(ysd[3])) nd = 3;
        if (isinf(ysd[0])) { ysd[0] = ysd[1]; ysd[1] = ysd[2]; ysd[2] = ysd[3]; x0d += 1.0; --nd; }
        const double xd = crossing64(ysd, x0d, nd, dist[2], dist[isL ? 1 : 3], isL, x, sh.rho);
        const double dd = isL ? -xd : xd;
        delta = (float)dd;
        fv = (float)fdelta<double>(dd, P.delta_c, 0);
        done = true;
      }
    }
    if (!done) fv = fdelta<float>(delta, dcf, P.uniform);
    if (isL) { fL = fv; uL = delta + 0.5f; } else { fR = fv; uR = delta + 0.5f; }
  }
  *WU = Lin ? uR : (Rin ? uL : fmaxf(0.f, uL + uR - 1.0f));
  if (Lin) W = fR;
  else if (Rin) W = fL;
  else W = fmaxf(0.f, fL + fR - 1.0f);
  *Wo = W;
  return true;
}

// A boundary point's term beyond the I that the sweep added.  Literal rule: I
// (W - 1); split-profile rule: the limb value c0f with the uniform weight, the
// rest with f(delta) (a spot, fsc, scales the point's whole brightness).
template <int LAW, class SH>
__device__ __forceinline__ float point_term(const SH& sh, const RayArgs& P, const Sec& S, float ri_, float d2,
                                            float fsc, float W, float WU) {
  const float rho32 = (float)sh.rho, irho2 = 1.0f / (rho32 * rho32);
  // I(d) = c0f + c1f mu + c2f mu^2, mu^2 = x = 1 - d^2/rho^2
  const float x = fmaxf(fmaf(-d2, irho2, 1.0f), 1e-30f);
  const float mu = x * rsqrtf(x);
  const float c0f = sh.c0f;
  float I = fmaf(sh.c2f, x, fmaf(sh.c1f, mu, c0f));
  if (LAW != 0 && sh.half) I = fmaf(sqrtf(mu), fmaf(sh.c3h, mu, sh.c1h), I);
  const float rw = ri_ * S.bxw;
  return fsc * (P.split ? rw * (c0f * (WU - 1.0f) + (I - c0f) * (W - 1.0f)) : rw * I * (W - 1.0f));
}

// The warp's points whose crossing needs FP64: four at a time, the five
// stencil rays of a point on five of its eight lanes.
template <int NL, int LAW, class SH>
__device__ __noinline__ void flush_exact(SH& sh, RayShared& rs, int n) {
  const RayArgs& P = rs.P;
  const int lane = threadIdx.x & 31;
  const int2* xq = rs.xq[threadIdx.x >> 5];
  __syncwarp();
  for (int e0 = 0; e0 < n; e0 += 4) {
    const int e = e0 + (lane >> 3), k = lane & 7;
    const bool has = e < n;
    const int2 v2 = has ? xq[e] : make_int2(0, 0);
    const int v = v2.x;
    const Sec& S = rs.sec[v >> 25];
    const int irow = (v >> 13) & 4095, m = v & 8191;
    const int gi_ = irow / S.gr;
    const float dri_ = ((float)(irow - gi_ * S.gr) + 0.5f - 0.5f * (float)S.gr) * S.dr32;
    const float ri_ = __fadd_rn(S.rc[gi_], dri_);
    float s1 = 0.f, f1 = 1.f;
    double dd1 = 0.0;
    if (has && k < 5) {
      const int l = m - 2 + k;
      float d2;
      const bool in = ray_classify<NL, LAW>(sh, rs, S, gi_, ri_, dri_, irow, l, &d2, &f1);
      s1 = in ? __int_as_float(__float_as_int(d2) | 0x80000000) : d2;
      const int lw = l < 0 ? l + P.NTH : (l >= P.NTH ? l - P.NTH : l);
      dd1 = (!S.periodic && lw != l) ? __longlong_as_double(0x7ff0000000000000LL)
                                     : sqrt(abs2(sec_offset64<NL>(sh.L.eps, sh.L.a, sh.wc, S, irow, lw)));
    }
    float sv[5];
    double dist[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      sv[i] = __shfl_sync(0xffffffffu, s1, (lane & 24) + i);
      dist[i] = __shfl_sync(0xffffffffu, dd1, (lane & 24) + i);
    }
    const float fsc = __shfl_sync(0xffffffffu, f1, (lane & 24) + 2);
    if (has && k == 0) {
      float W, WU;
      (void)boundary_weight(sh, P, sv, dist, &W, &WU);
      if (P.diag) atomicAdd(&sh.cnt[3], 1);
      P.pterm[v2.y] = point_term<LAW>(sh, P, S, ri_, -sv[2], fsc, W, WU);
    }
  }
  __syncwarp();
}

// n <= 32 queued points q, one per lane: each re-evaluates its stencil (rays m
// - 2 .. m + 2, signed squared distances, negative inside) and writes its term
// to its place (the point's second word).  Points that need FP64 go to the
// warp's second queue; xn of its entries are taken, the new number comes back.
template <int NL, int LAW, class SH>
__device__ __noinline__ int flush_points(SH& sh, RayShared& rs, const int2* q, int n, int xn) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  bool exact = false;
  int2 v2 = make_int2(0, 0);
  if (lane < n) {
    v2 = q[lane];
    const int v = v2.x;
    float term = 0.f;
    const Sec& S = rs.sec[v >> 25];
    const int irow = (v >> 13) & 4095, m = v & 8191;
    const int gi_ = irow / S.gr;
    const float dri_ = ((float)(irow - gi_ * S.gr) + 0.5f - 0.5f * (float)S.gr) * S.dr32;
    const float ri_ = __fadd_rn(S.rc[gi_], dri_);
    float sv[5] = {0.f, 0.f, 0.f, 0.f, 0.f}, fsc = 1.f;
#pragma unroll 1
    for (int k = 0; k < 5; ++k) {  // (rolled: sv moves up one place per ray)
      float d2, fs;
      const bool in = ray_classify<NL, LAW>(sh, rs, S, gi_, ri_, dri_, irow, m - 2 + k, &d2, LAW != 0 ? &fs : nullptr);
      sv[0] = sv[1]; sv[1] = sv[2]; sv[2] = sv[3]; sv[3] = sv[4];
      sv[4] = in ? __int_as_float(__float_as_int(d2) | 0x80000000) : d2;
      if (LAW != 0 && k == 2) fsc = fs;
    }
    if (signbit(sv[2])) {
      float W, WU;
      if (boundary_weight(sh, rs.P, sv, nullptr, &W, &WU)) term = point_term<LAW>(sh, rs.P, S, ri_, -sv[2], fsc, W, WU);
      else exact = true;
    }
    rs.P.pterm[v2.y] = term;
  }
  unsigned todo = __ballot_sync(0xffffffffu, exact);
  while (todo) {
    if (xn == XQ) { flush_exact<NL, LAW>(sh, rs, XQ); xn = 0; }
    const int src = __ffs(todo) - 1;
    if (lane == src) rs.xq[threadIdx.x >> 5][xn] = v2;
    ++xn;
    todo &= todo - 1u;
  }
  __syncwarp();
  return xn;
}

// The warp's queued points: all q[0 .. n - 1] (n <= FQ) and the xn that need
// FP64.
template <int NL, int LAW, class SH>
__device__ __noinline__ void flush_all(SH& sh, RayShared& rs, const int2* q, int n, int xn) {
  for (; n > 0; n -= min(n, 32)) {
    const int m = min(n, 32);
    xn = flush_points<NL, LAW>(sh, rs, q + n - m, m, xn);
  }
  if (xn) flush_exact<NL, LAW>(sh, rs, xn);
}

// A task that has more boundary points than places: the n <= PCAP terms so far
// become one, in the first two places (as a float pair), and the next points
// take the places after them.  (Two images in one sector and whole rows to a
// task give 4 points a row, 128 a task.)  The terms are added in the order of
// the points, which is the task's own, so the sum does not depend on the warp
// that took the task.
constexpr int PGATHERED = 2;
__device__ __forceinline__ void gather_points(float* pterm, int n) {
  static_assert(PCAP == 64, "two terms a lane");
  const int lane = threadIdx.x & 31;
  double s = lane < n ? (double)pterm[lane] : 0.0;
  if (lane + 32 < n) s += (double)pterm[lane + 32];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) {
    const float h = (float)s;
    pterm[0] = h;
    pterm[1] = isfinite(h) ? (float)(s - (double)h) : 0.0f;
  }
  __syncwarp();
}

// What a warp has queued, in one register: its points (bits 0 .. 7), those that
// need FP64 (8 .. 15), and the places that its task's points have taken (16 up).
__device__ __forceinline__ int q_points(unsigned q) { return (int)(q & 255u); }
__device__ __forceinline__ int q_exact(unsigned q) { return (int)((q >> 8) & 255u); }
__device__ __forceinline__ int q_places(unsigned q) { return (int)(q >> 16); }

// Room for c <= 32 more points of a task.  One function for both reasons to
// flush: its call is inlined at every place that pushes points.
template <int NL, int LAW, class SH>
__device__ __noinline__ unsigned make_room(SH& sh, RayShared& rs, int task, int c, unsigned q) {
  const int2* const dq = reinterpret_cast<const int2*>(rs.P.wqueue) + (threadIdx.x >> 5) * FQ;
  if (q_places(q) + c > PCAP) {
    flush_all<NL, LAW>(sh, rs, dq, q_points(q), q_exact(q));
    gather_points(rs.P.pterm + task * PCAP, q_places(q));
    return (unsigned)PGATHERED << 16;
  }
  const int n = q_points(q) - 32, xn = flush_points<NL, LAW>(sh, rs, dq + n, 32, q_exact(q));
  return (q & 0xffff0000u) | (unsigned)(xn << 8) | (unsigned)n;
}

// The next batch of sectors (rs.b0 .. rs.b1 - 1, none left: b0 = b1): its
// anchors and offset tables.  dr.store(an, x) takes what the derivative keeps
// of an anchor besides, dr.columns its own tables.
struct NoDer {
  template <int NL> __device__ void store(int, const AnchorX<NL>&) const {}
  __device__ void columns(const RayShared&, int, int) const {}
};
template <int NL, int LAW, class SH, class DR>
__device__ __noinline__ void ray_tables(SH& sh, RayShared& rs, const DR& dr) {
  const int tid = threadIdx.x, NT = blockDim.x;
  const RayArgs& P = rs.P;
  const float rho32 = (float)sh.rho;
  const bool spot = LAW != 0 && sh.spot;
  const int nbox = sh.nbox;
  if (tid == 0) {
    int b = rs.b1, na = 0, nc = 0, nt = 0;
    rs.b0 = b;
    for (; b < nbox; ++b) {
      Sec& S = rs.sec[b];
      if (b > rs.b0 && (na + S.nanch > MAXANCH || nc + S.gth + 2 > P.tabcap ||
                        nt + S.ntask > P.tcap || (P.ccap && (b - rs.b0 + 1) * P.NTH > P.ccap)))
        break;
      S.abase = na; S.tbase = nc; S.cbase = (b - rs.b0) * P.NTH; S.task0 = nt;
      na += S.nanch; nc += S.gth + 2; nt += S.ntask;
    }
    rs.b1 = b; rs.nanch = na; rs.ncol = nc; rs.ntask = nt; rs.next = 0;
  }
  __syncthreads();
  const int b0 = rs.b0, b1 = rs.b1;
  for (int an = tid; an < rs.nanch; an += NT) {
    int b = b0;
    while (b + 1 < b1 && an >= rs.sec[b + 1].abase) ++b;
    const Sec& S = rs.sec[b];
    AnchorX<NL> x;
    P.anch[an] = make_anchor<NL>(S, sh.L.eps, sh.L.a, sh.wc, rho32, an - S.abase, x);
    if (spot) P.spc[an] = make_float2((float)(sh.rho * (x.cs * sh.spot_x + x.sn * sh.spot_y)),
                                      (float)(sh.rho * (x.cs * sh.spot_y - x.sn * sh.spot_x)));
    dr.store(an, x);
  }
  // offsets within a theta group, (cos d - 1, sin d) with d = (o + 1/2 -
  // gth/2) dth; column pairs (o, o + 1), o even, are stored as 16 bytes (x_o,
  // x_o+1, y_o, y_o+1), so that a pair's x and y load as two adjacent float2
  // (gth is even); one entry past the group for the last superblock's end
  for (int o = NT - 1 - tid; o < rs.ncol; o += NT) {
    int b = b0;
    while (b + 1 < b1 && o >= rs.sec[b + 1].tbase) ++b;
    const Sec& S = rs.sec[b];
    const float d = ((float)(o - S.tbase) + 0.5f - 0.5f * (float)S.gth) * S.dth32;
    float s, c;
    sincosf(d, &s, &c);
    const float sh2 = sinf(0.5f * d);
    P.tabf[4 * (o >> 1) + (o & 1)] = -2.0f * sh2 * sh2;
    P.tabf[4 * (o >> 1) + 2 + (o & 1)] = s;
  }
  dr.columns(rs, b0, b1);
  __syncthreads();
}

// Sum over the epoch's sectors of this thread's share (FP64), ICRS_ST_* bits
// into sh.status.  Out of line: inlined into the epoch loop its sweeps shared
// their registers with the root and sector phases.
template <int NL, int LAW, class SH>
__device__ __noinline__ double ray_stage(SH& sh, RayShared& rs) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int NT = blockDim.x, NW = NT >> 5;
  const RayArgs P = rs.P;
  const int NR = P.NR, NTH = P.NTH;
  const float rho32 = (float)sh.rho;
  const float c0f = sh.c0f, c1f = sh.c1f, c2f = sh.c2f;
  const float irho2 = 1.0f / (rho32 * rho32);
  float2 acc = make_float2(0.f, 0.f);  // Kahan sum of this thread
  const unsigned lt_mask = (1u << lane) - 1u;
  const AnchorF* const anf = P.anch;
  const float* const tabf = P.tabf;
  unsigned queued = 0u;  // see make_room
  const int nbox = sh.nbox;

  if (tid < nbox) sec_setup(rs.sec[tid], sh.box[tid], NR, NTH);
  if (tid == 0) rs.b1 = 0;
  __syncthreads();

  // the anchor as broadcast pairs for two columns at once (binary), with the
  // negated copies that the evaluation needs
  struct AnchorP { float2 wsx, wsy, n0x, nn0y, n1x, nn1x, nn1y, p0x, p0y, p1x, p1y; };
  auto pairs_of = [](const AnchorF& a) -> AnchorP {
    AnchorP r;
    r.wsx = make_float2(a.ws.x, a.ws.x);        r.wsy = make_float2(a.ws.y, a.ws.y);
    r.n0x = make_float2(a.n[0].x, a.n[0].x);    r.nn0y = make_float2(-a.n[0].y, -a.n[0].y);
    r.n1x = make_float2(a.n[1].x, a.n[1].x);    r.nn1x = make_float2(-a.n[1].x, -a.n[1].x);
    r.nn1y = make_float2(-a.n[1].y, -a.n[1].y);
    r.p0x = make_float2(a.p[0].x, a.p[0].x);    r.p0y = make_float2(a.p[0].y, a.p[0].y);
    r.p1x = make_float2(a.p[1].x, a.p[1].x);    r.p1y = make_float2(a.p[1].y, a.p[1].y);
    return r;
  };
  // rays of columns (l, l + 1) of one row with paired FP32 operations (binary
  // lens): component k is rounded exactly as ray_eval rounds ray l + k,
  // operation by operation, so both give the same bits.  The y parts of N and
  // V are carried negated, which leaves two sign changes (dz.y by a product,
  // P.y) of the six that the direct form needs.
  auto ray_eval2 = [&](const AnchorP& a, float2 tx, float2 ty, float2 ri2, float2 nri2, float2 dri2) -> float2 {
    const float2 dzx = __ffma2_rn(ri2, tx, dri2), dzy = __fmul2_rn(ri2, ty), ndzy = __fmul2_rn(nri2, ty);
    const float2 Fx = __fadd2_rn(a.p1x, dzx), Fy = __fadd2_rn(a.p1y, dzy);
    const float2 Px = __ffma2_rn(dzx, Fx, __ffma2_rn(ndzy, Fy, a.p0x));
    const float2 Py = __ffma2_rn(dzx, Fy, __ffma2_rn(dzy, Fx, a.p0y));
    const float2 nPy = make_float2(-Py.x, -Py.y);
    const float2 Nx = __ffma2_rn(a.n1x, dzx, __ffma2_rn(a.nn1y, dzy, a.n0x));
    const float2 nNy = __ffma2_rn(a.nn1x, dzy, __ffma2_rn(a.nn1y, dzx, a.nn0y));
    const float2 q = __ffma2_rn(Px, Px, __fmul2_rn(Py, Py));
    const float2 ip = make_float2(rcp_fast(q.x), rcp_fast(q.y));
    const float2 Vx = __ffma2_rn(Nx, Px, __fmul2_rn(nNy, nPy));
    const float2 nVy = __ffma2_rn(nNy, Px, __fmul2_rn(Nx, Py));
    const float2 pvx = __ffma2_rn(dzx, Vx, __fmul2_rn(dzy, nVy));
    const float2 npvy = __ffma2_rn(dzx, nVy, __fmul2_rn(ndzy, Vx));
    const float2 dwx = __ffma2_rn(pvx, ip, __fadd2_rn(a.wsx, dzx));
    const float2 dwy = __ffma2_rn(npvy, ip, __fadd2_rn(a.wsy, dzy));
    return __ffma2_rn(dwx, dwx, __fmul2_rn(dwy, dwy));
  };
  const float2 nirho22 = make_float2(-irho2, -irho2), one2 = make_float2(1.0f, 1.0f);
  const float2 c1f2 = make_float2(c1f, c1f), c2f2 = make_float2(c2f, c2f);
  // 1, which the compiler does not know: J + sj2 directly after J's product is
  // otherwise contracted to one operation, with another rounding than where a
  // select stands between them
  const float2 one_rt = make_float2(P.one, P.one);
  // the half-power coefficients, read only by the generic instantiation
  const float2 c1h2 = LAW == 1 ? make_float2(sh.c1h, sh.c1h) : one2;
  const float2 c3h2 = LAW == 1 ? make_float2(sh.c3h, sh.c3h) : one2;
  const bool spot = LAW != 0 && sh.spot, generic = LAW != 0 && sh.generic;

  for (;;) {
    // ---- the next batch of sectors: their anchors and offset tables
    ray_tables<NL, LAW>(sh, rs, NoDer{});
    const int b0 = rs.b0, b1 = rs.b1;
    if (b0 >= b1) break;

    // ---- tasks.  A warp takes the next one when it is free: with superblocks
    // their costs differ by what is skipped (handed out in a fixed order, a
    // third of a 1024 x 2048 epoch's ray time was waiting for the last warp).
    // The sums do not depend on who computed what: a task leaves its rows' and
    // its boundary points' terms in shared memory, and they are added
    // afterwards in a fixed order.
    int b = b0;
    for (;;) {
      int task = 0;
      if (lane == 0) task = atomicAdd(&rs.next, 1);
      task = __shfl_sync(0xffffffffu, task, 0);
      if (task >= rs.ntask) break;
      while (b + 1 < b1 && task >= rs.sec[b + 1].task0) ++b;
      const Sec& S = rs.sec[b];
      const int rbk = (task - S.task0) / S.nch, chk = task - S.task0 - rbk * S.nch;
      queued &= 0xffffu;  // no place taken yet
      const int i = rbk * 32 + lane;
      const bool rowok = i < NR;
      const int ii = rowok ? i : NR - 1;
      const int gi = ii / S.gr;
      const float fri = (float)(ii - gi * S.gr) + 0.5f - 0.5f * (float)S.gr;
      const float dri = __fmul_rn(fri, S.dr32), ri = __fmaf_rn(fri, S.dr32, S.rc[gi]);
      const int c0 = chk * S.ch, c1 = min(c0 + S.ch, NTH);
      const int gth = S.gth, sb = S.sb;
      const float* const tps = tabf + 2 * S.tbase;
      // the row's inside rays: their count, and the sums of I - c0f = mu (c1f
      // + c2f mu) of the scalar and of the paired evaluations
      int cnt = 0;
      float sj = 0.f;
      float2 sj2 = make_float2(0.f, 0.f);
      // inside flags: bit k = column l - 1 - k before column l; the left halo
      // column c0 - 1 first
      unsigned win = halo_flag<NL, LAW>(sh, rs, b, gi, ri, dri, ii, c0 - 1);
      float lo2g = 0.f, hi2g = 0.f;  // the current group's band
      unsigned band = 0u;            // bits of its width
      int aidx = 0;                  // and its anchor
      AnchorF ar;     // the anchor in registers (triple)
      AnchorP ap;     // the anchor as broadcast pairs (binary)
      // binary: the scalar evaluations read the anchor from the table
      auto anchor = [&]() -> const AnchorF& {
        if constexpr (NL == 2) return anf[aidx];
        else return ar;
      };
      [[maybe_unused]] SpotBand spb;  // the current group's spot test
      int gbase = 0;  // first column of the current group
      const float* tpf = tps;  // offsets of the current group: pair rows by column
      const float2 ri2 = make_float2(ri, ri), nri2 = make_float2(-ri, -ri), dri2 = make_float2(dri, dri);
      // queue the boundary points among bits of bm, bit j = column base - j
      auto push_bits = [&](unsigned bm, int base) {
        while (__any_sync(0xffffffffu, bm != 0u)) {
          const bool has = bm != 0u;
          const int m = base - (has ? __ffs(bm) - 1 : 0);
          bm &= bm - 1u;
          const unsigned hm = __ballot_sync(0xffffffffu, has);
          const int at = __popc(hm & lt_mask), c = __popc(hm);
          if (q_points(queued) > FQ - 32 || q_places(queued) + c > PCAP)
            queued = make_room<NL, LAW>(sh, rs, task, c, queued);
          if (has) reinterpret_cast<int2*>(rs.P.wqueue)[warp * FQ + q_points(queued) + at] = make_int2(pack_point(b, i, m), task * PCAP + q_places(queued) + at);
          queued += (unsigned)c * 0x10001u;
        }
      };
      // boundary centres among columns l0 - 1 .. l0 + nb - 2 (bit j = column
      // l0 + nb - 2 - j) after the block [l0, l0 + nb); the first block's
      // column c0 - 1 belongs to the previous chunk
      auto centres = [&](int nb, bool first) -> unsigned {
        unsigned bm = ((win & ~((win << 1) & (win >> 1))) >> 1) & ((1u << nb) - 1u);
        if (first) bm &= ~(1u << (nb - 1));
        return rowok ? bm : 0u;
      };
      auto add_in = [&](bool in, float mu, bool h, float fs) {
        sj = __fadd_rn(sj, in ? ray_share(sh, c0f, c1f, c2f, mu, h, fs) : 0.0f);
      };
      auto block_end = [&](int l0, int nb, bool first, bool unc) {
        unsigned bm = centres(nb, first);
        if (__any_sync(0xffffffffu, unc || bm != 0u)) {
          if (unc) {
            float s_ = sj;
            win |= undecided_rays<NL, LAW>(sh, rs, b, aidx, gbase, ri, dri, ii, l0, nb, &s_);
            sj = s_;
            bm = centres(nb, first);
          }
          push_bits(bm, l0 + nb - 2);
        }
        cnt += __popc(win & ((1u << nb) - 1u));
      };
      // one column: classify against the band, flag, and if inside add its
      // share (x > 5 u there, as d^2 < lo2 <= rho^2 (1 - 8 u)); hc:
      // std::true_type for the generic law (half-integer powers of mu or a
      // spot, checked at run time)
      auto col = [&](int l, float tx, float ty, bool& unc, auto hc) {
        cf dw;
        constexpr bool GEN = decltype(hc)::value;
        const float d2 = ray_eval<NL>(anchor(), tx, ty, ri, dri, nullptr, GEN ? &dw : nullptr);
        const bool in = d2 < lo2g;
        unc = unc || !(in || d2 > hi2g);
        win = (win << 1) | (in ? 1u : 0u);
        const float x = __fmaf_rn(-d2, irho2, 1.0f);
        if constexpr (GEN)
          add_in(in, __fmul_rn(x, rsqrt_fast(x)), sh.half != 0,
                 in && spot ? spot_sweep<NL, LAW>(sh, rs, S, aidx, spb, dw, tx, ty, ri, dri, ii, l) : 1.0f);
        else
          add_in(in, __fmul_rn(x, rsqrt_fast(x)), false, 1.0f);
      };
      // J of a column pair (no spot); hh: std::true_type adds the half-integer
      // powers s (c1h + c3h mu), s = mu^(1/2)
      auto share2 = [&](float2 d2, auto hh) -> float2 {
        const float2 x = __ffma2_rn(d2, nirho22, one2);
        const float2 mu = __fmul2_rn(x, make_float2(rsqrt_fast(x.x), rsqrt_fast(x.y)));
        float2 J = __fmul2_rn(mu, __ffma2_rn(c2f2, mu, c1f2));
        if constexpr (decltype(hh)::value) {
          const float2 sq = __fmul2_rn(mu, make_float2(rsqrt_fast(mu.x), rsqrt_fast(mu.y)));
          J = __ffma2_rn(sq, __ffma2_rn(c3h2, mu, c1h2), J);
        }
        return J;
      };
      // two columns (l, l + 1) with paired operations (binary lens); the pair
      // row t4 = (x_l, x_l+1, y_l, y_l+1).  v = d^2 - lo2 is negative exactly
      // for a ray certainly inside, and as unsigned bits it is at most the
      // band's width exactly for an undecided one: one shift per ray collects
      // the flags and one minimum the undecided rays.
      auto col2 = [&](const float4 t4, unsigned& umin, auto hh) {
        const float2 d2 = ray_eval2(ap, make_float2(t4.x, t4.y), make_float2(t4.z, t4.w), ri2, nri2, dri2);
        const float2 v = __fadd2_rn(d2, make_float2(-lo2g, -lo2g));
        const unsigned u0 = __float_as_uint(v.x), u1 = __float_as_uint(v.y);
        win = __funnelshift_l(u1, __funnelshift_l(u0, win, 1), 1);
        umin = min(umin, min(u0, u1));
        const float2 J = share2(d2, hh);
        sj2 = __fadd2_rn(sj2, make_float2(v.x < 0.0f ? J.x : 0.0f, v.y < 0.0f ? J.y : 0.0f));
      };
      int l = c0;
      bool first = true;
      while (l < c1) {
        const int mgrp = (int)__umulhi((unsigned int)l, S.gmagic);
        aidx = S.abase + gi * S.mth + mgrp;
        lo2g = anf[aidx].lo2;
        hi2g = anf[aidx].hi2;
        // (an empty band, lo2 < 0 and hi2 = inf: every ray, NaN too, is undecided)
        band = lo2g < 0.f ? 0x7fffffffu : __float_as_uint(hi2g - lo2g);
        if constexpr (NL == 2) ap = pairs_of(anf[aidx]);
        else ar = anf[aidx];
        if (spot) spb = spot_band(sh, rs, anf[aidx], aidx);
        gbase = mgrp * gth;
        tpf = tps - 2 * gbase;
        const int lend = min(gbase + gth, c1);
        const bool test = __any_sync(0xffffffffu, sb && anf[aidx].rout < __int_as_float(0x7f800000));
        cf wa = mk(0.f, 0.f);
        if (test) {
          const cf t = tab_at(tps, l - gbase);
          (void)ray_eval<NL>(anchor(), t.x, t.y, ri, dri, nullptr, &wa);
        }
        while (l < lend) {
          const int ls = test ? min(l + sb, lend) : lend;  // end of the superblock
          if (test) {
            cf wb;
            const cf t = tab_at(tps, ls - gbase);
            const float db2 = ray_eval<NL>(anchor(), t.x, t.y, ri, dri, nullptr, &wb);
            bool out, inn;
            chord_test(anf[aidx], wa, wb, db2, out, inn);
            wa = wb;
            const bool all_out = __all_sync(0xffffffffu, out);
            const bool all_in = !spot && ls - l >= 2 && __all_sync(0xffffffffu, inn);
            if (all_out || all_in) {
              // boundary points that this decides: the column before the
              // superblock, and its own first column if the one before is
              // outside (the edge of a sector)
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
              if (all_out) {
                win = 0u;
                l = ls;
                continue;
              }
              win = 0xffffffffu;
              cnt += ls - l;
              // binary: blocks of columns in pairs.  (The triple lens takes one
              // column at a time: its evaluation is twice as long, and with an
              // unrolled block the fetches held up the warps.  A curve of 2,000
              // epochs at 1024 x 2048: 108 ms unrolled, 76 now.)
              if constexpr (NL == 2) {
                auto in_block = [&](auto hh) {
#pragma unroll
                  for (int k = 0; k < KB; k += 2) {
                    const float4 t4 = *reinterpret_cast<const float4*>(tpf + 2 * (l + k));
                    const float2 J = share2(
                        ray_eval2(ap, make_float2(t4.x, t4.y), make_float2(t4.z, t4.w), ri2, nri2, dri2), hh);
                    sj2 = __ffma2_rn(J, one_rt, sj2);  // a sum: see one_rt
                  }
                };
#pragma unroll 1
                for (; l + KB <= ls; l += KB) {
                  if (LAW == 1 && generic) in_block(std::true_type{});
                  else in_block(std::false_type{});
                }
              }
#pragma unroll 1
              for (; l < ls; ++l) {
                const cf tl = tab_at(tps, l - gbase);
                const float x = __fmaf_rn(-ray_eval<NL>(anchor(), tl.x, tl.y, ri, dri, nullptr, nullptr), irho2, 1.0f);
                add_in(true, __fmul_rn(x, rsqrt_fast(x)), generic && sh.half != 0, 1.0f);
              }
              continue;
            }
          }
          while (l < ls) {
            const int nb = min(KB, ls - l);
            bool unc = false;
            // a full block, columns l + k, l + k + 1 from one 16-byte row (l +
            // k - gbase even); hc selects the half-power terms
            auto full_block = [&](auto hc) {
              [[maybe_unused]] unsigned umin = 0xffffffffu;
#pragma unroll 1
              for (int k = 0; k < KB; k += 2) {
                const float4 t4 = *reinterpret_cast<const float4*>(tpf + 2 * (l + k));
                if constexpr (NL == 2) {
                  col2(t4, umin, hc);
                } else {
                  col(l + k, t4.x, t4.z, unc, hc);
                  col(l + k + 1, t4.y, t4.w, unc, hc);
                }
              }
              if constexpr (NL == 2) unc = umin <= band;
            };
            // (a spot, or the half-integer powers outside the generic
            // instantiation's paired sweep: the scalar loop)
            if (nb == KB && !generic) {
              full_block(std::false_type{});
            } else if (LAW == 1 && NL == 2 && nb == KB && !spot) {
              full_block(std::true_type{});
            } else {
#pragma unroll 1
              for (int k = 0; k < nb; ++k) {
                const cf t = tab_at(tps, l + k - gbase);
                if (generic) col(l + k, t.x, t.y, unc, std::true_type{});
                else col(l + k, t.x, t.y, unc, std::false_type{});
              }
            }
            block_end(l, nb, first, unc);
            first = false;
            l += nb;
          }
        }
      }
      // right halo column c1: finalizes column c1 - 1
      win = (win << 1) | halo_flag<NL, LAW>(sh, rs, b, gi, ri, dri, ii, c1);
      push_bits(rowok ? (((win & ~((win << 1) & (win >> 1))) >> 1) & 1u) : 0u, c1 - 1);
      const float rowacc = c0f * (float)cnt + (sj + (sj2.x + sj2.y));
      P.rowp[task * 32 + lane] = ri * rowacc;
      if (lane == 0) P.pcnt[task] = q_places(queued);
    }
    flush_all<NL, LAW>(sh, rs, reinterpret_cast<const int2*>(rs.P.wqueue) + warp * FQ, q_points(queued), q_exact(queued));
    queued = 0u;
    __syncthreads();

    // ---- the sums, as a fixed assignment of the tasks would take them: thread
    // (warp, lane) adds the rows of tasks warp, warp + NW, ... of each sector,
    // and of these tasks' boundary points, 32 to a batch, its lane's, a batch
    // when the first point after it comes (a compensated sum rounds each term
    // together with what it carries, so its order shows in the tenth digit)
    for (int bb = b0; bb < b1; ++bb) {
      const Sec& S = rs.sec[bb];
      int n = 0, q = lane;         // points so far, this lane's next
      int pt_ = warp, base = 0;    // the task that holds it, its first point
      auto add_points = [&](int upto) {  // q while q < upto
        while (q < upto) {
          int c = P.pcnt[S.task0 + pt_];
          while (q >= base + c) { base += c; pt_ += NW; c = P.pcnt[S.task0 + pt_]; }
          kahan_add(acc, P.pterm[(S.task0 + pt_) * PCAP + q - base]);
          q += 32;
        }
      };
      for (int tk = warp; tk < S.ntask; tk += NW) {
        n += P.pcnt[S.task0 + tk];
        // whole batches that a later point has pushed out
        if (n > 32) add_points((n - 1) & ~31);
        if ((tk / S.nch) * 32 + lane < NR) kahan_add(acc, P.rowp[(S.task0 + tk) * 32 + lane], S.bxw);
      }
      add_points(n);
    }
  }
  return (double)acc.x - (double)acc.y;
}

}  // namespace icrs
