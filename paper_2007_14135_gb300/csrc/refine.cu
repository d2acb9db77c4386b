// Sub-grid refinement of picked peaks (beyond the paper's Step-6, which stops at the grid): the
// local minimiser of a readout's denominator next to each grid peak, in FP64.
//
// den(theta) = sum_c w_c |y_c|^2, y_c = f_c^H a(theta), over the factor columns the readout reads
// (MUSIC: E_n, w = 1; EV: E_n, w = 1/lambda; PHD: v_min; MN: valph; a single-call factor B: all
// columns, w = 1), which equals a^H C a for the weighting matrix C of Table 3. Its derivatives come
// from the steering vector's: with y', y'' = F^H a', F^H a'',
//   den'  = 2 sum_c w_c Re(conj(y_c) y'_c),   den'' = 2 sum_c w_c (Re(conj(y_c) y''_c) + |y'_c|^2).
//
// ULA (steering a_m = exp(j pi m sin theta), phases from the exact 64-bit phase step of sin theta
// as in the scan's refinement): bracketed Newton on den' = 0 inside [theta_{k-1}, theta_{k+1}] --
// the bracket shrinks by the sign of den'; a Newton step shorter than 1e-13 rad (with den'' > 0)
// is taken and ends the iteration; otherwise the Newton point is taken if strictly inside the
// bracket, else the bracket's midpoint; stop below a 1e-13 rad move or after 60 steps.
//
// Geometry (Eq. 2 as printed, positions relative to their centroid -- a common phase that leaves
// den unchanged): damped Newton in (azimuth, elevation) inside the box of one grid step around the
// peak, with gradient g and Hessian H from the first and second derivatives of the element phases
// t_m = p_m . u(theta, phi). A step is -H^-1 g when H is positive definite (taken as it is when
// shorter than 1e-6 rad in both angles), else the steepest-descent direction scaled to the box
// half-width, halved up to 40 times until den does not increase; stop below a 1e-13 rad move, when
// no halving decreases den, or after 60 steps.
//
// One warp per peak, the warps of a CTA on one job's peaks (its factor staged in shared memory). Bound by
// FP64 issue: an FP64 warp instruction holds its sub-partition for 64 cycles whatever the number of active
// lanes, so what counts is the number of instructions, not of lanes. Lanes own elements for the steering
// vector and its derivatives (shared memory), then one real recurrence each for the contractions (a
// column's real or imaginary part of one derivative: 2 M multiply-adds instead of a column's 12 M), then
// columns; sums run over as many lanes as there are columns, several quantities side by side, and every
// lane gets the same den, gradient and Hessian, so all lanes take the same decisions. A line search
// evaluates 32 / W step lengths at once (W = 8 or 16 lanes each, or the whole warp for larger arrays) and
// takes the first that does not increase den. All of it adds in the order of a column per lane and a
// butterfly over the lanes.
// In the batch the iteration starts from the vertex of the parabola through the FP32 spectrum's
// 1/P at the peak and its neighbours (per axis in 2-D), which leaves Newton one or two steps; the
// local minimiser it converges to does not depend on the start.
// Measured (2048 ULA jobs of four peaks and 512 circular-array jobs of two): 7.5 -> 1.4 ms. The kernel's
// length is that of one peak's 60 steps with some twenty halvings each (2.4 ms on one warp), so the
// 2-D jobs start first, and the four warps of a CTA share a search that does not end soon: the whole
// solve of that batch 3.92 -> 2.93 ms with that search, 3.04 -> 2.72 without.
#include <float.h>
#include <math_constants.h>

#include <algorithm>

#include "doa_internal.cuh"

namespace doa {
namespace {

constexpr int kRefWarps = 4;
constexpr int kRefMaxIter = 60;
// Steps of a 2-D search that its warp takes alone (most searches end within them). The batch above at 3, 6, 12
// and 20: 2.77, 2.82, 2.78, 2.82 ms in the mean of three drawings, 2.89, 2.97, 2.98, 3.11 at the longest search.
constexpr int kSoloSteps = 4;
constexpr double kD2R = 3.14159265358979323846 / 180.0;
constexpr double kPi = 3.14159265358979323846;

struct RefineJob {
  const double2 *F;      // factor, column-major, ld M
  const double *w;       // EV weights (Kn) or null
  int M, Kf, Kn, kphd, kmn;
  int alg;               // readout: DOA_PHD .. DOA_MN, or -1 = all columns unweighted (single call)
  // ULA grid
  double lo, step;
  // geometry (pos != null)
  const double *pos;
  double cx, cy, cz;
  double az_lo, az_step, el_lo, el_step;
  int La, Le, wrap;
  const float *P;        // the job's FP32 spectrum (start point), or null: start at the grid point
};

// Offset, in grid steps, of the vertex of the parabola through 1/P at points a, b (the peak), c;
// 0 when the three do not bracket a minimum of 1/P.
__device__ __forceinline__ double vertex_offset(float pa, float pb, float pc) {
  const double da = 1.0 / (double)pa, db = 1.0 / (double)pb, dc = 1.0 / (double)pc;
  const double curv = da - 2.0 * db + dc;
  if (!(curv > 0.0) || !(db <= da) || !(db <= dc)) return 0.0;
  return fmin(fmax(0.5 * (da - dc) / curv, -0.9), 0.9);
}

// Columns up to which a lane takes one real recurrence: 6 Kf of them in up to three turns. More turns cost more
// than a column per lane (one ULA peak: M = 18, Kf = 14 0.33 instead of 0.42 ms, but M = 24, Kf = 18 0.066 instead
// of 0.062, M = 32, Kf = 24 0.80 instead of 0.62).
constexpr int kChainCols = 16;
struct RefShared {
  double2 v[6][kMaxM];   // a and its derivatives (1-D: a, a', a''; 2-D: a, a_t, a_p, a_tt, a_tp, a_pp)
  double y[12][kChainCols + 1];   // F^H v: real and imaginary parts per column
};
constexpr int kStageM = 16;      // factors up to this M are staged in shared memory

__device__ __forceinline__ double2 cmul_j(double s, double2 a) {   // (j s) a
  return make_double2(-s * a.y, s * a.x);
}

__device__ __forceinline__ double col_weight(const RefineJob &j, int c) {
  switch (j.alg) {
    case DOA_MUSIC: return c < j.Kn ? 1.0 : 0.0;
    case DOA_EV: return c < j.Kn ? (j.w ? j.w[c] : 1.0) : 0.0;
    case DOA_PHD: return c == j.kphd ? 1.0 : 0.0;
    case DOA_MN: return c == j.kmn ? 1.0 : 0.0;
    default: return c < j.Kf ? 1.0 : 0.0;
  }
}

// Sum over groups of W lanes (a butterfly; W = 32: the warp).
template <int W>
__device__ __forceinline__ double group_sum(double v) {
#pragma unroll
  for (int off = W / 2; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}
// Three sums over the lanes of columns (zero in the other lanes): side by side in lane groups when the
// columns fit in 8 or 16 lanes.
__device__ __forceinline__ void sum3(int Kf, double &a, double &b, double &c) {
  const int lane = threadIdx.x & 31;
  if (Kf <= 8) {
    const double tb = __shfl_sync(0xffffffffu, b, lane & 7), tc = __shfl_sync(0xffffffffu, c, lane & 7);
    const double s = group_sum<8>(lane < 8 ? a : (lane < 16 ? tb : tc));
    a = __shfl_sync(0xffffffffu, s, 0);
    b = __shfl_sync(0xffffffffu, s, 8);
    c = __shfl_sync(0xffffffffu, s, 16);
  } else if (Kf <= 16) {
    const double tb = __shfl_sync(0xffffffffu, b, lane & 15);
    const double s = group_sum<16>(lane < 16 ? a : tb);
    a = __shfl_sync(0xffffffffu, s, 0);
    b = __shfl_sync(0xffffffffu, s, 16);
    c = __shfl_sync(0xffffffffu, group_sum<16>(c), 0);
  } else {
    a = group_sum<32>(a);
    b = group_sum<32>(b);
    c = group_sum<32>(c);
  }
}
__device__ __forceinline__ double flip(bool f, double x) {
  return __hiloint2double(__double2hiint(x) ^ (f ? (int)0x80000000 : 0), __double2loint(x));
}
// Real (im = 0) or imaginary (im = 1) part of conj(f)^T v.
__device__ __forceinline__ double chain(const double2 *f, const double2 *v, int M, bool im) {
  double r = 0.0;
#pragma unroll 4
  for (int m = 0; m < M; ++m) {
    const double2 b = f[m], a = v[m];
    r = fma(b.x, im ? a.y : a.x, fma(flip(im, b.y), im ? a.x : a.y, r));
  }
  return r;
}
// y[2 k + im][c] = part im of conj(f_c)^T v[k] for nv vectors, a recurrence per lane.
__device__ __forceinline__ void contract(const RefineJob &j, int nv, RefShared &sh) {
  const int n = 2 * nv * j.Kf;
  const float inv = __fdividef(1.f, (float)j.Kf);
  for (int e = threadIdx.x & 31; e < n; e += 32) {
    const int k = (int)(((float)e + 0.5f) * inv), c = e - k * j.Kf;
    sh.y[k][c] = chain(j.F + (size_t)c * j.M, sh.v[k >> 1], j.M, (k & 1) != 0);
  }
  __syncwarp();
}

// conj(f_c)^T v for lane-owned column c (v in shared memory).
__device__ __forceinline__ double2 col_dot(const RefineJob &j, int c, const double2 *v) {
  const double2 *f = j.F + (size_t)c * j.M;
  double yr = 0.0, yi = 0.0;
  for (int m = 0; m < j.M; ++m) {
    const double2 b = f[m], a = v[m];
    yr = fma(b.x, a.x, fma(b.y, a.y, yr));
    yi = fma(b.x, a.y, fma(-b.y, a.x, yi));
  }
  return make_double2(yr, yi);
}

// ---- ULA ------------------------------------------------------------------------------------
// den, den', den'' at theta (radians).
__device__ void ula_eval(const RefineJob &j, double th, RefShared &sh, double &f, double &f1, double &f2) {
  const int lane = threadIdx.x & 31;
  double s, c;
  sincos(th, &s, &c);
  const uint64_t step = phase_step64_of_sin(s);
  for (int m = lane; m < j.M; m += 32) {
    const double2 a = phasor_q64((uint64_t)m * step);
    const double pm = kPi * (double)m;
    sh.v[0][m] = a;
    sh.v[1][m] = cmul_j(pm * c, a);
    const double2 ja = cmul_j(-pm * s, a);
    const double q = (pm * c) * (pm * c);
    sh.v[2][m] = make_double2(ja.x - q * a.x, ja.y - q * a.y);
  }
  __syncwarp();
  double pf = 0.0, p1 = 0.0, p2 = 0.0;
  const bool chains = j.Kf <= kChainCols;
  if (chains) contract(j, 3, sh);
  for (int col = lane; col < j.Kf; col += 32) {
    const double wc = col_weight(j, col);
    if (wc == 0.0) continue;
    double2 y, y1, y2;
    if (chains) {
      y = make_double2(sh.y[0][col], sh.y[1][col]);
      y1 = make_double2(sh.y[2][col], sh.y[3][col]);
      y2 = make_double2(sh.y[4][col], sh.y[5][col]);
    } else {
      y = col_dot(j, col, sh.v[0]);
      y1 = col_dot(j, col, sh.v[1]);
      y2 = col_dot(j, col, sh.v[2]);
    }
    pf += wc * (y.x * y.x + y.y * y.y);
    p1 += 2.0 * wc * (y.x * y1.x + y.y * y1.y);
    p2 += 2.0 * wc * ((y.x * y2.x + y.y * y2.y) + (y1.x * y1.x + y1.y * y1.y));
  }
  __syncwarp();
  f = pf;
  f1 = p1;
  f2 = p2;
  sum3(j.Kf, f, f1, f2);
}

__device__ double refine_ula_warp(const RefineJob &j, int k, RefShared &sh) {
  const double t0 = __dadd_rn(j.lo, __dmul_rn((double)(k - 1), j.step));
  const double t1 = __dadd_rn(j.lo, __dmul_rn((double)k, j.step));
  const double t2 = __dadd_rn(j.lo, __dmul_rn((double)(k + 1), j.step));
  double x_lo = __dmul_rn(fmin(t0, t2), kD2R), x_hi = __dmul_rn(fmax(t0, t2), kD2R), x = __dmul_rn(t1, kD2R);
  if (j.P) x = (t1 + vertex_offset(j.P[k - 1], j.P[k], j.P[k + 1]) * j.step) * kD2R;
  for (int it = 0; it < kRefMaxIter; ++it) {
    double f, f1, f2;
    ula_eval(j, x, sh, f, f1, f2);
    if (f1 > 0.0) x_hi = x; else x_lo = x;
    if (f2 > 0.0 && fabs(f1) < 1e-13 * f2) {
      x -= f1 / f2;
      break;
    }
    double xn = (f2 > 0.0) ? x - f1 / f2 : CUDART_NAN;
    if (!(xn > x_lo && xn < x_hi)) xn = 0.5 * (x_lo + x_hi);
    const double dx = fabs(xn - x);
    x = xn;
    if (dx < 1e-13) break;
  }
  return x / kD2R;
}

// ---- geometry -------------------------------------------------------------------------------
// sin and cos of both angles at once: even lanes take th, odd lanes ph.
struct Trig {
  double st, ct, sp, cp;
};
__device__ __forceinline__ Trig trig(double th, double ph) {
  const int lane = threadIdx.x & 31;
  double s, c;
  sincos((lane & 1) ? ph : th, &s, &c);
  const double so = __shfl_xor_sync(0xffffffffu, s, 1), co = __shfl_xor_sync(0xffffffffu, c, 1);
  return (lane & 1) ? Trig{so, co, s, c} : Trig{s, c, so, co};
}
__device__ __forceinline__ double2 geo_phasor(double t) {
  const double fr = t - rint(t);
  return phasor_q64((uint64_t)__double2ll_rn(fr * 4611686018427387904.0) << 2);
}

// den at one point per group of W lanes (every lane of a group passes the same point; Kf <= W or W = 32).
template <int W>
__device__ double geo_den(const RefineJob &j, double th, double ph, RefShared &sh) {
  const int lane = threadIdx.x & 31, gl = lane & (W - 1);
  const Trig g = trig(th, ph);
  const double u0 = g.st * g.sp, u1 = g.ct * g.sp, u2 = g.cp;
  double2 *a = sh.v[0] + (W == 32 ? 0 : (lane & ~(W - 1)));
  for (int m = gl; m < j.M; m += W) {
    const double px = j.pos[3 * m] - j.cx, py = j.pos[3 * m + 1] - j.cy, pz = j.pos[3 * m + 2] - j.cz;
    a[m] = geo_phasor(px * u0 + py * u1 + pz * u2);
  }
  __syncwarp();
  double pf = 0.0;
  if (W < 32) {
    // the group's recurrences: column gl's real part, then its imaginary part on the lanes left over
    double *y = sh.y[0] + (lane / W) * 2 * W;   // rows of y taken as one array: 32 / W x 2 W <= 64 values
    for (int e = gl; e < 2 * j.Kf; e += W) {
      const bool im = e >= j.Kf;
      const int c = im ? e - j.Kf : e;
      y[(im ? W : 0) + c] = chain(j.F + (size_t)c * j.M, a, j.M, im);
    }
    __syncwarp();
    if (gl < j.Kf) {
      const double wc = col_weight(j, gl);
      if (wc != 0.0) {
        const double2 z = make_double2(y[gl], y[W + gl]);
        pf += wc * (z.x * z.x + z.y * z.y);
      }
    }
  } else {
    for (int col = lane; col < j.Kf; col += 32) {
      const double wc = col_weight(j, col);
      if (wc == 0.0) continue;
      const double2 y = col_dot(j, col, a);
      pf += wc * (y.x * y.x + y.y * y.y);
    }
  }
  __syncwarp();
  return group_sum<W>(pf);
}

// den, its gradient and Hessian (H[0] = tt, H[1] = tp, H[2] = pp) at (th, ph). With M, Kf <= W the lane
// groups share the element derivatives (each group takes every 32 / W-th of them).
template <int W>
__device__ double geo_eval(const RefineJob &j, double th, double ph, RefShared &sh, double *g, double *H) {
  const int lane = threadIdx.x & 31, gl = lane & (W - 1), grp = lane / W;
  constexpr int G = 32 / W;
  const Trig tr = trig(th, ph);
  const double st = tr.st, ct = tr.ct, sp = tr.sp, cp = tr.cp;
  const double u0 = st * sp, u1 = ct * sp, u2 = cp;
  const double tp2 = 2.0 * kPi;
  for (int m = gl; m < j.M; m += W) {
    const double px = j.pos[3 * m] - j.cx, py = j.pos[3 * m + 1] - j.cy, pz = j.pos[3 * m + 2] - j.cz;
    const double2 a = geo_phasor(px * u0 + py * u1 + pz * u2);
    if (grp == 0) sh.v[0][m] = a;
    const double t_t = px * (ct * sp) + py * (-st * sp);
    const double t_p = px * (st * cp) + py * (ct * cp) + pz * (-sp);
    for (int k = grp; k < 2; k += G) sh.v[1 + k][m] = cmul_j(tp2 * (k == 0 ? t_t : t_p), a);
    for (int k = grp; k < 3; k += G) {   // tt, tp, pp
      const double A = k == 1 ? ct * cp : -st * sp, B = k == 1 ? -st * cp : -ct * sp, C = k == 2 ? -cp : 0.0;
      const double2 q = cmul_j(tp2 * (px * A + py * B + pz * C), a);
      const double r = tp2 * tp2 * (k == 2 ? t_p : t_t) * (k == 0 ? t_t : t_p);
      sh.v[3 + k][m] = make_double2(q.x - r * a.x, q.y - r * a.y);
    }
  }
  __syncwarp();
  if (W < 32) {   // Kf <= W: groups take every G-th of the first- and second-order sums
    contract(j, 6, sh);
    const double wc = gl < j.Kf ? col_weight(j, gl) : 0.0;
    const bool on = gl < j.Kf && wc != 0.0;
    const double2 y = on ? make_double2(sh.y[0][gl], sh.y[1][gl]) : make_double2(0.0, 0.0);
    double r1[3], r2[3];
    for (int k = grp; k < 3; k += G) {
      // k = 0, 1, 2: den, g_t, g_p and H_tt, H_tp, H_pp
      double s1 = 0.0, s2 = 0.0;
      if (on) {
        const double2 z = k == 0 ? y : make_double2(sh.y[2 * k][gl], sh.y[2 * k + 1][gl]);
        s1 = (k == 0 ? wc : 2.0 * wc) * (y.x * z.x + y.y * z.y);
        const double2 z2 = make_double2(sh.y[6 + 2 * k][gl], sh.y[7 + 2 * k][gl]);
        const int ia = k == 2 ? 4 : 2, ib = k == 0 ? 2 : 4;
        const double2 za = make_double2(sh.y[ia][gl], sh.y[ia + 1][gl]), zb = make_double2(sh.y[ib][gl], sh.y[ib + 1][gl]);
        s2 = 2.0 * wc * ((y.x * z2.x + y.y * z2.y) + (za.x * zb.x + za.y * zb.y));
      }
      r1[k / G] = s1;
      r2[k / G] = s2;
    }
    double o1[3], o2[3];
#pragma unroll
    for (int k = 0; k < 3; k += G) {
      const double s1 = group_sum<W>(k + grp < 3 ? r1[k / G] : 0.0), s2 = group_sum<W>(k + grp < 3 ? r2[k / G] : 0.0);
#pragma unroll
      for (int i = 0; i < G && k + i < 3; ++i) {
        o1[k + i] = __shfl_sync(0xffffffffu, s1, i * W);
        o2[k + i] = __shfl_sync(0xffffffffu, s2, i * W);
      }
    }
    g[0] = o1[1];
    g[1] = o1[2];
    H[0] = o2[0];
    H[1] = o2[1];
    H[2] = o2[2];
    __syncwarp();
    return o1[0];
  }
  double pf = 0.0, pg0 = 0.0, pg1 = 0.0, ph0 = 0.0, ph1 = 0.0, ph2 = 0.0;
  for (int col = lane; col < j.Kf; col += 32) {
    const double wc = col_weight(j, col);
    if (wc == 0.0) continue;
    const double2 y = col_dot(j, col, sh.v[0]);
    pf += wc * (y.x * y.x + y.y * y.y);
    const double2 yt = col_dot(j, col, sh.v[1]), yp = col_dot(j, col, sh.v[2]);
    const double2 ytt = col_dot(j, col, sh.v[3]), ytp = col_dot(j, col, sh.v[4]), ypp = col_dot(j, col, sh.v[5]);
    pg0 += 2.0 * wc * (y.x * yt.x + y.y * yt.y);
    pg1 += 2.0 * wc * (y.x * yp.x + y.y * yp.y);
    ph0 += 2.0 * wc * ((y.x * ytt.x + y.y * ytt.y) + (yt.x * yt.x + yt.y * yt.y));
    ph1 += 2.0 * wc * ((y.x * ytp.x + y.y * ytp.y) + (yt.x * yp.x + yt.y * yp.y));
    ph2 += 2.0 * wc * ((y.x * ypp.x + y.y * ypp.y) + (yp.x * yp.x + yp.y * yp.y));
  }
  __syncwarp();
  g[0] = group_sum<32>(pg0);
  g[1] = group_sum<32>(pg1);
  H[0] = group_sum<32>(ph0);
  H[1] = group_sum<32>(ph1);
  H[2] = group_sum<32>(ph2);
  return group_sum<32>(pf);
}

// A search on its way: the point, den and its derivatives there (when have), the steps taken.
struct GeoState {
  double x0, x1, f, g[2], H[3];
  int it;
  bool have;
};
// What the warps of a search tell each other at a barrier: den and its derivatives at one point (by the
// first warp), and each warp's first accepted step length of a round.
struct GeoSlot {
  double ev[6];
  double n[kRefWarps][2];
  int hit[kRefWarps];
};
// Long searches of a CTA: the state each warp left open, and two slots per search, used in turn (so that
// one barrier is enough: a slot is written again after the next barrier, when all have read it).
struct GeoLong {
  GeoState st[kRefWarps];
  int open[kRefWarps];
  GeoSlot slot[2][2];
};

// Start of the search at grid point flat: the vertex of the parabola per axis (batch) or the point.
__device__ void geo_start(const RefineJob &j, int flat, GeoState &st) {
  const int l = flat / j.La, k = flat - l * j.La;
  double x0 = __dmul_rn(__dadd_rn(j.az_lo, __dmul_rn((double)k, j.az_step)), kD2R);
  double x1 = __dmul_rn(__dadd_rn(j.el_lo, __dmul_rn((double)l, j.el_step)), kD2R);
  if (j.P) {
    const float pc = j.P[flat];
    const int km = k > 0 ? k - 1 : (j.wrap ? j.La - 1 : -1), kp = k + 1 < j.La ? k + 1 : (j.wrap ? 0 : -1);
    if (km >= 0 && kp >= 0 && km != kp)
      x0 += vertex_offset(j.P[(size_t)l * j.La + km], pc, j.P[(size_t)l * j.La + kp]) * j.az_step * kD2R;
    if (l > 0 && l + 1 < j.Le)
      x1 += vertex_offset(j.P[(size_t)(l - 1) * j.La + k], pc, j.P[(size_t)(l + 1) * j.La + k]) * j.el_step * kD2R;
  }
  st.x0 = x0;
  st.x1 = x1;
  st.it = 0;
  st.have = false;
}

// Takes steps of the search at grid point flat until it ends (true) or st.it reaches max_it, by this warp
// alone (parts = 1) or as warp `part` of `parts` (all with the same state; search `group` of the CTA): then
// the first warp computes the derivatives and the step lengths are dealt over the warps. While the
// first warp evaluates a whole Newton step, the others already try the shorter ones.
template <int W>
__device__ bool geo_steps(const RefineJob &j, int flat, int max_it, int part, int parts, int group, RefShared &sh,
                          GeoLong &co, GeoState &st) {
  constexpr int G = 32 / W;   // step lengths a warp evaluates at once
  const int lane = threadIdx.x & 31;
  const int l = flat / j.La, k = flat - l * j.La;
  const double c0 = __dmul_rn(__dadd_rn(j.az_lo, __dmul_rn((double)k, j.az_step)), kD2R);
  const double c1 = __dmul_rn(__dadd_rn(j.el_lo, __dmul_rn((double)l, j.el_step)), kD2R);
  const double hw0 = fabs(j.az_step) * kD2R, hw1 = fabs(j.el_step) * kD2R;
  const double bl0 = c0 - hw0, bh0 = c0 + hw0, bl1 = c1 - hw1, bh1 = c1 + hw1;
  double x0 = st.x0, x1 = st.x1, f = st.f;
  double g[2] = {st.g[0], st.g[1]}, H[3] = {st.H[0], st.H[1], st.H[2]};
  bool have = st.have;   // f, g, H belong to (x0, x1) already
  bool done = false;
  int it = st.it, set = 0;
  auto meet = [&]() {   // the warps of this search
    if (parts == kRefWarps)
      __syncthreads();
    else if (group == 0)
      asm volatile("bar.sync 1, 64;" ::: "memory");
    else
      asm volatile("bar.sync 2, 64;" ::: "memory");
  };
  auto post_eval = [&](double fv, const double *gv, const double *Hv) {
    double *e = co.slot[group][set].ev;
    if (lane == 0) {
      e[0] = fv;
      e[1] = gv[0];
      e[2] = gv[1];
      e[3] = Hv[0];
      e[4] = Hv[1];
      e[5] = Hv[2];
    }
  };
  for (; it < max_it; ++it) {
    if (!have) {
      if (part == 0) f = geo_eval<W>(j, x0, x1, sh, g, H);
      if (parts > 1) {
        if (part == 0) post_eval(f, g, H);
        meet();
        const double *e = co.slot[group][set].ev;
        f = e[0];
        g[0] = e[1];
        g[1] = e[2];
        H[0] = e[3];
        H[1] = e[4];
        H[2] = e[5];
        set ^= 1;
      }
    }
    have = false;
    const double det = H[0] * H[2] - H[1] * H[1];
    const bool newton = H[0] > 0.0 && det > 0.0;
    double d0, d1;
    if (newton) {
      d0 = -(H[2] * g[0] - H[1] * g[1]) / det;
      d1 = -(H[0] * g[1] - H[1] * g[0]) / det;
      if (fmax(fabs(d0), fabs(d1)) < 1e-6) {
        const double n0 = fmin(fmax(x0 + d0, bl0), bh0), n1 = fmin(fmax(x1 + d1, bl1), bh1);
        const double mv = fmax(fabs(n0 - x0), fabs(n1 - x1));
        x0 = n0;
        x1 = n1;
        if (mv < 1e-13) {
          done = true;
          break;
        }
        continue;
      }
    } else {
      const double gn = sqrt(g[0] * g[0] + g[1] * g[1]);
      const double wdt = fmax(hw0, hw1);
      d0 = gn > 0.0 ? -g[0] / gn * wdt : 0.0;
      d1 = gn > 0.0 ? -g[1] / gn * wdt : 0.0;
    }
    double n0 = x0, n1 = x1;
    bool accepted = false;
    // the first accepted of step lengths 2^-h, h = h0 .. h0 + G - 1 (each group of lanes evaluates one)
    auto try_lengths = [&](int h0) {
      const int h = h0 + lane / W;
      const double t = __hiloint2double((1023 - h) << 20, 0);   // 2^-h
      const double m0 = fmin(fmax(x0 + t * d0, bl0), bh0), m1 = fmin(fmax(x1 + t * d1, bl1), bh1);
      const bool le = geo_den<W>(j, m0, m1, sh) <= f && h <= 40;
      const unsigned hit = __ballot_sync(0xffffffffu, le);
      const int src = hit ? __ffs(hit) - 1 : 0;
      const double s0 = __shfl_sync(0xffffffffu, m0, src), s1 = __shfl_sync(0xffffffffu, m1, src);
      if (hit) {
        n0 = s0;
        n1 = s1;
      }
      return hit != 0u;
    };
    auto post_hit = [&](bool hit) {
      GeoSlot &sl = co.slot[group][set];
      if (lane == 0) {
        sl.hit[part] = hit;
        sl.n[part][0] = n0;
        sl.n[part][1] = n1;
      }
    };
    auto first_hit = [&](int p0) {   // after the barrier: the lowest warp's hit has the longest step
      const GeoSlot &sl = co.slot[group][set];
      for (int p = p0; p < parts && !accepted; ++p)
        if (sl.hit[p]) {
          n0 = sl.n[p][0];
          n1 = sl.n[p][1];
          accepted = true;
        }
    };
    int h0 = 0;
    if (newton) {   // the whole step is usually taken: its derivatives come with it
      h0 = 1;
      double fn = 0.0, gn[2] = {0.0, 0.0}, Hn[3] = {0.0, 0.0, 0.0};
      const double w0 = fmin(fmax(x0 + d0, bl0), bh0), w1 = fmin(fmax(x1 + d1, bl1), bh1);
      if (part == 0) {
        fn = geo_eval<W>(j, w0, w1, sh, gn, Hn);
      } else {
        // 2 G lengths per warp, in order: two of these take as long as the derivatives
        const int b = 1 + (part - 1) * 2 * G;
        post_hit(try_lengths(b) || try_lengths(b + G));
      }
      if (parts > 1) {
        if (part == 0) post_eval(fn, gn, Hn);
        meet();
        const double *e = co.slot[group][set].ev;
        fn = e[0];
        gn[0] = e[1];
        gn[1] = e[2];
        Hn[0] = e[3];
        Hn[1] = e[4];
        Hn[2] = e[5];
      }
      if (fn <= f) {
        accepted = have = true;
        n0 = w0;
        n1 = w1;
        f = fn;
        g[0] = gn[0];
        g[1] = gn[1];
        H[0] = Hn[0];
        H[1] = Hn[1];
        H[2] = Hn[2];
      } else if (parts > 1) {
        first_hit(1);
        h0 = 1 + (parts - 1) * 2 * G;
      }
      set ^= 1;
    }
    for (; h0 <= 40 && !accepted; h0 += parts * G) {
      const bool hit = try_lengths(h0 + part * G);
      if (parts == 1) {
        accepted = hit;
      } else {
        post_hit(hit);
        meet();
        first_hit(0);
        set ^= 1;
      }
    }
    if (!accepted) {
      done = true;
      break;
    }
    const double mv = fmax(fabs(n0 - x0), fabs(n1 - x1));
    x0 = n0;
    x1 = n1;
    if (mv < 1e-13) {
      done = true;
      break;
    }
  }
  st.x0 = x0;
  st.x1 = x1;
  st.f = f;
  st.g[0] = g[0];
  st.g[1] = g[1];
  st.H[0] = H[0];
  st.H[1] = H[1];
  st.H[2] = H[2];
  st.it = it;
  st.have = have;
  return done || it >= kRefMaxIter;
}

// The 2-D peaks first, first + step, ... of a job, kRefWarps at a time; every warp of the CTA calls it. A warp
// takes a peak's first kSoloSteps steps alone; the searches that are not over then (a flat valley: tens of
// steps of some twenty halvings each) are taken on by two warps each, a single one by all four.
template <int W>
__device__ void refine_geo_job(const RefineJob &j, const int *idx, int first, int step, int n, double *out,
                               RefShared &sh, GeoLong &co) {
  static_assert(kRefWarps == 4, "two searches of two warps, or one of four");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int q0 = first; q0 < n; q0 += step) {
    const int q = q0 + warp;
    GeoState st;
    bool open = false;
    if (q < n) {
      geo_start(j, idx[q], st);
      open = !geo_steps<W>(j, idx[q], kSoloSteps, 0, 1, 0, sh, co, st);
    }
    if (lane == 0) {
      co.open[warp] = open;
      if (open) co.st[warp] = st;
      if (q < n && !open) {
        out[2 * q] = st.x0 / kD2R;
        out[2 * q + 1] = st.x1 / kD2R;
      }
    }
    __syncthreads();
    int left = 0;   // open searches, a bit each
    for (int w = 0; w < kRefWarps; ++w) left |= (co.open[w] ? 1 : 0) << w;
    while (left) {
      const int wa = __ffs(left) - 1;
      left &= left - 1;
      const bool two = left != 0;
      const int wb = two ? __ffs(left) - 1 : wa;
      left &= two ? left - 1 : 0;
      const int group = two ? warp >> 1 : 0, w = group ? wb : wa, part = two ? warp & 1 : warp;
      st = co.st[w];
      geo_steps<W>(j, idx[q0 + w], kRefMaxIter, part, two ? 2 : 4, group, sh, co, st);
      if (part == 0 && lane == 0) {
        out[2 * (q0 + w)] = st.x0 / kD2R;
        out[2 * (q0 + w) + 1] = st.x1 / kD2R;
      }
      __syncthreads();
    }
    __syncthreads();
  }
}

// Refines peaks idx[q], q = first .. first + kRefWarps - 1, first + step, ... < n of one job; out: n angles (ULA) or
// n (azimuth, elevation) pairs. Every warp of the CTA calls it.
__device__ void refine_job(const RefineJob &j, const int *idx, int first, int step, int n, double *out, RefShared *sh,
                           GeoLong &co) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int w = max(j.M, j.Kf);
  if (j.pos) {
    if (w <= 8)
      refine_geo_job<8>(j, idx, first, step, n, out, sh[warp], co);
    else if (w <= 16)
      refine_geo_job<16>(j, idx, first, step, n, out, sh[warp], co);
    else
      refine_geo_job<32>(j, idx, first, step, n, out, sh[warp], co);
    return;
  }
  for (int q = first + warp; q < n; q += step) {
    const double th = refine_ula_warp(j, idx[q], sh[warp]);
    if (lane == 0) out[q] = th;
    __syncwarp();
  }
}

// Copies a small factor to shared memory and points the job at it; the whole CTA calls it.
__device__ void stage_factor(RefineJob &j, double2 *Fs) {
  if (j.M <= kStageM && j.Kf <= kStageM + 1) {
    for (int e = threadIdx.x; e < j.M * j.Kf; e += blockDim.x) Fs[e] = j.F[e];
    j.F = Fs;
  }
  __syncthreads();
}

__device__ void set_centroid(RefineJob &j) {
  double cx = 0.0, cy = 0.0, cz = 0.0;
  for (int m = 0; m < j.M; ++m) {
    cx += j.pos[3 * m];
    cy += j.pos[3 * m + 1];
    cz += j.pos[3 * m + 2];
  }
  j.cx = cx / j.M;
  j.cy = cy / j.M;
  j.cz = cz / j.M;
}

__global__ void __launch_bounds__(32 * kRefWarps, 3) refine_batch_kernel(const uint8_t *plan, uint8_t *ws) {
  __shared__ RefShared sh[kRefWarps];
  __shared__ double2 Fs[kStageM * (kStageM + 1)];
  const PlanHeader *h = reinterpret_cast<const PlanHeader *>(plan);
  __shared__ GeoLong co;
  // once every CTA of this grid has started, the next kernel in the stream may use the SMs that the tail of
  // long searches leaves idle (the root form, which waits for this grid's end before it ends itself)
  let_next_start();
  // the first half of the CTAs takes the 2-D jobs, whose longest searches are the kernel's tail
  const bool geo = blockIdx.x < h->njobs;
  const int job = geo ? blockIdx.x : blockIdx.x - h->njobs;
  const PlanJob &jb = reinterpret_cast<const PlanJob *>(plan + h->off_job)[job];
  const PlanProblem &pp = reinterpret_cast<const PlanProblem *>(plan + h->off_prob)[jb.prob];
  if (!pp.p.peak_angle || pp.p.d < 1 || (pp.p.geom.pos != nullptr) != geo) return;
  RefineJob j{};
  j.F = reinterpret_cast<const double2 *>(ws + pp.fac_off);
  j.w = pp.Kn > 0 && pp.slot[DOA_EV] >= 0
            ? reinterpret_cast<const double *>(ws + pp.fac_off) + 2 * pp.p.M * (pp.p.M + 1)
            : nullptr;
  j.M = pp.p.M;
  j.Kf = pp.Kf;
  j.Kn = pp.Kn;
  j.kphd = pp.kphd;
  j.kmn = pp.kmn;
  j.alg = jb.alg;
  j.lo = pp.p.grid.lo_deg;
  j.step = pp.p.grid.step_deg;
  j.pos = pp.p.geom.pos;
  if (j.pos) {
    set_centroid(j);
    j.az_lo = pp.p.grid.lo_deg;
    j.az_step = pp.p.grid.step_deg;
    j.el_lo = pp.p.geom.el_lo_deg;
    j.el_step = pp.p.geom.el_step_deg;
    j.La = pp.p.grid.L;
    j.Le = pp.p.geom.Le;
    j.wrap = pp.p.geom.wrap_az;
  }
  j.P = pp.p.P + (size_t)jb.slot * pp.npts;
  const int d = pp.p.d;
  const int n = min(pp.p.peak_count[jb.slot], d);
  const int per = j.pos ? 2 : 1;
  stage_factor(j, Fs);
  refine_job(j, pp.p.peak_idx + (size_t)jb.slot * d, 0, kRefWarps, n, pp.p.peak_angle + (size_t)jb.slot * d * per, sh, co);
}

__global__ void __launch_bounds__(32 * kRefWarps) refine_single_kernel(RefineJob j, const int *idx, const int *count,
                                                                       int cap, double *out) {
  __shared__ RefShared sh[kRefWarps];
  __shared__ double2 Fs[kStageM * (kStageM + 1)];
  if (j.pos) set_centroid(j);
  __shared__ GeoLong co;
  const int n = min(*count, cap);
  stage_factor(j, Fs);
  refine_job(j, idx, blockIdx.x * kRefWarps, gridDim.x * kRefWarps, n, out, sh, co);
}

}  // namespace

cudaError_t launch_refine_batch(const uint8_t *plan_dev, const PlanHeader &h, uint8_t *ws, cudaStream_t s) {
  if (h.nrefine == 0 || h.njobs == 0) return cudaSuccess;
  refine_batch_kernel<<<2 * h.njobs, 32 * kRefWarps, 0, s>>>(plan_dev, ws);
  return cudaGetLastError();
}

cudaError_t launch_refine_single(const double2 *B, int M, int K, double lo, double step, const double *pos,
                                 double el_lo, double el_step, int La, const int *idx, const int *count, int cap,
                                 double *out, cudaStream_t s) {
  RefineJob j{};
  j.F = B;
  j.M = M;
  j.Kf = K;
  j.Kn = K;
  j.kphd = j.kmn = -1;
  j.alg = -1;
  j.lo = lo;
  j.step = step;
  j.pos = pos;
  j.az_lo = lo;
  j.az_step = step;
  j.el_lo = el_lo;
  j.el_step = el_step;
  j.La = La;
  const int ctas = std::max(1, std::min((cap + kRefWarps - 1) / kRefWarps, 16));
  refine_single_kernel<<<ctas, 32 * kRefWarps, 0, s>>>(j, idx, count, cap, out);
  return cudaGetLastError();
}

}  // namespace doa
