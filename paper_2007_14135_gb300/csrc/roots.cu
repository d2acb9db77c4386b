// Root form of the ULA scan (root-MUSIC; beyond the paper, which evaluates the spectrum on a grid).
// On the unit circle, with z = e^{j pi sin theta}, the scan's denominator is a Laurent polynomial:
//   a(theta)^H C a(theta) = sum_{l=-(M-1)}^{M-1} c_l z^l,   c_l = sum_{j-i=l} C_ij,
// and with C = sum_k w_k f_k f_k^H (the readout's factor columns and weights, Table 3),
//   c_l = sum_k w_k sum_n f_nk conj(f_{n+l,k}).
// z^{M-1} D(z) is a polynomial of degree 2M-2 whose roots pair up as z, 1/conj(z); the d roots with
// |z| <= 1 closest to the unit circle give the estimates theta = asin(arg(z) / pi).
//
// Roots by the Aberth-Ehrlich iteration (simultaneous Newton corrections with the repulsion sum
// over the other roots), all corrections computed from the previous iterate, started on the unit
// circle at angles 2 pi i / n + 0.4: first in FP32 on the rounded coefficients (to corrections of
// 1e-6 |z| or the FP32 rounding bound), then in FP64 from there; in FP64 a root counts as converged
// when its correction is below 1e-14 max(1, |z|) or when |p(z)| is within the rounding bound of its
// Horner evaluation,
// 8 n eps sum_t |a_t| |z|^t (clustered roots -- the pairs z, 1/conj(z) near the circle -- cannot be
// resolved further). A converged root keeps its value and takes no further correction; the
// iteration ends when all have converged, 400 iterations at most (else DOA_ENOCONV). Outside the unit
// circle p is evaluated as z^n q(1/z) with the reversed coefficients, so powers never overflow: with
// plain Horner a root beyond 20 or so (a small leading coefficient) put infinities into the FP32 phase,
// which then ran to its cap and left the FP64 phase to start from the circle.
// The coefficients are divided by the power of two of the largest one (the roots are the same), so the
// FP32 phase and the squares below stay in range whatever the factor's scale or the EV weights.
// One warp per (problem, algorithm) job: lanes own coefficients, then roots, then selected roots.
//
// Bound by FP64 issue (an FP64 warp instruction holds its sub-partition for 64 cycles), so the FP64
// iteration keeps the two Horner recurrences and what decides its stop in FP64, while the repulsion sum,
// which only steers the step, is taken in FP32 from the roots' leading parts and remainders (in FP64
// where that leaves its range: far roots, or two iterates that meet); the selection works in parallel
// lanes.
// Measured (2048 jobs of degree 30): 4.6 -> 0.61 ms (0.56 with the stop's bound in FP32).
#include <math_constants.h>

#include "doa_internal.cuh"

namespace doa {
namespace {

constexpr int kRootWarps = 4;
constexpr int kMaxDeg = 2 * kMaxM - 2;
constexpr int kRootsPerLane = (kMaxDeg + 31) / 32;
constexpr int kRootMaxIter = 400;
constexpr int kRootMaxIterF = 64;    // FP32 phase

struct RootShared {
  float2 af[kMaxDeg + 1];   // the coefficients rounded to FP32 (first phase)
  float amf[kMaxDeg + 1];
  float2 zf[kMaxDeg];       // FP32 roots; in the second phase the FP64 roots' leading parts
  float2 wf[kMaxDeg];       // FP32 corrections; in the second phase the FP64 roots' remainders
  double2 a[kMaxDeg + 1];   // polynomial coefficients, a[t] multiplies z^t
  double am[kMaxDeg + 1];   // |a_t| (for the rounding bound of the Horner evaluation)
  double2 z[kMaxDeg];       // current roots
  double2 w[kMaxDeg];       // corrections of this iteration
  int conv[kMaxDeg];        // root converged (its correction is no longer computed)
};

__device__ __forceinline__ float2 fcmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 fcadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 fcsub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 fcdiv(float2 a, float2 b) {
  const float inv = __frcp_rn(fmaf(b.x, b.x, b.y * b.y));
  return make_float2(fmaf(a.x, b.x, a.y * b.y) * inv, fmaf(a.y, b.x, -a.x * b.y) * inv);
}
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cdiv(double2 a, double2 b) {
  const double inv = __drcp_rn(b.x * b.x + b.y * b.y);
  return make_double2((a.x * b.x + a.y * b.y) * inv, (a.y * b.x - a.x * b.y) * inv);
}
__device__ __forceinline__ double2 crcp(double2 b) {   // 1 / b
  const double inv = __drcp_rn(b.x * b.x + b.y * b.y);
  return make_double2(b.x * inv, -b.y * inv);
}

struct RootJob {
  const double2 *F;   // factor, column-major, ld M
  const double *w;    // EV weights or null
  int M, Kf, Kn, kphd, kmn, alg, d;
};

__device__ __forceinline__ double root_weight(const RootJob &j, int c) {
  switch (j.alg) {
    case DOA_MUSIC: return c < j.Kn ? 1.0 : 0.0;
    case DOA_EV: return c < j.Kn ? (j.w ? j.w[c] : 1.0) : 0.0;
    case DOA_PHD: return c == j.kphd ? 1.0 : 0.0;
    case DOA_MN: return c == j.kmn ? 1.0 : 0.0;
    default: return c < j.Kf ? 1.0 : 0.0;
  }
}

// sum_{k != i} 1 / (z_i - z_k): in FP32 from the roots' leading parts and remainders; in FP64 when that is
// not finite (two iterates within 2^-48, or one beyond FP32's range) or was not asked for. An iterate
// equal to z_i adds nothing.
__device__ __forceinline__ double2 repulsion(const RootShared &sh, int i, int n, bool fp32) {
  if (fp32) {
    const float2 zh = sh.zf[i], zl = sh.wf[i];
    float2 rep = make_float2(0.f, 0.f);
    for (int k = 0; k < n; ++k) {
      if (k == i) continue;
      const float2 kh = sh.zf[k], kl = sh.wf[k];
      const float2 d = make_float2((zh.x - kh.x) + (zl.x - kl.x), (zh.y - kh.y) + (zl.y - kl.y));
      rep = fcadd(rep, fcdiv(make_float2(1.f, 0.f), d));
    }
    if (isfinite(rep.x) && isfinite(rep.y)) return make_double2((double)rep.x, (double)rep.y);
  }
  double2 rep = make_double2(0.0, 0.0);
  for (int k = 0; k < n; ++k) {
    const double2 d = csub(sh.z[i], sh.z[k]);
    if (k == i || (d.x == 0.0 && d.y == 0.0)) continue;
    const double2 r = crcp(d);
    rep = make_double2(rep.x + r.x, rep.y + r.y);
  }
  return rep;
}

// Writes the d angles (degrees, ascending) of one job to out; returns 0 or DOA_ENOCONV.
__device__ int root_music_warp(const RootJob &j, RootShared &sh, double *out) {
  const int lane = threadIdx.x & 31;
  const int M = j.M, n = 2 * M - 2;
  // coefficients: a[t] = c_{t - (M-1)}, c_{-l} = conj(c_l); lanes pair up on an l >= 0, each taking every
  // other column
  int top = 0;
  for (int l0 = 0; l0 < M; l0 += 16) {
    const int l = l0 + (lane >> 1);
    double cr = 0.0, ci = 0.0;
    for (int c = lane & 1; c < j.Kf && l < M; c += 2) {
      const double wc = root_weight(j, c);
      if (wc == 0.0) continue;
      const double2 *f = j.F + (size_t)c * M;
      double sr = 0.0, si = 0.0;
      for (int q = 0; q + l < M; ++q) {   // f_q conj(f_{q+l})
        const double2 x = f[q], y = f[q + l];
        sr = fma(x.x, y.x, fma(x.y, y.y, sr));
        si = fma(x.y, y.x, fma(-x.x, y.y, si));
      }
      cr = fma(wc, sr, cr);
      ci = fma(wc, si, ci);
    }
    cr += __shfl_xor_sync(0xffffffffu, cr, 1);
    ci += __shfl_xor_sync(0xffffffffu, ci, 1);
    if (l < M && (l > 0 || (lane & 1) == 0)) {   // the even lane writes c_l, the odd one c_{-l}
      const int t = (lane & 1) ? M - 1 - l : M - 1 + l;
      const double im = (lane & 1) ? -ci : (l == 0 ? 0.0 : ci);
      sh.a[t] = make_double2(cr, im);
      top = max(top, max(__double2hiint(cr) & 0x7fffffff, __double2hiint(im) & 0x7fffffff));
    }
  }
  top = __reduce_max_sync(0xffffffffu, top) >> 20;    // the largest coefficient's exponent field
  const int ex = top == 0 || top == 0x7ff ? 0 : 1023 - top;   // (zero or not finite: left as it is)
  __syncwarp();
  for (int t = lane; t <= n; t += 32) {
    const double2 c = make_double2(scalbn(sh.a[t].x, ex), scalbn(sh.a[t].y, ex));
    const double m = sqrt(c.x * c.x + c.y * c.y);
    sh.a[t] = c;
    sh.am[t] = m;
    sh.af[t] = make_float2((float)c.x, (float)c.y);
    sh.amf[t] = (float)m;
  }
  for (int i = lane; i < n; i += 32) {
    float s, c;
    sincosf(6.283185307179586f * (float)i / (float)n + 0.4f, &s, &c);
    sh.zf[i] = make_float2(c, s);
    sh.wf[i] = make_float2(0.f, 0.f);
    sh.conv[i] = 0;
  }
  __syncwarp();
  int st = DOA_ENOCONV;
  const double2 lead = sh.a[n];
  const bool usable = lead.x * lead.x + lead.y * lead.y > 0.0;
  // first phase, FP32 (the FP64 rate is 1/73 of FP32 here): corrections down to 1e-6 |z| or the
  // FP32 rounding bound of p(z); the FP64 phase then polishes the same roots
  if (usable) {
    for (int it = 0; it < kRootMaxIterF; ++it) {
      bool small = true;
      for (int i = lane; i < n; i += 32) {
        if (sh.conv[i]) continue;
        const float2 zi = sh.zf[i];
        const float zm2 = fmaf(zi.x, zi.x, zi.y * zi.y), zm = sqrtf(zm2);
        const bool outer = zm2 > 1.f;               // evaluate q(x) = x^n p(1/x) at x = 1/z
        const float2 x = outer ? fcdiv(make_float2(1.f, 0.f), zi) : zi;
        const float xm = outer ? 1.f / zm : zm;
        int t = outer ? 0 : n;
        const int dt = outer ? 1 : -1;
        float2 p = sh.af[t], dp = make_float2(0.f, 0.f);
        float pe = sh.amf[t];
        for (int k = 0; k < n; ++k) {
          t += dt;
          dp = fcadd(fcmul(dp, x), p);
          p = fcadd(fcmul(p, x), sh.af[t]);
          pe = fmaf(pe, xm, sh.amf[t]);
        }
        float2 rep = make_float2(0.f, 0.f);
        for (int k = 0; k < n; ++k) {
          if (k == i) continue;
          rep = fcadd(rep, fcdiv(make_float2(1.f, 0.f), fcsub(zi, sh.zf[k])));
        }
        // Newton ratio p / p': outside it is q / (x (n q - x q'))
        if (outer) dp = fcmul(x, fcsub(make_float2(n * p.x, n * p.y), fcmul(x, dp)));
        const float2 ratio = fcdiv(p, dp);
        const float2 wi = fcdiv(ratio, fcsub(make_float2(1.f, 0.f), fcmul(ratio, rep)));
        sh.wf[i] = wi;
        const float mag = sqrtf(fmaf(wi.x, wi.x, wi.y * wi.y)), res = sqrtf(fmaf(p.x, p.x, p.y * p.y));
        const bool ok = isfinite(mag) && (mag <= 1e-6f * fmaxf(1.f, zm) || res <= 8.f * n * 5.9604645e-08f * pe);
        small = small && ok;
        if (ok) sh.conv[i] = 1;
      }
      __syncwarp();
      for (int i = lane; i < n; i += 32) {
        sh.zf[i] = fcsub(sh.zf[i], sh.wf[i]);
        sh.wf[i] = make_float2(0.f, 0.f);
      }
      __syncwarp();
      if (__all_sync(0xffffffffu, small)) break;
    }
  }
  bool finite_start = true;
  for (int i = lane; i < n; i += 32) finite_start = finite_start && isfinite(sh.zf[i].x) && isfinite(sh.zf[i].y);
  finite_start = __all_sync(0xffffffffu, finite_start);
  for (int i = lane; i < n; i += 32) {
    if (finite_start) {
      sh.z[i] = make_double2((double)sh.zf[i].x, (double)sh.zf[i].y);
    } else {
      double s, c;
      sincos(2.0 * CUDART_PI * (double)i / (double)n + 0.4, &s, &c);
      sh.z[i] = make_double2(c, s);
      sh.zf[i] = make_float2((float)c, (float)s);
    }
    sh.wf[i] = make_float2((float)(sh.z[i].x - (double)sh.zf[i].x), (float)(sh.z[i].y - (double)sh.zf[i].y));
    sh.w[i] = make_double2(0.0, 0.0);
    sh.conv[i] = 0;
  }
  __syncwarp();
  if (usable) {
    for (int it = 0; it < kRootMaxIter; ++it) {
      bool small = true;
      for (int i = lane; i < n; i += 32) {
        if (sh.conv[i]) continue;                    // converged: no more correction
        const double2 zi = sh.z[i];
        const double r2 = zi.x * zi.x + zi.y * zi.y, zm = sqrt(r2);
        const bool outer = zm > 1.0;
        const double inv = outer ? __drcp_rn(r2) : 1.0;
        const double2 x = outer ? make_double2(zi.x * inv, -zi.y * inv) : zi;
        const double xm = zm * inv;
        int t = outer ? 0 : n;
        const int dt = outer ? 1 : -1;
        double2 p = sh.a[t], dp = make_double2(0.0, 0.0);
        double pe = sh.am[t];
        for (int k = 0; k < n; ++k) {                // Horner for p, p' and the bound sum |a_t| |x|^t
          t += dt;
          const double2 at = sh.a[t];
          dp = make_double2(fma(dp.x, x.x, fma(-dp.y, x.y, p.x)), fma(dp.x, x.y, fma(dp.y, x.x, p.y)));
          p = make_double2(fma(p.x, x.x, fma(-p.y, x.y, at.x)), fma(p.x, x.y, fma(p.y, x.x, at.y)));
          pe = fma(pe, xm, sh.am[t]);
        }
        const double2 rep = repulsion(sh, i, n, zm < 1e15);
        // Newton ratio p / p': outside it is z q / (n q - x q')
        if (outer) dp = csub(make_double2(n * p.x, n * p.y), cmul(x, dp));
        const double2 pdp = cdiv(p, dp), ratio = outer ? cmul(zi, pdp) : pdp;
        const double2 den = csub(make_double2(1.0, 0.0), cmul(ratio, rep));
        const double2 wi = cdiv(ratio, den);
        sh.w[i] = wi;
        const double mag = sqrt(wi.x * wi.x + wi.y * wi.y);
        const double res = sqrt(p.x * p.x + p.y * p.y);
        const bool ok = isfinite(mag) && isfinite(zm) && (mag <= 1e-14 * fmax(1.0, zm) || res <= 8.0 * n * 1.1102230246251565e-16 * pe);
        small = small && ok;
        if (ok) sh.conv[i] = 1;
      }
      __syncwarp();
      for (int i = lane; i < n; i += 32) {
        const double2 z = csub(sh.z[i], sh.w[i]);
        sh.z[i] = z;
        sh.zf[i] = make_float2((float)z.x, (float)z.y);
        sh.wf[i] = make_float2((float)(z.x - (double)sh.zf[i].x), (float)(z.y - (double)sh.zf[i].y));
        sh.w[i] = make_double2(0.0, 0.0);
      }
      __syncwarp();
      if (__all_sync(0xffffffffu, small)) {
        st = 0;
        break;
      }
    }
  }
  // the d roots with |z| <= 1 of largest modulus (lower index on a tie): d rounds of an arg-max over the
  // lanes' roots, moduli compared by their bits (all are >= 0)
  long long m[kRootsPerLane];
#pragma unroll
  for (int k = 0; k < kRootsPerLane; ++k) {
    const int i = lane + 32 * k;
    m[k] = -1;
    if (i < n) {
      const double2 zi = sh.z[i];
      const double r = sqrt(zi.x * zi.x + zi.y * zi.y);
      if (r <= 1.0) m[k] = __double_as_longlong(r);
    }
  }
  int ns = 0;
  int *taken = sh.conv;                     // root indices of the selection (the flags are done with)
  __syncwarp();
  for (int q = 0; q < j.d && st == 0; ++q) {
    long long best = -1;
    int bi = 1 << 30;
#pragma unroll
    for (int k = 0; k < kRootsPerLane; ++k)
      if (m[k] > best) {
        best = m[k];
        bi = lane + 32 * k;
      }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const long long ob = __shfl_xor_sync(0xffffffffu, best, off);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
      if (ob > best || (ob == best && oi < bi)) {
        best = ob;
        bi = oi;
      }
    }
    if (best < 0) break;
#pragma unroll
    for (int k = 0; k < kRootsPerLane; ++k)
      if (bi == lane + 32 * k) m[k] = -1;
    if (lane == 0) taken[q] = bi;
    ns = q + 1;
  }
  __syncwarp();
  double *sel = reinterpret_cast<double *>(sh.w);
  for (int q = lane; q < ns; q += 32) {
    const double2 zb = sh.z[taken[q]];
    const double sx = fmin(fmax(atan2(zb.y, zb.x) / CUDART_PI, -1.0), 1.0);
    sel[q] = asin(sx) * (180.0 / CUDART_PI);
  }
  __syncwarp();
  for (int q = lane; q < ns; q += 32) {     // ascending: every angle goes to its rank
    const double v = sel[q];
    int rank = 0;
    for (int k = 0; k < ns; ++k) rank += sel[k] < v || (sel[k] == v && k < q);
    out[rank] = v;
  }
  for (int q = ns + lane; q < j.d; q += 32) out[q] = CUDART_NAN;
  if (ns < j.d) st = DOA_ENOCONV;
  __syncwarp();
  return st;
}

__device__ __forceinline__ void roots_job(const uint8_t *plan, uint8_t *ws, int *status, RootShared *sh) {
  const PlanHeader *h = reinterpret_cast<const PlanHeader *>(plan);
  const int warp = threadIdx.x >> 5;
  const int job = blockIdx.x * kRootWarps + warp;
  if (job >= h->njobs) return;
  const PlanJob &jb = reinterpret_cast<const PlanJob *>(plan + h->off_job)[job];
  const PlanProblem &pp = reinterpret_cast<const PlanProblem *>(plan + h->off_prob)[jb.prob];
  if (!pp.p.root_angle || pp.p.d < 1) return;
  if (status[jb.prob] != 0) return;     // no decomposition to root
  RootJob j{};
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
  j.d = pp.p.d;
  const int st = root_music_warp(j, sh[warp], pp.p.root_angle + (size_t)jb.slot * pp.p.d);
  if (st && (threadIdx.x & 31) == 0) atomicCAS(status + jb.prob, 0, st);
}

// The refinement before it in the stream shares nothing it writes with this kernel, and its tail leaves
// most SMs idle: this kernel starts inside it (programmatic dependent launch) and ends after it, so that
// what follows in the stream finds both done. 2048 ULA and 512 circular-array estimates: 2.87 -> 2.61 ms
// (one after the other: refinement 1.35, root form 0.6 ms).
__global__ void __launch_bounds__(32 * kRootWarps) roots_batch_kernel(const uint8_t *plan, uint8_t *ws, int *status) {
  __shared__ RootShared sh[kRootWarps];
  roots_job(plan, ws, status, sh);
  end_after_previous();
}

__global__ void __launch_bounds__(32) roots_single_kernel(RootJob j, double *theta, int *info) {
  __shared__ RootShared sh;
  const int st = root_music_warp(j, sh, theta);
  if (threadIdx.x == 0) *info = st ? -st : 0;
}

}  // namespace

cudaError_t launch_roots_batch(const uint8_t *plan_dev, const PlanHeader &h, uint8_t *ws, int *status, cudaStream_t s) {
  if (h.nroots == 0 || h.njobs == 0) return cudaSuccess;
  const int grid = (h.njobs + kRootWarps - 1) / kRootWarps, block = 32 * kRootWarps;
  if (h.nrefine > 0) return launch_beside(roots_batch_kernel, grid, block, 0, s, plan_dev, ws, status);
  roots_batch_kernel<<<grid, block, 0, s>>>(plan_dev, ws, status);
  return cudaGetLastError();
}

cudaError_t launch_roots_single(const double2 *B, int M, int K, int d, double *theta, int *info, cudaStream_t s) {
  RootJob j{};
  j.F = B;
  j.M = M;
  j.Kf = K;
  j.Kn = K;
  j.kphd = j.kmn = -1;
  j.alg = -1;
  j.d = d;
  roots_single_kernel<<<1, 32, 0, s>>>(j, theta, info);
  return cudaGetLastError();
}

}  // namespace doa
