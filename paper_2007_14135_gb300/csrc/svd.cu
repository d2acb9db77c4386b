// Step-2 of Table 2 taken as an SVD of the snapshot matrix X itself (the paper computes Step-2 with
// a Jacobi SVD, Sec. 4.2): one-sided Jacobi (Hestenes) on the M rows of X, so R = X X^H / N is
// never formed and the small singular values keep their relative accuracy.
//
// GPU form: one cooperative launch. The rows are rotated in place in an FP64 copy Y of X (workspace).
//   1. pass: one streaming pass over Y on all CTAs that applies the accumulated rotation V of the last
//      sweeps (Y <- V^H Y; the first pass promotes X) and forms the Gram matrix G = Y Y^H in FP64
//      (partial sums per CTA, then summed in a fixed order, a warp per entry);
//   2. sweeps: CTA 0 runs row-cyclic sweeps of rotations on G itself (G <- J^H G J for each pair, the
//      Hermitian Jacobi rotation built from alpha = G_pp, beta = G_qq, gamma = G_pq) and records them;
//   3. rows: a warp per row of V and of U applies the recorded rotations (a rotation mixes two columns,
//      so the rows are independent).
// The iteration stops after the first sweep that rotates nothing on a Gram matrix formed afresh from
// the rows: then every off-diagonal entry of it meets the threshold, exactly the stopping rule of the
// row-by-row form, and S_k^2 = G_kk. While off-diagonal entries above 1e-4 sqrt(alpha beta) are still
// met and the diagonal spans less than 1e4, the next sweep goes on from the rotated G (whose entries
// then hold to 1e-12 of their scale); from there on every sweep starts from fresh rows, as it
// does throughout for graded or rank-deficient X.
//
// Why this shape. An FP64 warp instruction holds its sub-partition for 64 cycles here (measured,
// whatever the number of active lanes), so the row-cyclic sweep is bound by the serial chain of its
// rotations. Pairs of equal p + q are disjoint and every pair that (p, q) depends on in row-cyclic
// order has a smaller p + q, so the sweep runs in 2M - 3 levels of simultaneous rotations (29 instead
// of 120 steps at M = 16, 125 instead of 2016 at M = 64) with the same results up to rounding. One
// launch instead of two per sweep also spares the launches left over after convergence.
// Measured (a call): M = 16, N = 4096 in 6.3 -> 0.69 ms, M = 64, N = 16384 in 131 -> 8.8 ms against two
// kernels per sweep with one rotation after the other. A level at M = 16 takes about 4600 cycles: 1900
// for the rotations' FP64 chain, 400 for the diagonal, 2000 for the element updates; at M = 64 the
// element updates are bound by one SM's FP64 rate (8200 of 11100 cycles).
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>
#include <math_constants.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "doa.h"
#include "doa_internal.cuh"

namespace doa {
namespace {

constexpr int kSvdThreads = 256;
constexpr int kSvdT = 32;              // snapshots per chunk
constexpr int kSvdMaxBlocks = 256;     // pass CTAs (partial Gram blocks) at most
constexpr int kSvdMaxE = (kMaxM * (kMaxM + 1) / 2 + kSvdThreads - 1) / kSvdThreads;   // Gram entries per thread

constexpr int kSvdInner = 8;           // sweeps on one Gram matrix at most (room for their records)
constexpr int kSvdPolls = 1 << 24;     // polls of a grid barrier before it gives up (seconds)

struct SvdState {
  unsigned bar;   // arrivals at the grid barriers
  int abort;      // a barrier's wait ran out: everybody leaves
  int cmd;        // what CTA 0 decided: recorded sweeps to apply, or 0: outputs written
  int pad;
};

struct SvdRot {
  double c, sr, si;   // cosine and sigma = s e^{j phi}; c = 0: the pair was not rotated
};

struct SvdLayout {
  int64_t off_state, off_G, off_V, off_U, off_part, off_Y, bytes;
};

inline int64_t align16(int64_t x) { return (x + 15) / 16 * 16; }

SvdLayout svd_layout(int M, int N) {
  SvdLayout l{};
  const int64_t E = (int64_t)M * (M + 1) / 2;
  static_assert(kSvdInner * sizeof(SvdRot) <= kSvdMaxBlocks * sizeof(double2), "records fit in the partial sums");
  l.off_state = 0;
  l.off_G = 64;
  l.off_V = l.off_G + align16((int64_t)M * M * 16);
  l.off_U = l.off_V + align16((int64_t)M * M * 16);
  l.off_part = l.off_U + align16((int64_t)M * M * 16);
  l.off_Y = l.off_part + align16((int64_t)kSvdMaxBlocks * E * 16);
  l.bytes = l.off_Y + align16((int64_t)M * N * 16);
  return l;
}

// Row i and column j of the upper-triangle entry e (row-major over i <= j).
__device__ __forceinline__ void tri_index(int e, int M, int &i, int &j) {
  int r = 0, left = e;
  while (left >= M - r) {
    left -= M - r;
    ++r;
  }
  i = r;
  j = r + left;
}

// Barrier over the grid (cooperative launch: all CTAs are resident). False when the wait ran out, here
// or in another CTA: the caller leaves the kernel.
__device__ bool grid_barrier(SvdState *st, unsigned &phase) {
  phase += gridDim.x;
  __syncthreads();
  int ok = 1;
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(&st->bar, 1u);
    ok = 0;
    for (int i = 0; i < kSvdPolls; ++i) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&st->bar) : "memory");
      if (v >= phase) {
        ok = 1;
        break;
      }
      if (*(volatile int *)&st->abort) break;
      __nanosleep(40);
    }
    if (!ok) atomicExch(&st->abort, 1);
    __threadfence();
  }
  return __syncthreads_and(ok) != 0;
}

// One pass: Y <- V^H Y (first: Y <- X promoted to FP64) chunk by chunk, and the CTA's partial
// Gram sums G_ij = sum_t y_i(t) conj(y_j(t)), i <= j, over its chunks.
__device__ void svd_pass(const void *X, bool c128, bool first, int ldx, int M, int N, uint8_t *ws, const SvdLayout &lay,
                         uint8_t *smem) {
  double2 *S0 = reinterpret_cast<double2 *>(smem);         // M x kSvdT source chunk
  double2 *S1 = S0 + M * kSvdT;                            // M x kSvdT rotated chunk
  double2 *Vs = S1 + M * kSvdT;                            // M x M rotation (row-major)
  double2 *Y = reinterpret_cast<double2 *>(ws + lay.off_Y);
  const int tid = threadIdx.x;
  if (!first) {
    const double2 *V = reinterpret_cast<const double2 *>(ws + lay.off_V);
    for (int e = tid; e < M * M; e += kSvdThreads) Vs[e] = __ldcg(&V[e]);
  }
  const int E = M * (M + 1) / 2;
  int ei[kSvdMaxE], ej[kSvdMaxE];
  double2 acc[kSvdMaxE];
#pragma unroll
  for (int k = 0; k < kSvdMaxE; ++k) {
    const int e = tid + k * kSvdThreads;
    ei[k] = ej[k] = 0;
    if (e < E) tri_index(e, M, ei[k], ej[k]);
    acc[k] = make_double2(0.0, 0.0);
  }
  const int nchunks = (N + kSvdT - 1) / kSvdT;
  for (int c = blockIdx.x; c < nchunks; c += gridDim.x) {
    const int64_t t0 = (int64_t)c * kSvdT;
    const int cnt = (int)(N - t0 < kSvdT ? N - t0 : kSvdT);
    __syncthreads();   // the previous chunk's Gram sums have finished reading S1
    for (int e = tid; e < M * kSvdT; e += kSvdThreads) {
      const int i = e / kSvdT, t = e % kSvdT;
      double2 v = make_double2(0.0, 0.0);
      if (t < cnt) {
        if (!first) {
          v = Y[(int64_t)i * N + t0 + t];
        } else if (c128) {
          v = reinterpret_cast<const double2 *>(X)[(int64_t)i * ldx + t0 + t];
        } else {
          const float2 a = reinterpret_cast<const float2 *>(X)[(int64_t)i * ldx + t0 + t];
          v = make_double2((double)a.x, (double)a.y);
        }
      }
      S0[e] = v;
    }
    __syncthreads();
    for (int e = tid; e < M * kSvdT; e += kSvdThreads) {
      const int i = e / kSvdT, t = e % kSvdT;
      double2 y = S0[e];
      if (!first) {
        // (V^H Y)_i = sum_j conj(V_ji) y_j
        double re = 0.0, im = 0.0;
        for (int jj = 0; jj < M; ++jj) {
          const double2 v = Vs[jj * M + i], x = S0[jj * kSvdT + t];
          re = fma(v.x, x.x, fma(v.y, x.y, re));
          im = fma(v.x, x.y, fma(-v.y, x.x, im));
        }
        y = make_double2(re, im);
      }
      S1[e] = y;
      if (t < cnt) Y[(int64_t)i * N + t0 + t] = y;   // the chunks of a CTA are the same in every pass
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kSvdMaxE; ++k) {
      if (tid + k * kSvdThreads < E) {
        const double2 *yi = S1 + ei[k] * kSvdT, *yj = S1 + ej[k] * kSvdT;
        double re = acc[k].x, im = acc[k].y;
        for (int t = 0; t < kSvdT; ++t) {
          const double2 a = yi[t], b = yj[t];   // a conj(b)
          re = fma(a.x, b.x, fma(a.y, b.y, re));
          im = fma(a.y, b.x, fma(-a.x, b.y, im));
        }
        acc[k] = make_double2(re, im);
      }
    }
  }
  double2 *part = reinterpret_cast<double2 *>(ws + lay.off_part) + (int64_t)blockIdx.x * E;
#pragma unroll
  for (int k = 0; k < kSvdMaxE; ++k) {
    const int e = tid + k * kSvdThreads;
    if (e < E) part[e] = acc[k];
  }
}

// Sign and zero tests on the bits: FP64 negations, selections and comparisons take the FP64 pipe too.
__device__ __forceinline__ double flip_if(bool f, double x) {
  return __hiloint2double(__double2hiint(x) ^ (f ? (int)0x80000000 : 0), __double2loint(x));
}
__device__ __forceinline__ bool is_zero(double x) { return ((__double2hiint(x) & 0x7fffffff) | __double2loint(x)) == 0; }
// x <= y for y >= 0 (false for a NaN x): negative numbers down to -inf, or by the order of the bits
__device__ __forceinline__ bool at_most(double x, double y) {
  const long long bx = __double_as_longlong(x);
  return bx < 0 ? bx <= (long long)0xfff0000000000000ull : bx <= __double_as_longlong(y);
}

// Level s of a row-cyclic sweep: the disjoint pairs (p, s - p), p = first .. first + count - 1.
struct SvdLevel {
  int first, count;
};
__device__ __forceinline__ SvdLevel svd_level(int s, int M) {
  SvdLevel l;
  l.first = max(0, s - M + 1);
  l.count = (s - 1) / 2 - l.first + 1;
  return l;
}

// One sweep on G in shared memory (row stride ld, odd, so that columns spread over the banks); records
// its rotations. Returns bit 0: a pair was rotated (or, when
// `last`, would have been), bit 1: one had |gamma| > 1e-4 sqrt(alpha beta).
__device__ int svd_sweep(double2 *G, SvdRot *rot, int M, int ld, double tol2, double floor_d, bool last, SvdRot *rec) {
  __shared__ int flag[kMaxM / 2];
  const int tid = threadIdx.x, lane = tid & 31;
  int seen = 0;
  double shift = 0.0;
  for (int s = 1; s <= 2 * M - 3; ++s) {
    const SvdLevel lv = svd_level(s, M);
    // warp 0 forms every pair's rotation while warp 1 decides which pairs rotate: on one warp the two
    // would follow each other on one FP64 pipe
    if (tid < 64 && lane < lv.count) {
      const int p = lv.first + lane, q = s - p;
      const double alpha = G[p * ld + p].x, beta = G[q * ld + q].x;
      const double2 gamma = G[p * ld + q];
      const double n2 = fma(gamma.x, gamma.x, gamma.y * gamma.y);
      if (tid < 32) {
        // cos and sin of the rotation angle from cos(2 angle) = |d| / h, sin(2 angle) = 2 |gamma| / h
        const double d = beta - alpha;
        const double rh = rsqrt(fma(4.0, n2, d * d));          // 1 / h
        const double w = fma(fabs(d) * rh, 0.5, 0.5);           // cos^2
        const double rc = rsqrt(w);                             // 1 / cos
        const double k = copysign(rh * rc, d);                  // s / |gamma|
        rot[lane] = SvdRot{w * rc, k * gamma.x, k * gamma.y};
        shift = k * n2 * rc;                                    // t |gamma|
      } else {
        const double ab = alpha * beta;
        const bool act = !at_most(alpha, floor_d) && !at_most(beta, floor_d) && !is_zero(n2) && !(n2 <= tol2 * ab);
        flag[lane] = act;
        // |gamma| above about 1e-4 sqrt(alpha beta), from the exponents
        if (act) seen |= (__double2hiint(n2) >> 20) - (__double2hiint(ab) >> 20) > -27 ? 3 : 1;
      }
    }
    if (last) continue;   // the cap is reached: report, do not rotate
    __syncthreads();
    if (tid < 32 && lane < lv.count) {   // the pairs' own 2 x 2 blocks, in closed form
      const bool act = flag[lane] != 0;
      if (act) {
        const int p = lv.first + lane, q = s - p;
        G[p * ld + p].x -= shift;
        G[q * ld + q].x += shift;
        G[p * ld + q] = G[q * ld + p] = make_double2(0.0, 0.0);
      }
      rec[lane] = act ? rot[lane] : SvdRot{0.0, 0.0, 0.0};
    }
    rec += lv.count;
    // pairs a < b: the 2 x 2 block of rows of a and columns of b, four lanes, one element each: the row
    // mix of the lane's element, exchanged with the lane of the other column, then the column mix
    const int np = lv.count, nq = (np + 1) & ~1;
    const int nblk = nq / 2 * (nq - 1);
    const float inv_nq = __fdividef(1.f, (float)(nq - 1));   // quotients of small integers: exact after the +0.5
    for (int e0 = tid & ~31; e0 < nblk * 4; e0 += kSvdThreads) {
      const int e = e0 + lane, blk = e >> 2;
      int a = np, b = np;
      if (blk < nblk) {
        const int i = (int)(((float)blk + 0.5f) * inv_nq), j = blk - i * (nq - 1);
        a = j >= i ? i : nq - 1 - i;
        b = j >= i ? j + 1 : nq - 1 - j;
      }
      const bool in = a < np && b < np;
      const bool acta = in && flag[a], actb = in && flag[b], act = acta || actb;
      const int pa = lv.first + a, qa = s - pa, pb = lv.first + b, qb = s - pb;
      const bool lo_row = (lane & 2) == 0, lo_col = (lane & 1) == 0;
      const int row = lo_row ? pa : qa, col = lo_col ? pb : qb;
      double2 x = make_double2(0.0, 0.0);
      if (act) {
        const double2 xp = G[pa * ld + col], xq = G[qa * ld + col];
        x = lo_row ? xp : xq;
        if (acta) {
          const SvdRot ra = rot[a];
          // row p: c x_p - sigma x_q; row q: conj(sigma) x_p + c x_q
          const double2 y = lo_row ? xq : xp;
          const double sr = flip_if(lo_row, ra.sr);
          x = make_double2(fma(ra.c, x.x, fma(sr, y.x, ra.si * y.y)), fma(ra.c, x.y, fma(sr, y.y, -ra.si * y.x)));
        }
      }
      double2 y;
      y.x = __shfl_xor_sync(0xffffffffu, x.x, 1);
      y.y = __shfl_xor_sync(0xffffffffu, x.y, 1);
      if (act) {
        if (actb) {
          const SvdRot rb = rot[b];
          // column p: c x_p - conj(sigma) x_q; column q: sigma x_p + c x_q
          const double sr = flip_if(lo_col, rb.sr);
          x = make_double2(fma(rb.c, x.x, fma(sr, y.x, -rb.si * y.y)), fma(rb.c, x.y, fma(sr, y.y, rb.si * y.x)));
        }
        G[row * ld + col] = x;
        G[col * ld + row] = make_double2(x.x, flip_if(true, x.y));
      }
    }
    // pairs and single indices: two lanes an element pair, the row mix alone
    // (taken from the last warp down: the blocks above may leave those idle)
    const int ns = M - 2 * np, hole = (s & 1) ? -1 : s / 2;
    const float inv_ns = __fdividef(1.f, (float)ns);
    for (int e0 = (kSvdThreads - 32) - (tid & ~31); e0 < np * ns; e0 += kSvdThreads) {
      const int e = e0 + lane;
      if (e < np * ns) {
        const int a = (int)(((float)e + 0.5f) * inv_ns), j = e - a * ns;
        // single j: below the paired range, above it, or the middle index
        int col = j < lv.first ? j : s - lv.first + 1 + (j - lv.first);
        if (j == ns - 1 && hole >= 0) col = hole;
        if (flag[a]) {
          const SvdRot ra = rot[a];
          const int pa = lv.first + a, qa = s - pa;
          const double2 xp = G[pa * ld + col], xq = G[qa * ld + col];
          const double2 np_ = make_double2(fma(ra.c, xp.x, fma(-ra.sr, xq.x, ra.si * xq.y)),
                                           fma(ra.c, xp.y, fma(-ra.sr, xq.y, -ra.si * xq.x)));
          const double2 nq_ = make_double2(fma(ra.c, xq.x, fma(ra.sr, xp.x, ra.si * xp.y)),
                                           fma(ra.c, xq.y, fma(ra.sr, xp.y, -ra.si * xp.x)));
          G[pa * ld + col] = np_;
          G[qa * ld + col] = nq_;
          G[col * ld + pa] = make_double2(np_.x, flip_if(true, np_.y));
          G[col * ld + qa] = make_double2(nq_.x, flip_if(true, nq_.y));
        }
      }
    }
    __syncthreads();
  }
  return __syncthreads_or(seen & 1) | (__syncthreads_or(seen & 2) ? 2 : 0);
}

// Applies nsw recorded sweeps to row r of A (columns mixed pair by pair); A starts as the identity
// when `fresh`. One warp per row; the next level's rotations are loaded ahead.
__device__ void svd_rows(const SvdRot *rec, int nsw, int M, int r, bool fresh, double2 *A, double2 *row) {
  const int lane = threadIdx.x & 31;
  for (int k = lane; k < M; k += 32) row[k] = fresh ? make_double2(k == r ? 1.0 : 0.0, 0.0) : __ldcg(&A[r * M + k]);
  __syncwarp();
  auto load = [&](int s) {
    SvdRot v{0.0, 0.0, 0.0};
    if (lane < svd_level(s, M).count) {
      const double *p = reinterpret_cast<const double *>(rec + lane);
      v = SvdRot{__ldcg(p), __ldcg(p + 1), __ldcg(p + 2)};
    }
    return v;
  };
  const int levels = 2 * M - 3;
  SvdRot next = load(1);
  for (int i = 0; i < nsw * levels; ++i) {
    const int s = i % levels + 1;
    const SvdLevel lv = svd_level(s, M);
    const SvdRot ro = next;
    rec += lv.count;
    if (i + 1 < nsw * levels) next = load((i + 1) % levels + 1);
    if (!is_zero(ro.c)) {
      const int p = lv.first + lane, q = s - p;
      const double2 xp = row[p], xq = row[q];
      row[p] = make_double2(fma(ro.c, xp.x, fma(-ro.sr, xq.x, -ro.si * xq.y)),
                            fma(ro.c, xp.y, fma(-ro.sr, xq.y, ro.si * xq.x)));
      row[q] = make_double2(fma(ro.c, xq.x, fma(ro.sr, xp.x, -ro.si * xp.y)),
                            fma(ro.c, xq.y, fma(ro.sr, xp.y, ro.si * xp.x)));
    }
    __syncwarp();
  }
  for (int k = lane; k < M; k += 32) A[r * M + k] = row[k];
  __syncwarp();
}

__global__ void __launch_bounds__(kSvdThreads, 1) svd_kernel(const void *X, int c128, int ldx, int M, int N, double tol,
                                                              int max_sweeps, uint8_t *ws, SvdLayout lay, double *evals,
                                                              double2 *Uout, int *info) {
  extern __shared__ __align__(16) uint8_t svd_smem[];
  __shared__ SvdRot rot[kMaxM / 2];
  __shared__ double ev[kMaxM];
  __shared__ int order[kMaxM];
  __shared__ double s_min, s_max;
  SvdState *st = reinterpret_cast<SvdState *>(ws + lay.off_state);
  double2 *Gg = reinterpret_cast<double2 *>(ws + lay.off_G);
  double2 *Vg = reinterpret_cast<double2 *>(ws + lay.off_V);
  double2 *Ug = reinterpret_cast<double2 *>(ws + lay.off_U);
  const double2 *part = reinterpret_cast<const double2 *>(ws + lay.off_part);
  SvdRot *rec = reinterpret_cast<SvdRot *>(ws + lay.off_part);   // after the partial sums are consumed
  const int tid = threadIdx.x, E = M * (M + 1) / 2, npairs = M * (M - 1) / 2;
  const int nblk = gridDim.x;
  unsigned phase = 0;
  int sweeps = 0;        // CTA 0: sweeps taken
  bool first = true, ok = true;
  while (true) {
    svd_pass(X, c128 != 0, first, ldx, M, N, ws, lay, svd_smem);
    if (!(ok = grid_barrier(st, phase))) break;
    // a warp per entry; lanes over the CTAs' partial sums, then a shuffle tree: a fixed order
    for (int e = blockIdx.x + (tid >> 5) * nblk; e < E; e += nblk * (kSvdThreads / 32)) {
      double re = 0.0, im = 0.0;
      for (int b = tid & 31; b < nblk; b += 32) {
        const double2 v = __ldcg(&part[(int64_t)b * E + e]);
        re += v.x;
        im += v.y;
      }
      for (int off = 16; off > 0; off >>= 1) {
        re += __shfl_xor_sync(0xffffffffu, re, off);
        im += __shfl_xor_sync(0xffffffffu, im, off);
      }
      if ((tid & 31) == 0) Gg[e] = make_double2(re, im);
    }
    if (!(ok = grid_barrier(st, phase))) break;
    if (blockIdx.x == 0) {
      double2 *G = reinterpret_cast<double2 *>(svd_smem);   // M x M row-major, stride ld
      const int ld = M | 1;
      auto extremes = [&]() {   // smallest and largest diagonal entry
        if (tid < 32) {
          double lo = CUDART_INF, hi = 0.0;
          for (int i = tid; i < M; i += 32) {
            lo = fmin(lo, G[i * ld + i].x);
            hi = fmax(hi, G[i * ld + i].x);
          }
          for (int off = 16; off > 0; off >>= 1) {
            lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, off));
            hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, off));
          }
          if (tid == 0) {
            s_min = lo;
            s_max = hi;
          }
        }
        __syncthreads();
      };
      for (int e = tid; e < E; e += kSvdThreads) {
        int i, j;
        tri_index(e, M, i, j);
        const double2 v = __ldcg(&Gg[e]);
        G[i * ld + j] = make_double2(v.x, i == j ? 0.0 : v.y);   // y_i y_i^H is real
        if (i != j) G[j * ld + i] = make_double2(v.x, -v.y);
      }
      __syncthreads();
      extremes();
      // a power of two brings the largest squared norm to [1, 2): the squares below stay in range
      int ex = 0;
      const bool scaled = s_max > 0.0 && s_max < CUDART_INF;
      if (scaled) ex = ilogb(s_max);
      __syncthreads();
      for (int e = tid; scaled && e < M * ld; e += kSvdThreads) {
        G[e].x = scalbn(G[e].x, -ex);
        G[e].y = scalbn(G[e].y, -ex);
      }
      // rows whose squared norm is below 1e-30 of the largest (fresh Gram diagonal) are numerically
      // zero (a rank-deficient X leaves them at the rounding level, where |gamma| stays comparable to
      // sqrt(alpha beta)): pairs with one are not rotated
      const double floor_d = 1e-30 * (scaled ? scalbn(s_max, -ex) : s_max);
      __syncthreads();
      bool fin = false, rotated = false;
      int nrec = 0;
      while (true) {
        const bool last = sweeps + 1 >= max_sweeps;
        const int seen = svd_sweep(G, rot, M, ld, tol * tol, floor_d, last, rec + (int64_t)nrec * npairs);
        ++sweeps;
        rotated = (seen & 1) != 0;
        if ((!rotated && nrec == 0) || last) {   // converged on fresh rows, or the cap
          fin = true;
          break;
        }
        if (rotated) ++nrec;
        else --sweeps;                           // a sweep to be confirmed on fresh rows does not count
        extremes();
        // the last sweep allowed decides on fresh rows
        if (!(seen & 2) || nrec >= kSvdInner || sweeps + 1 >= max_sweeps || !(s_min > 1e-4 * s_max)) break;
        __syncthreads();
      }
      if (fin) {
        // eigenvalues of R = S^2 / N descending, equal values in index order
        if (tid < M) ev[tid] = (scaled ? scalbn(G[tid * ld + tid].x, ex) : G[tid * ld + tid].x) / (double)N;
        __syncthreads();
        if (tid == 0) {
          for (int i = 0; i < M; ++i) order[i] = i;
          for (int i = 1; i < M; ++i) {
            const int cur = order[i];
            int j = i - 1;
            while (j >= 0 && ev[order[j]] < ev[cur]) {
              order[j + 1] = order[j];
              --j;
            }
            order[j + 1] = cur;
          }
        }
        __syncthreads();
        if (tid < M) evals[tid] = ev[order[tid]];
        for (int e = tid; e < M * M; e += kSvdThreads) {
          const int col = e / M, r = e % M;   // column-major: column col = singular vector col
          // no rotation was recorded before: U is the identity
          Uout[e] = first ? make_double2(r == order[col] ? 1.0 : 0.0, 0.0) : __ldcg(&Ug[r * M + order[col]]);
        }
        if (tid == 0) *info = rotated ? -(int)DOA_ENOCONV : sweeps;
      }
      if (tid == 0) st->cmd = fin ? 0 : nrec;
    }
    if (!(ok = grid_barrier(st, phase))) break;
    const int nsw = __ldcg(&st->cmd);
    if (nsw == 0) break;
    {
      // a warp per row of V, then of U; row r on CTA r mod nblk
      double2 *row = reinterpret_cast<double2 *>(svd_smem) + (tid >> 5) * M;
      for (int r = blockIdx.x + (tid >> 5) * nblk; r < 2 * M; r += nblk * (kSvdThreads / 32)) {
        const bool isv = r < M;
        svd_rows(rec, nsw, M, isv ? r : r - M, isv || first, isv ? Vg : Ug, row);
      }
    }
    first = false;
    if (!(ok = grid_barrier(st, phase))) break;
  }
  if (!ok && blockIdx.x == 0 && tid == 0) *info = -(int)DOA_ETIMEOUT;
}

// SMs that kernels of a stream may use: the device's, or those of the stream's green context. The CTAs of the
// grid wait for one another, so a launch of more of them than can be resident is refused.
int stream_sm_count(cudaStream_t s) {
  auto entry = [](const char *name, unsigned version) {
    cudaDriverEntryPointQueryResult q;
    void *fn = nullptr;
    const cudaError_t e = cudaGetDriverEntryPointByVersion(name, &fn, version, cudaEnableDefault, &q);
    return e == cudaSuccess && q == cudaDriverEntryPointSuccess ? fn : nullptr;
  };
  static const auto stream_ctx = reinterpret_cast<PFN_cuStreamGetCtx_v12050>(entry("cuStreamGetCtx", 12050));
  static const auto ctx_res = reinterpret_cast<PFN_cuCtxGetDevResource_v12040>(entry("cuCtxGetDevResource", 12040));
  static const auto green_res =
      reinterpret_cast<PFN_cuGreenCtxGetDevResource_v12040>(entry("cuGreenCtxGetDevResource", 12040));
  const int all = device_sm_count();
  CUcontext ctx = nullptr;
  CUgreenCtx green = nullptr;
  CUdevResource r{};
  if (!stream_ctx || !ctx_res || !green_res || stream_ctx(s, &ctx, &green) != CUDA_SUCCESS) return all;
  const CUresult got = green ? green_res(green, &r, CU_DEV_RESOURCE_TYPE_SM) : ctx_res(ctx, &r, CU_DEV_RESOURCE_TYPE_SM);
  return got == CUDA_SUCCESS && r.sm.smCount > 0 ? std::min(all, (int)r.sm.smCount) : all;
}

}  // namespace
}  // namespace doa

using namespace doa;

extern "C" {

size_t doa_svd_data_ws_bytes(int M, int N) {
  if (M < 2 || M > kMaxM || N < 1) return 0;
  return (size_t)svd_layout(M, N).bytes;
}

doa_status doa_svd_data(const void *X, int x_c128, int M, int N, int ldx, double tol, int max_sweeps, double *evals,
                        double *U, int *info, void *ws, size_t ws_bytes, void *stream) {
  if (!X || !evals || !U || !info || !ws || M < 2 || M > kMaxM || N < 1 || ldx < N || (x_c128 != 0 && x_c128 != 1))
    return DOA_EINVAL;
  if (!(tol > 0.0) || !std::isfinite(tol) || max_sweeps < 1 || max_sweeps > 1000) return DOA_EINVAL;
  auto aligned = [](const void *p, size_t a) { return reinterpret_cast<uintptr_t>(p) % a == 0; };
  if (!aligned(X, x_c128 ? 16 : 8) || !aligned(evals, 8) || !aligned(U, 16) || !aligned(info, 4) || !aligned(ws, 16))
    return DOA_EINVAL;
  const SvdLayout lay = svd_layout(M, N);
  if (ws_bytes < (size_t)lay.bytes) return DOA_ENOMEM;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int nchunks = (N + kSvdT - 1) / kSvdT;
  const int nblk = std::min(std::min(nchunks, kSvdMaxBlocks), stream_sm_count(s));
  const int smem = (int)((size_t)(2 * M * kSvdT + M * M) * sizeof(double2));
  if (ensure_smem_attr((const void *)svd_kernel, smem) != cudaSuccess) return DOA_ECUDA;
  uint8_t *w = static_cast<uint8_t *>(ws);
  if (cudaMemsetAsync(w + lay.off_state, 0, sizeof(SvdState), s) != cudaSuccess) return DOA_ECUDA;
  // cooperative: the CTAs (one per SM at most) wait for one another
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)nblk);
  cfg.blockDim = dim3(kSvdThreads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = s;
  cudaLaunchAttribute coop{};
  coop.id = cudaLaunchAttributeCooperative;
  coop.val.cooperative = 1;
  cfg.attrs = &coop;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, svd_kernel, X, x_c128, ldx, M, N, tol, max_sweeps, w, lay, evals,
                         reinterpret_cast<double2 *>(U), info) != cudaSuccess)
    return DOA_ECUDA;
  return DOA_OK;
}

}  // extern "C"
