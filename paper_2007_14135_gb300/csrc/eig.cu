// Steps 2-4 (Table 2 Step-2, Table 3): Hermitian eigendecomposition of R by FP64 cyclic Jacobi,
// followed by the noise-subspace factor B of each algorithm's weighting matrix C = B B^H (one
// call), or, in the batch, one scan factor per problem from which every requested algorithm's
// spectrum is read (E_n with EV weights 1/lambda, v_min, valph).
//
// Jacobi (Golub & Van Loan, Sec. 8.5, with a phase factor for complex Hermitian matrices):
// for a pair (p, q) with a_pq = |a_pq| e^{j phi}, tau = (a_qq - a_pp) / (2 |a_pq|),
// t = sgn(tau) / (|tau| + sqrt(1 + tau^2)), c = 1/sqrt(1 + t^2), s = t c, sigma = s e^{j phi};
// J = [[c, sigma], [-conj(sigma), c]] on coordinates (p, q) zeroes (J^H A J)_pq.
// The parameters use reciprocal square roots (no hypot or sqrt; in FP64 no tau or t either, see
// rotation_of), so c^2 + |sigma|^2 = 1 holds to rounding.
//
// Parallel ordering: n/2 disjoint rotations per round (round-robin "circle" ordering over
// n = M rounded up to even; a pair that touches the padding index is not rotated). A pair is
// rotated when |a_pq|^2 > tol^2 |a_pp a_qq|; a matrix has converged after a sweep that rotates
// nothing. A round updates A block by block: the 2 x 2 block of the rows of pair a and the columns of
// pair b >= a takes four lanes, one element each -- the row mix A <- J^H A of the lane's element,
// exchanged with the lane of the other column, then the column mix A <- A J -- and is written to its
// mirror image as well, so only half of A is computed; V <- V J takes a lane per pair and row. Both halves
// are computed, each element by the row mix and then the column mix, for matrices of M <= 8 (where half the
// blocks take as many warp steps as all of them), for geometry problems (where a minimum of the planar
// array's spectrum meets its mirror image at the array plane, the refined angle moves by the square root of a
// rounding error) and in double-float: it rotates down to 1e-12 only, so noise eigenvectors whose eigenvalues
// nearly meet keep 1e-7 to 1e-6 of whatever is added in another order.
//
// Two shapes, with the same arithmetic and results. A warp per matrix (or G packed matrices, every
// lane owning one pair's rotation) keeps the most matrices resident and suits large batches of M <= 16.
// A CTA per matrix (3, 4 or 5, 16 or 17 warps at M <= 8, 16, 32) suits single calls, small batches and M <= 32,
// which otherwise wait for one warp's chain of instructions: one FP64 matrix of M = 8 in 78 instead of
// 141 us, 256 double-float matrices of M = 32 in 0.81 instead of 2.84 ms. Half of A: one FP64 matrix of M = 64
// in 6.8 instead of 9.6 ms. Double-float takes two lanes a block, a column each, which share the indices and
// rotations of two elements: 4096 matrices of M = 16 (warp form) in 1.09 ms, 1.21 with four.
// M <= 64 gets a 512-thread CTA in FP64, or in double-float a cluster of four CTAs that split its
// rows (jacobi_cluster_df).
#include <cooperative_groups.h>
#include <type_traits>
#include <math_constants.h>

#include "doa_internal.cuh"

namespace doa {
namespace {

namespace cg = cooperative_groups;

struct Rot {
  double c, sr, si;  // cosine and sigma = s e^{j phi}
};

template <int NP>
struct EigSmem {
  // A and V row-major without padding; element (i, k) sits in column slot k ^ (i & 7), so that
  // both row walks (fixed i) and column walks (fixed k, consecutive rows) touch distinct banks
  double2 A[NP][NP];
  double2 V[NP][NP];
  Rot rot[NP / 2];      // the sweeps' rotations; after the sweeps the same bytes hold lam, order
  int2 pq[NP / 2];
  __device__ __forceinline__ double2 &a(int i, int k) { return A[i][k ^ (i & 7)]; }
  __device__ __forceinline__ double2 &v(int i, int k) { return V[i][k ^ (i & 7)]; }
  __device__ __forceinline__ double *lam() { return reinterpret_cast<double *>(rot); }
  __device__ __forceinline__ int *order() { return reinterpret_cast<int *>(reinterpret_cast<double *>(rot) + NP); }
  static_assert(sizeof(Rot) * (NP / 2) >= NP * (sizeof(double) + sizeof(int)), "lam and order fit in rot");
};

// Threads per matrix of the CTA form. A round's warp steps (blocks of A, then rows of V) are 2 + 1 at M = 8; in
// double-float 4 + 4 at M = 16 and 16 + 16 at M = 32, two turns of four and 16 warps; in FP64 with half of A
// 5 + 4 and 17 + 16, which suits five and 17 (double-float, five / four warps: 1024 matrices of M = 16 0.36 /
// 0.32 ms; FP64 one 0.23 / 0.28, 256 0.37 / 0.43, 1024 0.90 / 0.89). A bucket with both takes FP64's.
template <int NP, bool kDF = true>
__host__ __device__ constexpr int cta_threads() {
  return NP <= 8 ? 96 : NP <= 16 ? (kDF ? 128 : 160) : NP <= 32 ? (kDF ? 512 : 544) : 512;
}
// Largest batch that takes the CTA form (the eig stage, warp form against CTA form): at M <= 8, 63 / 47
// us for 1 matrix, 82 / 74 for 1024, 112 / 131 for 2048; at M <= 16, 0.32 / 0.14 ms for 1, 0.55 / 0.32
// for 1024, 0.80 / 0.59 for 2048; at M <= 32 always (1.9 / 0.41 ms for 1, 5.3 / 2.6 for 1024).
template <int NP>
__host__ constexpr int eig_cta_limit() { return NP <= 8 ? 1024 : 2048; }
template <int NP>
__host__ __device__ constexpr int mats_per_warp() { return 64 / NP; }
// Warps per CTA of the warp form, at most (the launch picks the count for the resident total).
template <int NP>
__host__ __device__ constexpr int eig_warps() { return NP <= 8 ? 4 : 9; }
// CTAs per SM its register budget is set for: three nine-warp CTAs at M <= 16, 64 registers a thread
// at M <= 8.
template <int NP>
__host__ __device__ constexpr int eig_min_ctas() { return NP <= 8 ? 8 : 3; }

// FP64 matrices whose largest element is outside 2^-400 .. 2^400 are brought to the nearer end by a power of two
// (exactly) for the Jacobi, whose rotations square differences and elements.
constexpr int kEigSafeExp = 400;

template <int T>
struct Grp {
  __device__ static int id() { return (int)(threadIdx.x % T); }
  __device__ static void sync() {
    if (T == 32) __syncwarp(); else __syncthreads();
  }
  __device__ static bool all(bool p) { return T == 32 ? __all_sync(0xffffffffu, p) : __syncthreads_and(p) != 0; }
  __device__ static bool any(bool p) { return T == 32 ? __any_sync(0xffffffffu, p) : __syncthreads_or(p) != 0; }
};

__device__ __forceinline__ int rr_player(int pos, int r, int n) {
  const int v = pos - 1 + r;   // < 2 (n - 1)
  return pos == 0 ? 0 : (v >= n - 1 ? v - (n - 1) : v) + 1;
}

// Rotation of a pair from its entries; returns false if the pair is below threshold. An FP64 warp
// instruction holds its sub-partition for 64 cycles here, so the chain is kept short: cos^2 = 1/2 +
// |d| / (2h) and sigma = a_pq / (h cos) with d = a_qq - a_pp, h = sqrt(d^2 + 4 |a_pq|^2) -- the same
// rotation as through tau and t, with two reciprocal square roots and no division.
__device__ __forceinline__ bool rotation_of(const double app, const double aqq, const double2 apq, Rot &ro) {
  const double n2 = fma(apq.x, apq.x, apq.y * apq.y);
  if (!(n2 > kJacobiTol * kJacobiTol * fabs(app * aqq))) return false;
  const double d = aqq - app;
  const double rh = rsqrt(fma(4.0, n2, d * d));        // 1 / h
  const double w = fma(fabs(d) * rh, 0.5, 0.5);         // cos^2
  const double rc = rsqrt(w);                           // 1 / cos
  const double k = copysign(rh * rc, d);                // sin / |a_pq|, of the sign of tau
  ro = Rot{w * rc, k * apq.x, k * apq.y};
  return true;
}

// ------------------------------------------------------------------------------------------
// Double-float Jacobi for the batch. GB300 issues FP64 at ~1/64 of its FP32 rate, so the batch
// runs the same cyclic Jacobi with A and V held as unevaluated sums hi + lo of two FP32 numbers
// (about 48 significant bits) and every element update done on the FP32 pipe: each new real part
// is a three-term dot product of double-float numbers, formed with exact FMA products and
// TwoSum (a compensated dot product, relative error a few 2^-48 of the sum of |terms|).
// The rotation angle only needs to be good to FP32: tau, t and (c, sigma) are computed in FP32
// from the hi parts (the diagonal difference from hi and lo), then (c, sigma) is scaled by
// 1/sqrt(c^2 + |sigma|^2) to double-float accuracy, so every applied rotation is unitary to
// ~1e-15; a_pq is left at its computed residual (about 1e-7 of its old value) instead of being
// set to zero, and the next sweep removes it. Converged when a sweep rotates no pair with
// |a_pq| > kJacobiTolDF sqrt(|a_pp a_qq|). A and V are converted to FP64 in place at the end.
// ------------------------------------------------------------------------------------------
constexpr float kJacobiTolDF = 1e-12f;

struct F2 {
  float h, l;
};

__device__ __forceinline__ void two_sum_f(float a, float b, float &s, float &e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// u1 v1 + u2 v2 + u3 v3 in double-float.
__device__ __forceinline__ F2 dot3(F2 u1, F2 v1, F2 u2, F2 v2, F2 u3, F2 v3) {
  const float p1 = __fmul_rn(u1.h, v1.h), p2 = __fmul_rn(u2.h, v2.h), p3 = __fmul_rn(u3.h, v3.h);
  float low = __fmaf_rn(u1.h, v1.h, -p1);
  low = __fadd_rn(low, __fmaf_rn(u2.h, v2.h, -p2));
  low = __fadd_rn(low, __fmaf_rn(u3.h, v3.h, -p3));
  low = __fadd_rn(low, __fmaf_rn(u1.h, v1.l, __fmul_rn(u1.l, v1.h)));
  low = __fadd_rn(low, __fmaf_rn(u2.h, v2.l, __fmul_rn(u2.l, v2.h)));
  low = __fadd_rn(low, __fmaf_rn(u3.h, v3.l, __fmul_rn(u3.l, v3.h)));
  float s, e1, e2;
  two_sum_f(p1, p2, s, e1);
  two_sum_f(s, p3, s, e2);
  low = __fadd_rn(low, __fadd_rn(e1, e2));
  F2 r;
  two_sum_f(s, low, r.h, r.l);
  return r;
}

__device__ __forceinline__ F2 neg(F2 a) { return F2{-a.h, -a.l}; }
__device__ __forceinline__ F2 re_of(float4 v) { return F2{v.x, v.y}; }
__device__ __forceinline__ F2 im_of(float4 v) { return F2{v.z, v.w}; }
__device__ __forceinline__ float4 cplx(F2 re, F2 im) { return make_float4(re.h, re.l, im.h, im.l); }
__device__ __forceinline__ float4 df_of(double2 v) {
  const float rh = (float)v.x, ih = (float)v.y;
  return make_float4(rh, (float)(v.x - (double)rh), ih, (float)(v.y - (double)ih));
}

struct RotDF {
  F2 c, sr, si;   // cosine and sigma = s e^{j phi}, each hi + lo
};

template <int NP>
struct EigSmemDF {   // the same bytes as EigSmem<NP>, viewed as double-float
  float4 A[NP][NP];
  float4 V[NP][NP];
  RotDF rot[NP / 2];
  __device__ __forceinline__ float4 &a(int i, int k) { return A[i][k ^ (i & 7)]; }
  __device__ __forceinline__ float4 &v(int i, int k) { return V[i][k ^ (i & 7)]; }
};
static_assert(sizeof(RotDF) == sizeof(Rot), "rotation records share storage");

// Rotation of a pair from its entries a_pp, a_qq, a_pq; returns false below threshold.
__device__ __forceinline__ bool rotation_df_of(const float4 app, const float4 aqq, const float4 apq, RotDF &ro) {
  const float n2 = apq.x * apq.x + apq.z * apq.z;
  if (!(n2 > 0.f) || !(n2 > kJacobiTolDF * kJacobiTolDF * fabsf(app.x * aqq.x))) return false;
  const float r = rsqrtf(n2);                                   // 1 / |a_pq|
  const float diff = __fadd_rn(__fsub_rn(aqq.x, app.x), __fsub_rn(aqq.y, app.y));
  const float tau = diff * (0.5f * r);
  float t;
  if (fabsf(tau) > 1e4f) {
    t = 0.5f / tau;                                             // 1/(2 tau), relative error < tau^-2 / 4
  } else {
    t = copysignf(1.f / (fabsf(tau) + sqrtf(fmaf(tau, tau, 1.f))), tau);
  }
  const float c0 = rsqrtf(fmaf(t, t, 1.f));
  const float sn = t * c0 * r;
  const float sr0 = sn * apq.x, si0 = sn * apq.z;
  // n = c0^2 + sr0^2 + si0^2 exactly to double-float; scale all three by 1/sqrt(n) = 1 + eps
  const float q1 = __fmul_rn(c0, c0), q2 = __fmul_rn(sr0, sr0), q3 = __fmul_rn(si0, si0);
  float low = __fadd_rn(__fadd_rn(__fmaf_rn(c0, c0, -q1), __fmaf_rn(sr0, sr0, -q2)), __fmaf_rn(si0, si0, -q3));
  float sum, e1, e2;
  two_sum_f(q1, q2, sum, e1);
  two_sum_f(sum, q3, sum, e2);
  const float delta = __fadd_rn(__fsub_rn(sum, 1.f), __fadd_rn(low, __fadd_rn(e1, e2)));
  const float eps = delta * fmaf(0.375f, delta, -0.5f);        // (1 + delta)^(-1/2) - 1 to O(delta^3)
  ro = RotDF{F2{c0, c0 * eps}, F2{sr0, sr0 * eps}, F2{si0, si0 * eps}};
  return true;
}

// The two arithmetics of the Jacobi: element type, rotation of a pair, and the mix of an element with
// its partner: c own + sr oth + (si oth_im, -si oth_re). With (sr, si) = (-+Re sigma, Im sigma) that is
// row p (-) or q (+) of J^H A, with -Im sigma column p (-) or q (+) of A J.
template <int NP>
struct ArithF64 {
  using El = double2;
  using Ro = Rot;
  static __device__ __forceinline__ El &a(EigSmem<NP> &s, int i, int k) { return s.a(i, k); }
  static __device__ __forceinline__ El &v(EigSmem<NP> &s, int i, int k) { return s.v(i, k); }
  static __device__ __forceinline__ Ro *rot(EigSmem<NP> &s) { return s.rot; }
  static __device__ __forceinline__ El from(double2 x) { return x; }
  static __device__ __forceinline__ bool rotation(El app, El aqq, El apq, Ro &ro) {
    return rotation_of(app.x, aqq.x, apq, ro);
  }
  // sign changes on the bits: an FP64 negation costs as much as a multiply-add
  static __device__ __forceinline__ double neg(double x) {
    return __hiloint2double(__double2hiint(x) ^ (int)0x80000000, __double2loint(x));
  }
  static __device__ __forceinline__ El mix(double c, double sr, double si, El own, El oth) {
    return make_double2(fma(c, own.x, fma(sr, oth.x, si * oth.y)), fma(c, own.y, fma(sr, oth.y, -si * oth.x)));
  }
  static __device__ __forceinline__ El conj(El x) { return make_double2(x.x, neg(x.y)); }
  static __device__ __forceinline__ El real(El x) { return make_double2(x.x, 0.0); }
  static constexpr bool kZeroes = true;   // the annihilated entry is set to zero
  static constexpr bool kBoth = false;    // half of A, unless asked for
};

template <int NP>
struct ArithDF {
  using El = float4;
  using Ro = RotDF;
  static __device__ __forceinline__ EigSmemDF<NP> &df(EigSmem<NP> &s) { return *reinterpret_cast<EigSmemDF<NP> *>(&s); }
  static __device__ __forceinline__ El &a(EigSmem<NP> &s, int i, int k) { return df(s).a(i, k); }
  static __device__ __forceinline__ El &v(EigSmem<NP> &s, int i, int k) { return df(s).v(i, k); }
  static __device__ __forceinline__ Ro *rot(EigSmem<NP> &s) { return df(s).rot; }
  static __device__ __forceinline__ El from(double2 x) { return df_of(x); }
  static __device__ __forceinline__ bool rotation(El app, El aqq, El apq, Ro &ro) {
    return rotation_df_of(app, aqq, apq, ro);
  }
  static __device__ __forceinline__ F2 neg(F2 x) { return F2{-x.h, -x.l}; }
  static __device__ __forceinline__ El mix(F2 c, F2 sr, F2 si, El own, El oth) {
    return cplx(dot3(c, re_of(own), sr, re_of(oth), si, im_of(oth)),
                dot3(c, im_of(own), sr, im_of(oth), neg(si), re_of(oth)));
  }
  static __device__ __forceinline__ El conj(El x) { return make_float4(x.x, x.y, -x.z, -x.w); }
  static __device__ __forceinline__ El real(El x) { return make_float4(x.x, x.y, 0.f, 0.f); }
  static constexpr bool kZeroes = false;  // it keeps its computed residual for the next sweep
  static constexpr bool kBoth = true;     // both halves of A
};

__device__ __forceinline__ double2 shfl_xor1(double2 x) {
  return make_double2(__shfl_xor_sync(0xffffffffu, x.x, 1), __shfl_xor_sync(0xffffffffu, x.y, 1));
}
__device__ __forceinline__ float4 shfl_xor1(float4 x) {
  return make_float4(__shfl_xor_sync(0xffffffffu, x.x, 1), __shfl_xor_sync(0xffffffffu, x.y, 1),
                     __shfl_xor_sync(0xffffffffu, x.z, 1), __shfl_xor_sync(0xffffffffu, x.w, 1));
}

// Brings the n x n matrix in s.A into that range; ex: the exponent of this thread's largest element. Returns
// the exponent of the power of two that it was divided by.
template <int T, int NP>
__device__ __noinline__ int scale_to_safe(EigSmem<NP> &s, int n, int ex) {
  __shared__ int warp_top[T / 32];
  int top = __reduce_max_sync(0xffffffffu, ex);
  if (T > 32) {
    if ((threadIdx.x & 31) == 0) warp_top[threadIdx.x >> 5] = top;
    __syncthreads();
    for (int w = 0; w < T / 32; ++w) top = max(top, warp_top[w]);
  }
  top -= top > 0 ? kEigSafeExp : -kEigSafeExp;
  for (int e = Grp<T>::id(); e < n * n; e += T) {   // the elements this thread wrote
    double2 &v = s.a(e / n, e % n);
    v = make_double2(scalbn(v.x, -top), scalbn(v.y, -top));
  }
  Grp<T>::sync();
  return top;
}

// Runs Jacobi on the G matrices of a group of T threads (matrix j has size Ms[j] <= NP, 0 = unused),
// all loaded from Rs[j] (upper triangle). T = 32: a warp; otherwise the whole CTA on one matrix.
// both[j]: compute both halves of A (always at M <= 8 and in double-float). res[j] receives sweeps (> 0) or -status; on return A (its diagonal) and V hold FP64.
template <class Ar, int NP, int G, int T>
__device__ void jacobi_group(EigSmem<NP> *mats, const int *Ms, const double2 *const *Rs, const bool *both, int *res) {
  static_assert(T == 32 || G == 1, "a CTA works on one matrix");
  constexpr int HP = NP / 2, W = T / 32;
  // a lane per column of a block, not per element (a CTA of M <= 8 has a warp for each element step)
  constexpr bool kColumns = Ar::kBoth && (T == 32 || NP > 8);
  using g = Grp<T>;
  using El = typename Ar::El;
  __shared__ unsigned smask[2];   // the round's rotations, by round parity (CTA form)
  const int tid = g::id(), lane = tid & 31, wp = tid >> 5;
  unsigned live = 0u;  // matrices still iterating
  int scaled[G];       // the exponent of the power of two it was divided by
  for (int j = 0; j < G; ++j) {
    const int M = Ms[j], n = (M + 1) & ~1;
    res[j] = scaled[j] = 0;
    if (M <= 0) continue;
    EigSmem<NP> &s = mats[j];
    const double2 *R = Rs[j];
    bool finite = true;
    int top = 0;       // high word of the largest |re|, |im|
    for (int e = tid; e < n * n; e += T) {
      const int i = e / n, k = e - i * n;
      double2 v = make_double2(0.0, 0.0);   // an odd M is padded with a zero row and column
      if (i < M && k < M) {
        v = R[min(i, k) * M + max(i, k)];
        if (i > k) v.y = -v.y;
        if (i == k) v.y = 0.0;
      }
      finite = finite && isfinite(v.x) && isfinite(v.y);
      top = max(top, max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff));
      Ar::a(s, i, k) = Ar::from(v);
      Ar::v(s, i, k) = Ar::from(make_double2(i == k ? 1.0 : 0.0, 0.0));
    }
    if (g::all(finite))
      live |= 1u << j;
    else
      res[j] = -DOA_ENONFINITE;
    if constexpr (Ar::kZeroes) {
      const int ex = (top >> 20) - 1023;
      if (((live >> j) & 1u) && (g::any(ex > kEigSafeExp) || !g::any(ex >= -kEigSafeExp)))
        scaled[j] = scale_to_safe<T>(s, n, ex);
    }
  }
  g::sync();
  int maxn = 0;
  for (int j = 0; j < G; ++j)
    if ((live >> j) & 1u) maxn = max(maxn, (Ms[j] + 1) & ~1);
  // lane of the first warp -> (matrix, pair) for the rotation parameters
  const int lj = wp == 0 ? lane / HP : G, li = lane % HP;
  unsigned t = 0u;     // rounds so far
  for (int sweep = 1; sweep <= kMaxSweeps && live; ++sweep) {
    unsigned rotated = 0u;
    for (int r = 0; r < maxn - 1; ++r, ++t) {
      unsigned mask = 0u;
      if (wp == 0) {
        bool act = false;
        if (lj < G && ((live >> lj) & 1u)) {
          const int M = Ms[lj], n = (M + 1) & ~1;
          if (r < n - 1 && li < n / 2) {
            const int a = rr_player(li, r, n), b = rr_player(n - 1 - li, r, n);
            const int p = min(a, b), q = max(a, b);
            EigSmem<NP> &s = mats[lj];
            s.pq[li] = make_int2(p, q);
            if (q < M) {
              typename Ar::Ro ro;
              act = Ar::rotation(Ar::a(s, p, p), Ar::a(s, q, q), Ar::a(s, p, q), ro);
              if (act) Ar::rot(s)[li] = ro;
            }
          }
        }
        mask = __ballot_sync(0xffffffffu, act);
        if (T > 32 && lane == 0) smask[t & 1u] = mask;
      }
      if (T > 32) {
        __syncthreads();
        mask = smask[t & 1u];
      }
      if (mask == 0u) continue;
      g::sync();
      for (int j = 0; j < G; ++j) {
        const unsigned seg = (mask >> (j * HP)) & ((HP == 32) ? 0xffffffffu : ((1u << HP) - 1u));
        if (!seg) continue;
        rotated |= 1u << j;
        EigSmem<NP> &s = mats[j];
        const int M = Ms[j], m = (M + 1) >> 1;
        const bool full = NP <= 8 || Ar::kBoth || both[j];
        const int na = ((kColumns ? 2 * m * m : full ? 4 * m * m : 2 * m * (m + 1)) + 31) >> 5, nv = (m * M + 31) >> 5;   // warp steps: blocks of A, V
        const int wid = full ? m : m + ((m & 1) ^ 1);   // the square of blocks, or the triangle of blocks a <= b, folded into rows of equal length
        const float inv_w = __fdividef(1.f, (float)wid), inv_m = __fdividef(1.f, (float)M);
        for (int st = wp; st < na + nv; st += W) {
          if (kColumns && st < na) {
            const int blk = (st << 4) + (lane >> 1);
            const int a = (int)(((float)blk + 0.5f) * inv_w), b = blk - a * m;
            const bool in = blk < m * m, lo_col = (lane & 1) == 0;
            const bool acta = in && ((seg >> a) & 1u), actb = in && ((seg >> b) & 1u);
            int2 pa = make_int2(0, 0);
            int col = 0;
            El xp{}, xq{};
            if (acta || actb) {
              pa = s.pq[a];
              const int2 pb = s.pq[b];
              col = lo_col ? pb.x : pb.y;
              xp = Ar::a(s, pa.x, col);
              xq = Ar::a(s, pa.y, col);
              if (acta) {
                const typename Ar::Ro ro = Ar::rot(s)[a];
                const El np = Ar::mix(ro.c, Ar::neg(ro.sr), ro.si, xp, xq);
                xq = Ar::mix(ro.c, ro.sr, ro.si, xq, xp);
                xp = np;
              }
            }
            const El yp = shfl_xor1(xp), yq = shfl_xor1(xq);   // the block's other column, same rows
            if (acta || actb) {
              if (actb) {
                const typename Ar::Ro ro = Ar::rot(s)[b];
                const auto sr = lo_col ? Ar::neg(ro.sr) : ro.sr;
                xp = Ar::mix(ro.c, sr, Ar::neg(ro.si), xp, yp);
                xq = Ar::mix(ro.c, sr, Ar::neg(ro.si), xq, yq);
              }
              if (a == b) {              // the diagonal of a Hermitian matrix is real
                if (lo_col)
                  xp = Ar::real(xp);
                else
                  xq = Ar::real(xq);
              }
              Ar::a(s, pa.x, col) = xp;
              Ar::a(s, pa.y, col) = xq;
            }
          } else if (st < na) {
            const int blk = (st << 3) + (lane >> 2);
            const int i = (int)(((float)blk + 0.5f) * inv_w), jj = blk - i * wid;
            const bool head = full || jj < m - i;
            const int a = head ? i : (m & 1 ? m - i : m - 1 - i);
            const int b = full ? jj : (head ? i + jj : a + jj - (m - i));
            const bool in = blk < (full ? m * m : (m * (m + 1)) >> 1);
            const bool acta = in && ((seg >> a) & 1u), actb = in && ((seg >> b) & 1u);
            const bool lo_row = (lane & 2) == 0, lo_col = (lane & 1) == 0;
            int row = 0, col = 0;
            El x{};
            if (acta || actb) {
              const int2 pa = s.pq[a], pb = s.pq[b];
              row = lo_row ? pa.x : pa.y;
              col = lo_col ? pb.x : pb.y;
              x = Ar::a(s, row, col);
              if (acta) {
                const typename Ar::Ro ro = Ar::rot(s)[a];
                x = Ar::mix(ro.c, lo_row ? Ar::neg(ro.sr) : ro.sr, ro.si, x, Ar::a(s, lo_row ? pa.y : pa.x, col));
              }
            }
            const El y = shfl_xor1(x);   // the block's other column, same row
            if (acta || actb) {
              if (actb) {
                const typename Ar::Ro ro = Ar::rot(s)[b];
                x = Ar::mix(ro.c, lo_col ? Ar::neg(ro.sr) : ro.sr, Ar::neg(ro.si), x, y);
              }
              if (a == b) {              // the diagonal of a Hermitian matrix is real
                if (lo_row == lo_col)
                  x = Ar::real(x);
                else if (Ar::kZeroes)
                  x = El{};
              } else if (!full) {
                Ar::a(s, col, row) = Ar::conj(x);
              }
              Ar::a(s, row, col) = x;
            }
          } else {
            const int it = ((st - na) << 5) + lane;
            const int i = (int)(((float)it + 0.5f) * inv_m), k = it - i * M;
            if (i < m && ((seg >> i) & 1u)) {
              const typename Ar::Ro ro = Ar::rot(s)[i];
              const int2 pq = s.pq[i];
              const El xp = Ar::v(s, k, pq.x), xq = Ar::v(s, k, pq.y);
              Ar::v(s, k, pq.x) = Ar::mix(ro.c, Ar::neg(ro.sr), Ar::neg(ro.si), xp, xq);
              Ar::v(s, k, pq.y) = Ar::mix(ro.c, ro.sr, Ar::neg(ro.si), xq, xp);
            }
          }
        }
      }
      g::sync();
    }
    // matrices without a rotation in this sweep have converged
    for (int j = 0; j < G; ++j)
      if (((live >> j) & 1u) && !((rotated >> j) & 1u)) {
        res[j] = sweep;
        live &= ~(1u << j);
      }
  }
  for (int j = 0; j < G; ++j)
    if ((live >> j) & 1u) res[j] = -DOA_ENOCONV;
  if constexpr (Ar::kZeroes) {
    for (int j = 0; j < G; ++j)
      if (scaled[j] != 0) {
        for (int e = tid; e < Ms[j]; e += T) mats[j].a(e, e).x = scalbn(mats[j].a(e, e).x, scaled[j]);
        g::sync();
      }
  } else {
    // double-float -> FP64 in place (same bytes per element; every element has one owner lane)
    for (int j = 0; j < G; ++j) {
      const int M = Ms[j];
      if (M <= 0) continue;
      EigSmem<NP> &s = mats[j];
      for (int e = tid; e < M * M; e += T) {
        const int i = e / M, k = e % M;
        const El a = Ar::a(s, i, k), v = Ar::v(s, i, k);
        s.a(i, k) = make_double2((double)a.x + (double)a.y, (double)a.z + (double)a.w);
        s.v(i, k) = make_double2((double)v.x + (double)v.y, (double)v.z + (double)v.w);
      }
    }
    g::sync();
  }
}

// ---- One matrix of 33 <= M <= 64 on a cluster of four CTAs (double-float) ----
// The same rounds as jacobi_group with the rows of A and V spread over the cluster: CTA c owns
// rows 16c .. 16c+15 (one per warp). For a round's rotation J (n/2 disjoint pairs) the element
// (i, col) of J^H A J needs only rows i and partner(i) at the columns of col's pair, so warp w
// forms row i's new values pair by pair (lane j: columns p_j, q_j): first the row mix with the
// partner row (read through distributed shared memory when another CTA owns it), then the column
// mix, in the double-float operations of jacobi_group (which computes half of A and mirrors it,
// where here both halves are computed); V's rows take the column mix in place. A is double-buffered, so one cluster
// barrier per round orders every CTA's reads of the current buffer before the writes that reuse
// it. Warp 0 of every CTA forms the round's rotations from the same bytes with the same code, so
// every CTA takes the same decisions (rounds to skip, sweeps, convergence) and meets the same
// barriers. A round takes about 4500 cycles: 1100 for the rotations (three remote entries, then the
// dependent arithmetic), 2300 for the rows' FP32 work, the rest the cluster barrier; V's third of the FP32
// work fills the time between arriving and waiting there (a 64 x 64 matrix: 1.37 -> 1.22 ms). Eight CTAs
// of 8 rows take 1.01 ms, but 32 matrices at once 3.2 instead of 1.5 ms: not kept.
constexpr int kClRanks = 4;                 // CTAs per matrix
constexpr int kClRows = 64 / kClRanks;      // rows of A and V owned by a CTA (one per warp)
constexpr int kClThreads = 32 * kClRows;
static_assert(kClThreads == cta_threads<64>(), "the cluster's rank 0 runs the M <= 64 finishing code");

struct ClusterDF {
  float4 A[2][kClRows][64];    // double-float (hi, lo) re, (hi, lo) im
  float4 V[kClRows][64];
  RotDF rot[2][32];            // the round's rotations, by round parity
  int2 pq[2][32];
  unsigned mask[2];
};

// Shared memory of a cluster kernel: the FP64 record that rank 0 finishes in, then the rows.
constexpr int kClFinBytes = (int)((sizeof(EigSmem<64>) + 15) / 16 * 16);
constexpr int kClSmemBytes = kClFinBytes + (int)sizeof(ClusterDF);

// Row mixes of A <- J^H A: row p of the pair becomes c x_p - sigma x_q, row q conj(sigma) x_p + c x_q.
__device__ __forceinline__ float4 mix_row_p(const RotDF &ro, float4 xp, float4 xq) {
  return cplx(dot3(ro.c, re_of(xp), neg(ro.sr), re_of(xq), ro.si, im_of(xq)),
              dot3(ro.c, im_of(xp), neg(ro.sr), im_of(xq), neg(ro.si), re_of(xq)));
}
__device__ __forceinline__ float4 mix_row_q(const RotDF &ro, float4 xp, float4 xq) {
  return cplx(dot3(ro.c, re_of(xq), ro.sr, re_of(xp), ro.si, im_of(xp)),
              dot3(ro.c, im_of(xq), ro.sr, im_of(xp), neg(ro.si), re_of(xp)));
}
// Column mix of A <- A J (and V <- V J): column p becomes c x_p - conj(sigma) x_q, column q
// sigma x_p + c x_q.
__device__ __forceinline__ void mix_cols(const RotDF &ro, float4 &xp, float4 &xq) {
  const float4 np = cplx(dot3(ro.c, re_of(xp), neg(ro.sr), re_of(xq), neg(ro.si), im_of(xq)),
                         dot3(ro.c, im_of(xp), neg(ro.sr), im_of(xq), ro.si, re_of(xq)));
  const float4 nq = cplx(dot3(ro.c, re_of(xq), ro.sr, re_of(xp), neg(ro.si), im_of(xp)),
                         dot3(ro.c, im_of(xq), ro.sr, im_of(xp), ro.si, re_of(xp)));
  xp = np;
  xq = nq;
}

// Cyclic Jacobi of the Hermitian M x M matrix R (FP64, row-major; the upper triangle is read) in
// double-float over the calling cluster. Returns the sweep count (> 0), -DOA_ENONFINITE or
// -DOA_ENOCONV, the same in every CTA; on a positive return rank 0's fin holds V and the diagonal
// of A in FP64 (the finishing code reads nothing else of A).
__device__ int jacobi_cluster_df(ClusterDF &w, EigSmem<64> &fin, int M, const double2 *__restrict__ R) {
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank();
  const int tid = threadIdx.x, wp = tid >> 5, lane = tid & 31;
  const int row = rank * kClRows + wp;
  // every CTA checks the whole upper triangle, so all reach the same verdict
  bool finite = true;
  for (int e = tid; e < M * M; e += kClThreads) {
    const int i = e / M, k = e % M;
    if (i > k) continue;
    const double2 v = R[e];
    finite = finite && isfinite(v.x) && (i == k || isfinite(v.y));
  }
  for (int e = tid; e < kClRows * 64; e += kClThreads) {
    const int li = e / 64, k = e % 64, i = rank * kClRows + li;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), v = a;
    if (i < M && k < M) {
      double2 x;
      if (i <= k) {
        x = R[i * M + k];
      } else {
        x = R[k * M + i];
        x.y = -x.y;
      }
      if (i == k) x.y = 0.0;
      a = df_of(x);
      v.x = i == k ? 1.f : 0.f;
    }
    w.A[0][li][k] = a;
    w.A[1][li][k] = make_float4(0.f, 0.f, 0.f, 0.f);
    w.V[li][k] = v;
  }
  const bool ok = __syncthreads_and(finite) != 0;
  cl.sync();   // every CTA's rows are in place before the first remote read
  if (!ok) return -DOA_ENONFINITE;
  const int n = (M + 1) & ~1;
  int cur = 0, res = -DOA_ENOCONV;
  unsigned t = 0;   // rounds so far: the parity selects the rotation record
  for (int sweep = 1; sweep <= kMaxSweeps; ++sweep) {
    bool rotated = false;
    for (int r = 0; r < n - 1; ++r, ++t) {
      const int sl = (int)(t & 1u);
      if (wp == 0) {
        bool act = false;
        if (lane < n / 2) {
          const int a = rr_player(lane, r, n), b = rr_player(n - 1 - lane, r, n);
          const int p = min(a, b), q = max(a, b);
          w.pq[sl][lane] = make_int2(p, q);
          if (q < M) {
            const float4 *Ap = cl.map_shared_rank(&w.A[cur][p % kClRows][0], p / kClRows);
            const float4 *Aq = cl.map_shared_rank(&w.A[cur][q % kClRows][0], q / kClRows);
            RotDF ro;
            act = rotation_df_of(Ap[p], Aq[q], Ap[q], ro);
            if (act) w.rot[sl][lane] = ro;
          }
        }
        const unsigned m = __ballot_sync(0xffffffffu, act);
        if (lane == 0) w.mask[sl] = m;
      }
      __syncthreads();
      const unsigned mask = w.mask[sl];
      if (mask == 0u) continue;   // nothing written: the buffers stay as they are
      rotated = true;
      const int nxt = cur ^ 1;
      const bool mine = row < M && lane < n / 2;
      const int2 pj = mine ? w.pq[sl][lane] : make_int2(0, 0);
      if (mine) {
        float4 xp = w.A[cur][wp][pj.x], xq = w.A[cur][wp][pj.y];
        // the pair that holds this row: its position in the round-robin order, folded
        const int back = row - 1 - r;
        const int pos = row == 0 ? 0 : (back < 0 ? back + n - 1 : back) + 1;
        const int k = min(pos, n - 1 - pos);
        if ((mask >> k) & 1u) {
          const RotDF rk = w.rot[sl][k];
          const int2 pk = w.pq[sl][k];
          const int other = pk.x + pk.y - row;
          const float4 *Ao = cl.map_shared_rank(&w.A[cur][other % kClRows][0], other / kClRows);
          const float4 yp = Ao[pj.x], yq = Ao[pj.y];
          if (row == pk.x) {
            xp = mix_row_p(rk, xp, yp);
            xq = mix_row_p(rk, xq, yq);
          } else {
            xp = mix_row_q(rk, yp, xp);
            xq = mix_row_q(rk, yq, xq);
          }
        }
        if ((mask >> lane) & 1u) mix_cols(w.rot[sl][lane], xp, xq);
        if (row == pj.x) xp.z = xp.w = 0.f;   // the diagonal of a Hermitian matrix is real
        if (row == pj.y) xq.z = xq.w = 0.f;
        w.A[nxt][wp][pj.x] = xp;
        w.A[nxt][wp][pj.y] = xq;
      }
      // the round's barrier: its writes become visible, and nobody still reads the old buffer; V, whose
      // rows are nobody else's, is mixed while the other CTAs arrive
      cl.barrier_arrive();
      if (mine && ((mask >> lane) & 1u)) {
        float4 vp = w.V[wp][pj.x], vq = w.V[wp][pj.y];
        mix_cols(w.rot[sl][lane], vp, vq);
        w.V[wp][pj.x] = vp;
        w.V[wp][pj.y] = vq;
      }
      cl.barrier_wait();
      cur = nxt;
    }
    if (!rotated) {
      res = sweep;
      break;
    }
  }
  if (res > 0 && rank == 0) {
    for (int e = tid; e < M * M; e += kClThreads) {
      const int i = e / M, k = e % M;
      const float4 v = cl.map_shared_rank(&w.V[i % kClRows][0], i / kClRows)[k];
      fin.v(i, k) = make_double2((double)v.x + (double)v.y, (double)v.z + (double)v.w);
      if (i == k) {
        const float4 a = cl.map_shared_rank(&w.A[cur][i % kClRows][0], i / kClRows)[i];
        fin.a(i, i) = make_double2((double)a.x + (double)a.y, (double)a.z + (double)a.w);
      }
    }
  }
  cl.sync();   // the other CTAs' rows stay in place until rank 0 has read them
  return res;
}

// Stable descending order of the eigenvalues (equal values keep index order).
template <int NP, int T>
__device__ void sort_desc(int M, EigSmem<NP> &s) {
  using g = Grp<T>;
  const int lane = g::id();
  for (int i = lane; i < M; i += T) s.lam()[i] = s.a(i, i).x;
  g::sync();
  // ranks form a permutation even for non-finite values (NaN ranks below every number)
  for (int i = lane; i < M; i += T) {
    const double li = isnan(s.lam()[i]) ? -INFINITY : s.lam()[i];
    int rank = 0;
    for (int j = 0; j < M; ++j) {
      const double lj = isnan(s.lam()[j]) ? -INFINITY : s.lam()[j];
      rank += (lj > li) || (lj == li && j < i);
    }
    s.order()[rank] = i;
  }
  g::sync();
}

// Writes B (column-major, ld M) of algorithm alg; returns 0 or a doa_status.
template <int NP, int T>
__device__ int build_factor(int M, int d, int alg, EigSmem<NP> &s, double2 *__restrict__ B) {
  using g = Grp<T>;
  const int lane = g::id();
  const int Kn = M - d;  // noise subspace dimension
  if (alg == DOA_PHD) {
    int col = s.order()[M - 1];
    for (int r = lane; r < M; r += T) B[r] = s.v(r, col);
    return 0;
  }
  if (alg == DOA_MUSIC || alg == DOA_EV) {
    bool bad = false;
    for (int e = lane; e < M * Kn; e += T) {
      int c = e / M, r = e % M;
      int col = s.order()[d + c];
      double2 v = s.v(r, col);
      if (alg == DOA_EV) {
        double l = s.lam()[col];
        if (!(l > 0.0)) {
          bad = true;
          v = make_double2(0.0, 0.0);
        } else {
          double w = 1.0 / sqrt(l);
          v.x *= w;
          v.y *= w;
        }
      }
      B[c * M + r] = v;
    }
    bad = g::any(bad);
    return bad ? DOA_ERANK : 0;
  }
  // MN: valph = P_n e1 / (e1^H P_n e1); (P_n e1)_r = sum_c V[r][c] conj(V[0][c]) over noise c
  double nrm = 0.0;
  for (int c = 0; c < Kn; ++c) {
    double2 g = s.v(0, s.order()[d + c]);
    nrm += g.x * g.x + g.y * g.y;
  }
  if (!(nrm > 0.0)) {
    for (int r = lane; r < M; r += T) B[r] = make_double2(0.0, 0.0);
    return DOA_ERANK;
  }
  const double inv = 1.0 / nrm;
  for (int r = lane; r < M; r += T) {
    double2 acc = make_double2(0.0, 0.0);
    for (int c = 0; c < Kn; ++c) {
      int col = s.order()[d + c];
      double2 v = s.v(r, col), g = s.v(0, col);
      // v * conj(g)
      acc.x += v.x * g.x + v.y * g.y;
      acc.y += v.y * g.x - v.x * g.y;
    }
    B[r] = make_double2(acc.x * inv, acc.y * inv);
  }
  return 0;
}

// FP64 check that the noise eigenvectors are orthonormal: max |E_n^H E_n - I| <= kOrthoTol.
constexpr double kOrthoTol = 1e-10;

template <int NP, int T>
__device__ bool noise_orthonormal(int M, int d, EigSmem<NP> &s) {
  using g = Grp<T>;
  const int lane = g::id();
  const int Kn = M - d;
  bool ok = true;
  for (int e = lane; e < Kn * Kn; e += T) {
    const int a = e / Kn, b = e % Kn;
    if (a > b) continue;
    const int ca = s.order()[d + a], cb = s.order()[d + b];
    double gr = 0.0, gi = 0.0;
    for (int r = 0; r < M; ++r) {   // conj(V[r][ca]) * V[r][cb]
      const double2 x = s.v(r, ca), y = s.v(r, cb);
      gr = fma(x.x, y.x, fma(x.y, y.y, gr));
      gi = fma(x.x, y.y, fma(-x.y, y.x, gi));
    }
    if (a == b) gr -= 1.0;
    ok = ok && fabs(gr) <= kOrthoTol && fabs(gi) <= kOrthoTol;
  }
  return g::all(ok);
}

// Model-order estimates (Wax and Kailath's criteria for complex data) from the sorted eigenvalues:
// for k assumed sources, L(k) = N (M-k) log(a/g) over the M-k smallest eigenvalues (arithmetic and
// geometric means; +inf when one is not positive), MDL(k) = L + k(2M-k) log(N)/2, AIC(k) = 2L +
// 2k(2M-k); out[0] = argmin MDL, out[1] = argmin AIC (the smaller k on a tie). The group's lanes
// take one k each; the criterion values go to the A matrix's first row (no longer needed here).
template <int NP, int T>
__device__ void model_order(int M, int N, EigSmem<NP> &s, int32_t *out) {
  using g = Grp<T>;
  const int lane = g::id();
  const double logN = log((double)N);
  for (int k = lane; k < M; k += T) {
    const int n = M - k;
    double sum = 0.0, ls = 0.0;
    bool bad = false;
    for (int i = k; i < M; ++i) {
      const double l = s.lam()[s.order()[i]];
      sum += l;
      if (l > 0.0) ls += log(l); else bad = true;
    }
    const double L = bad ? CUDART_INF : (double)N * (double)n * (log(sum / (double)n) - ls / (double)n);
    const double pen = (double)k * (double)(2 * M - k);
    s.a(0, k) = make_double2(L + 0.5 * pen * logN, 2.0 * L + 2.0 * pen);
  }
  g::sync();
  if (lane == 0) {
    int bm = 0, ba = 0;
    double vm = CUDART_INF, va = CUDART_INF;
    for (int k = 0; k < M; ++k) {
      const double2 v = s.a(0, k);
      if (v.x < vm) {
        vm = v.x;
        bm = k;
      }
      if (v.y < va) {
        va = v.y;
        ba = k;
      }
    }
    out[0] = bm;
    out[1] = ba;
  }
  g::sync();
}

// Writes a batch problem's scan factor F (columns as laid out by the plan: E_n, or v_min; then
// valph) and the EV weights w_c = 1 / lambda_{d+c}; returns 0 or a doa_status.
template <int NP, int T>
__device__ int build_scan_factor(const PlanProblem &pp, EigSmem<NP> &s, double2 *__restrict__ F,
                                 double *__restrict__ w) {
  using g = Grp<T>;
  const int lane = g::id();
  const int M = pp.p.M, d = pp.p.d;
  int st = 0;
  if (pp.Kn > 0) {
    build_factor<NP, T>(M, d, DOA_MUSIC, s, F);
    if (pp.slot[DOA_EV] >= 0) {
      bool bad = false;
      for (int c = lane; c < pp.Kn; c += T) {
        const double l = s.lam()[s.order()[d + c]];
        bad = bad || !(l > 0.0);
        w[c] = l > 0.0 ? 1.0 / l : 0.0;
      }
      if (g::any(bad)) st = DOA_ERANK;
    }
  } else if (pp.kphd >= 0) {
    build_factor<NP, T>(M, d, DOA_PHD, s, F + (size_t)pp.kphd * M);
  }
  if (pp.kmn >= 0) {
    const int e = build_factor<NP, T>(M, d, DOA_MN, s, F + (size_t)pp.kmn * M);
    if (e && !st) st = e;
  }
  return st;
}

// The eigenvalues, B and the status of a single call from a finished decomposition (res: the
// sweep count, or minus a doa_status).
template <int NP, int T>
__device__ void finish_single(int M, int d, int alg, EigSmem<NP> &s, int res, double *evals, double2 *B, int *K_out,
                              int *info) {
  const int lane = Grp<T>::id();
  int st = 0;
  if (res > 0) {
    sort_desc<NP, T>(M, s);
    if (evals)
      for (int i = lane; i < M; i += T) evals[i] = s.lam()[s.order()[i]];
    st = build_factor<NP, T>(M, d, alg, s, B);
  } else {
    st = -res;
  }
  if (lane == 0) {
    *info = st ? -st : res;
    if (K_out) *K_out = (alg == DOA_PHD || alg == DOA_MN) ? 1 : M - d;
  }
}

template <int NP, bool kDF>
using Arith = std::conditional_t<kDF, ArithDF<NP>, ArithF64<NP>>;

template <int NP, bool kDF>
__global__ void __launch_bounds__(cta_threads<NP, kDF>()) eig_single_kernel(const double2 *R64, int M, int d, int alg, double *evals,
                                                       double2 *B, int *K_out, int *info) {
  start_after_previous();
  let_next_start();
  extern __shared__ __align__(16) uint8_t smem[];
  constexpr int T = cta_threads<NP, kDF>();
  EigSmem<NP> *mats = reinterpret_cast<EigSmem<NP> *>(smem);
  const int Ms[1] = {M};
  const double2 *Rs[1] = {R64};
  const bool both[1] = {false};
  int res[1];
  jacobi_group<Arith<NP, kDF>, NP, 1, T>(mats, Ms, Rs, both, res);
  finish_single<NP, T>(M, d, alg, mats[0], res[0], evals, B, K_out, info);
}

// Single call, 33 <= M <= 64, double-float: one four-CTA cluster; rank 0 finishes.
__global__ void __cluster_dims__(kClRanks, 1, 1) __launch_bounds__(kClThreads, 1)
    eig_cluster_single_kernel(const double2 *R64, int M, int d, int alg, double *evals, double2 *B, int *K_out,
                              int *info) {
  start_after_previous();
  let_next_start();
  extern __shared__ __align__(16) uint8_t smem[];
  EigSmem<64> &s = *reinterpret_cast<EigSmem<64> *>(smem);
  ClusterDF &w = *reinterpret_cast<ClusterDF *>(smem + kClFinBytes);
  const int res = jacobi_cluster_df(w, s, M, R64);
  if (cg::this_cluster().block_rank() != 0) return;
  finish_single<64, kClThreads>(M, d, alg, s, res, evals, B, K_out, info);
}

// A batch problem's outputs from its finished decomposition (res: the sweep count, or minus a
// doa_status): evals, the scan factor and EV weights, the optional B, order estimates and
// proposal features, and the status.
template <int NP, int T>
__device__ void finish_batch(const PlanProblem &pp, const PlanJob *jobs, EigSmem<NP> &s, int res, uint8_t *ws,
                             int *status) {
  const int lane = Grp<T>::id();
  const int M = pp.p.M, d = pp.p.d;
  int st = 0;
  if (pp.p.features) {
    // proposal-network input: upper triangle of R / tr(R), (re, im) pairs row by row
    const double2 *R = reinterpret_cast<const double2 *>(ws + pp.r64_off);
    double tr = 0.0;
    for (int i = 0; i < M; ++i) tr += R[i * M + i].x;
    const double inv = tr > 0.0 ? 1.0 / tr : 0.0;
    for (int e = lane; e < M * (M + 1) / 2; e += T) {
      int i = 0, rem = e;
      while (rem >= M - i) { rem -= M - i; ++i; }
      const double2 v = R[i * M + i + rem];
      pp.p.features[2 * e] = (float)(v.x * inv);
      pp.p.features[2 * e + 1] = (float)(v.y * inv);
    }
  }
  double2 *F = reinterpret_cast<double2 *>(ws + pp.fac_off);
  double *w = reinterpret_cast<double *>(F + (size_t)M * (M + 1));
  if (res > 0) {
    sort_desc<NP, T>(M, s);
    if (pp.p.evals)
      for (int i = lane; i < M; i += T) pp.p.evals[i] = s.lam()[s.order()[i]];
    st = build_scan_factor<NP, T>(pp, s, F, w);
    if (!noise_orthonormal<NP, T>(M, d, s) && !st) st = DOA_ENOCONV;
    if (pp.p.B_out) build_factor<NP, T>(M, d, jobs[pp.first_job].alg, s, reinterpret_cast<double2 *>(pp.p.B_out));
    if (pp.p.order_est) {
      Grp<T>::sync();
      model_order<NP, T>(M, pp.p.N, s, pp.p.order_est);
    }
  } else {
    st = -res;
    // a failed decomposition leaves a zero factor, so the scan writes the 1/FLT_MIN sentinel
    for (int e = lane; e < M * pp.Kf; e += T) F[e] = make_double2(0.0, 0.0);
    for (int e = lane; e < pp.Kn; e += T) w[e] = 0.0;
  }
  if (lane == 0) *status = st;
  Grp<T>::sync();
}

template <int NP, int G>
__global__ void __launch_bounds__(32 * eig_warps<NP>(), eig_min_ctas<NP>()) eig_batch_kernel(const uint8_t *plan, uint8_t *ws, int bucket,
                                                                         int *status, int dep) {
  if (dep) start_after_previous();
  let_next_start();
  extern __shared__ __align__(16) uint8_t smem[];
  const int grp = threadIdx.x / 32;
  EigSmem<NP> *mats = reinterpret_cast<EigSmem<NP> *>(smem) + grp * G;
  const PlanHeader *h = reinterpret_cast<const PlanHeader *>(plan);
  const int base = (blockIdx.x * (int)(blockDim.x / 32) + grp) * G;
  const int count = h->eig_count[bucket];
  if (base >= count) return;
  const int32_t *list = reinterpret_cast<const int32_t *>(plan + h->off_eig[bucket]);
  const PlanProblem *probs = reinterpret_cast<const PlanProblem *>(plan + h->off_prob);
  const PlanJob *jobs = reinterpret_cast<const PlanJob *>(plan + h->off_job);
  int Ms[G], prob[G], res[G];
  const double2 *Rs[G];
  for (int j = 0; j < G; ++j) {
    prob[j] = base + j < count ? list[base + j] : -1;
    Ms[j] = prob[j] >= 0 ? probs[prob[j]].p.M : 0;
    Rs[j] = prob[j] >= 0 ? reinterpret_cast<const double2 *>(ws + probs[prob[j]].r64_off) : nullptr;
  }
  bool fp64 = false;   // a group runs FP64 when any of its problems asks for it
  bool both[G];
  for (int j = 0; j < G; ++j) both[j] = prob[j] >= 0 && probs[prob[j]].p.geom.pos != nullptr;
  for (int j = 0; j < G; ++j) fp64 = fp64 || (prob[j] >= 0 && probs[prob[j]].p.eig_prec == DOA_EIG_FP64);
  if (fp64)
    jacobi_group<ArithF64<NP>, NP, G, 32>(mats, Ms, Rs, both, res);
  else
    jacobi_group<ArithDF<NP>, NP, G, 32>(mats, Ms, Rs, both, res);
  for (int j = 0; j < G; ++j) {
    if (prob[j] < 0) continue;
    finish_batch<NP, 32>(probs[prob[j]], jobs, mats[j], res[j], ws, status + prob[j]);
  }
  end_after_previous();
}

// The CTA form of the batch: a CTA of T threads per matrix.
template <int NP, int T>
__global__ void __launch_bounds__(T) eig_batch_cta_kernel(const uint8_t *plan, uint8_t *ws, int bucket, int *status,
                                                          int dep) {
  if (dep) start_after_previous();
  let_next_start();
  extern __shared__ __align__(16) uint8_t smem[];
  EigSmem<NP> &s = *reinterpret_cast<EigSmem<NP> *>(smem);
  const PlanHeader *h = reinterpret_cast<const PlanHeader *>(plan);
  const int prob = reinterpret_cast<const int32_t *>(plan + h->off_eig[bucket])[blockIdx.x];
  const PlanProblem &pp = reinterpret_cast<const PlanProblem *>(plan + h->off_prob)[prob];
  const PlanJob *jobs = reinterpret_cast<const PlanJob *>(plan + h->off_job);
  const int Ms[1] = {pp.p.M};
  const double2 *Rs[1] = {reinterpret_cast<const double2 *>(ws + pp.r64_off)};
  const bool both[1] = {pp.p.geom.pos != nullptr};
  int res[1];
  if (pp.p.eig_prec == DOA_EIG_FP64)
    jacobi_group<ArithF64<NP>, NP, 1, T>(&s, Ms, Rs, both, res);
  else
    jacobi_group<ArithDF<NP>, NP, 1, T>(&s, Ms, Rs, both, res);
  finish_batch<NP, T>(pp, jobs, s, res[0], ws, status + prob);
  end_after_previous();
}

// Bucket M <= 64 of the batch in double-float: one four-CTA cluster per problem; rank 0 finishes.
// A problem that asks for the FP64 Jacobi runs it in rank 0 alone (the other CTAs leave at once).
__global__ void __cluster_dims__(kClRanks, 1, 1) __launch_bounds__(kClThreads, 1)
    eig_cluster_batch_kernel(const uint8_t *plan, uint8_t *ws, int bucket, int *status, int dep) {
  if (dep) start_after_previous();
  let_next_start();
  extern __shared__ __align__(16) uint8_t smem[];
  EigSmem<64> &s = *reinterpret_cast<EigSmem<64> *>(smem);
  ClusterDF &w = *reinterpret_cast<ClusterDF *>(smem + kClFinBytes);
  const PlanHeader *h = reinterpret_cast<const PlanHeader *>(plan);
  const int idx = (int)(blockIdx.x / kClRanks);   // the same for every CTA of the cluster
  if (idx >= h->eig_count[bucket]) return;
  const int32_t *list = reinterpret_cast<const int32_t *>(plan + h->off_eig[bucket]);
  const PlanProblem *probs = reinterpret_cast<const PlanProblem *>(plan + h->off_prob);
  const PlanJob *jobs = reinterpret_cast<const PlanJob *>(plan + h->off_job);
  const int prob = list[idx];
  const PlanProblem &pp = probs[prob];
  const double2 *R = reinterpret_cast<const double2 *>(ws + pp.r64_off);
  const bool rank0 = cg::this_cluster().block_rank() == 0;
  int res;
  if (pp.p.eig_prec == DOA_EIG_FP64) {
    if (!rank0) return;
    int Ms[1] = {pp.p.M}, r1[1];
    const double2 *Rs[1] = {R};
    const bool both[1] = {pp.p.geom.pos != nullptr};
    jacobi_group<ArithF64<64>, 64, 1, kClThreads>(&s, Ms, Rs, both, r1);
    res = r1[0];
  } else {
    res = jacobi_cluster_df(w, s, pp.p.M, R);
    if (!rank0) return;
  }
  finish_batch<64, kClThreads>(pp, jobs, s, res, ws, status + prob);
  end_after_previous();
}


template <int NP, bool kDF>
cudaError_t run_single_p(const double2 *R64, int M, int d, int alg, double *evals, double2 *B, int *K_out,
                         int *info, cudaStream_t st) {
  const int smem = (int)sizeof(EigSmem<NP>);
  cudaError_t e = ensure_smem_attr((const void *)eig_single_kernel<NP, kDF>, smem);
  if (e != cudaSuccess) return e;
  return launch_chained(eig_single_kernel<NP, kDF>, 1, cta_threads<NP, kDF>(), smem, st, R64, M, d, alg, evals, B, K_out, info);
}

cudaError_t run_single_cluster(const double2 *R64, int M, int d, int alg, double *evals, double2 *B, int *K_out,
                               int *info, cudaStream_t st) {
  cudaError_t e = ensure_smem_attr(reinterpret_cast<const void *>(eig_cluster_single_kernel), kClSmemBytes);
  if (e != cudaSuccess) return e;
  return launch_chained(eig_cluster_single_kernel, kClRanks, kClThreads, kClSmemBytes, st, R64, M, d, alg, evals, B, K_out,
                          info);
}

template <int NP>
cudaError_t run_single(const double2 *R64, int M, int d, int alg, int prec, double *evals, double2 *B, int *K_out,
                       int *info, cudaStream_t st) {
  if (prec == DOA_EIG_FP64) return run_single_p<NP, false>(R64, M, d, alg, evals, B, K_out, info, st);
  if constexpr (NP == 64)
    return run_single_cluster(R64, M, d, alg, evals, B, K_out, info, st);
  else
    return run_single_p<NP, true>(R64, M, d, alg, evals, B, K_out, info, st);
}

// Warps per CTA: the count (up to eig_warps) that keeps the most matrices resident per SM, the
// larger count on a tie. Shared memory is the limit (each CTA also costs the driver's reserve),
// so for M <= 16, nine one-matrix warps per CTA hold 27 matrices per SM where two held 24: a
// 4096-matrix batch then runs in one wave instead of 1.12.
template <int NP, int G>
int eig_cta_warps() {
  const SmemLimits lim = device_smem_limits();
  const int per_mat = (int)sizeof(EigSmem<NP>);
  int best = 1, best_res = -1;
  for (int w = 1; w <= eig_warps<NP>(); ++w) {
    const int bytes = w * G * per_mat;
    if (bytes > lim.per_block) break;
    const int ctas = lim.per_sm / (bytes + lim.reserve);
    if (ctas * w * G >= best_res) {
      best_res = ctas * w * G;
      best = w;
    }
  }
  return best;
}

template <int NP, int G>
cudaError_t run_batch_g(const uint8_t *plan, int count, uint8_t *ws, int *status, int bucket, bool beside, cudaStream_t st) {
  const int W = eig_cta_warps<NP, G>();
  const int per_cta = W * G;
  const int smem = (int)sizeof(EigSmem<NP>) * per_cta;
  cudaError_t e = ensure_smem_attr(reinterpret_cast<const void *>(eig_batch_kernel<NP, G>), smem);
  if (e != cudaSuccess) return e;
  return launch_programmatic(beside || chained_grid((count + per_cta - 1) / per_cta, true), eig_batch_kernel<NP, G>,
                             (count + per_cta - 1) / per_cta, 32 * W, smem, st, plan, ws, bucket, status,
                          (int)!beside);
}

template <int NP, int T>
cudaError_t run_batch_cta_t(const uint8_t *plan, int count, uint8_t *ws, int *status, int bucket, bool beside, cudaStream_t st) {
  const int smem = (int)sizeof(EigSmem<NP>);
  cudaError_t e = ensure_smem_attr(reinterpret_cast<const void *>(eig_batch_cta_kernel<NP, T>), smem);
  if (e != cudaSuccess) return e;
  return launch_programmatic(beside || chained_grid(count, true), eig_batch_cta_kernel<NP, T>, count, T, smem, st, plan,
                             ws, bucket, status, (int)!beside);
}

template <int NP>
cudaError_t run_batch_cta(const uint8_t *plan, const PlanHeader &h, uint8_t *ws, int *status, int bucket, bool beside, cudaStream_t st) {
  const int count = h.eig_count[bucket];
  if (count == 0) return cudaSuccess;
  return (h.eig_fp64 >> bucket) & 1
             ? run_batch_cta_t<NP, cta_threads<NP, false>()>(plan, count, ws, status, bucket, beside, st)
             : run_batch_cta_t<NP, cta_threads<NP>()>(plan, count, ws, status, bucket, beside, st);
}

// M <= 16: the CTA form for small batches unless the plan packs matrices (G in {1, 2, 4, 8} up to the
// bucket's maximum per warp), else the warp form.
template <int NP>
cudaError_t run_batch(const uint8_t *plan, const PlanHeader &h, uint8_t *ws, int *status, int bucket,
                      bool beside, cudaStream_t st) {
  const int count = h.eig_count[bucket];
  const int g = h.eig_mats[bucket];
  if (g == 1 && count <= eig_cta_limit<NP>()) return run_batch_cta<NP>(plan, h, ws, status, bucket, beside, st);
  if (count == 0) return cudaSuccess;
  if (g >= 8 && mats_per_warp<NP>() >= 8) return run_batch_g<NP, (mats_per_warp<NP>() >= 8 ? 8 : 1)>(plan, count, ws, status, bucket, beside, st);
  if (g >= 4) return run_batch_g<NP, 4>(plan, count, ws, status, bucket, beside, st);
  if (g >= 2) return run_batch_g<NP, 2>(plan, count, ws, status, bucket, beside, st);
  return run_batch_g<NP, 1>(plan, count, ws, status, bucket, beside, st);
}

// Bucket M <= 64: one four-CTA cluster per problem.
cudaError_t run_batch_cluster(const uint8_t *plan, const PlanHeader &h, uint8_t *ws, int *status, int bucket,
                              bool beside, cudaStream_t st) {
  const int count = h.eig_count[bucket];
  if (count == 0) return cudaSuccess;
  cudaError_t e = ensure_smem_attr(reinterpret_cast<const void *>(eig_cluster_batch_kernel), kClSmemBytes);
  if (e != cudaSuccess) return e;
  return launch_programmatic(beside || chained_grid((int64_t)count * kClRanks, true), eig_cluster_batch_kernel, (int64_t)count * kClRanks, kClThreads, kClSmemBytes, st, plan, ws, bucket,
                          status, (int)!beside);
}

}  // namespace

namespace {
__global__ void __launch_bounds__(32) model_order_single_kernel(const double *evals, int M, int N, int *mdl, int *aic) {
  __shared__ double2 v[kMaxM];
  const int lane = threadIdx.x;
  const double logN = log((double)N);
  for (int k = lane; k < M; k += 32) {
    const int n = M - k;
    double sum = 0.0, ls = 0.0;
    bool bad = false;
    for (int i = k; i < M; ++i) {
      const double l = evals[i];
      sum += l;
      if (l > 0.0) ls += log(l); else bad = true;
    }
    const double L = bad ? CUDART_INF : (double)N * (double)n * (log(sum / (double)n) - ls / (double)n);
    const double pen = (double)k * (double)(2 * M - k);
    v[k] = make_double2(L + 0.5 * pen * logN, 2.0 * L + 2.0 * pen);
  }
  __syncwarp();
  if (lane == 0) {
    int bm = 0, ba = 0;
    double vm = CUDART_INF, va = CUDART_INF;
    for (int k = 0; k < M; ++k) {
      if (v[k].x < vm) {
        vm = v[k].x;
        bm = k;
      }
      if (v[k].y < va) {
        va = v[k].y;
        ba = k;
      }
    }
    if (mdl) *mdl = bm;
    if (aic) *aic = ba;
  }
}
}  // namespace

cudaError_t launch_model_order_single(const double *evals, int M, int N, int *mdl, int *aic, cudaStream_t s) {
  model_order_single_kernel<<<1, 32, 0, s>>>(evals, M, N, mdl, aic);
  return cudaGetLastError();
}

cudaError_t launch_eig_single(const double2 *R64, int M, int d, int alg, int prec, double *evals, double2 *B,
                              int *K_out, int *info, cudaStream_t s) {
  switch (m_bucket(M)) {
    case 0: return run_single<8>(R64, M, d, alg, prec, evals, B, K_out, info, s);
    case 1: return run_single<16>(R64, M, d, alg, prec, evals, B, K_out, info, s);
    case 2: return run_single<32>(R64, M, d, alg, prec, evals, B, K_out, info, s);
    default: return run_single<64>(R64, M, d, alg, prec, evals, B, K_out, info, s);
  }
}

cudaError_t launch_eig_batch(const uint8_t *plan_dev, const PlanHeader &h, uint8_t *ws, int *status,
                             cudaStream_t s) {
  cudaError_t e;
  // the buckets beside each other, the largest matrices first: theirs take longest
  bool beside = false;
  if ((e = run_batch_cluster(plan_dev, h, ws, status, 3, beside, s)) != cudaSuccess) return e;
  beside = beside || h.eig_count[3] > 0;
  if ((e = run_batch_cta<32>(plan_dev, h, ws, status, 2, beside, s)) != cudaSuccess) return e;
  beside = beside || h.eig_count[2] > 0;
  if ((e = run_batch<16>(plan_dev, h, ws, status, 1, beside, s)) != cudaSuccess) return e;
  beside = beside || h.eig_count[1] > 0;
  return run_batch<8>(plan_dev, h, ws, status, 0, beside, s);
}

}  // namespace doa
