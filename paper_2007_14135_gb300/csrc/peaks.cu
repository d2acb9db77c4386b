// Step-6 (Table 2): findPeaks + PeakSelection(peakVals, inds, D), one CTA or one cluster of eight per
// spectrum.
//
// A peak is the left end i of a maximal run [i..j] of equal values with 1 <= i, j <= L-2,
// P[i-1] < P[i] and P[j+1] < P[j]. The D largest peaks are selected (equal values: lower
// index first) and written in ascending index order.
//
// Thread t owns the aligned quads of four points t, t + 256, ... (16-byte coalesced loads) and
// keeps its best kCache peaks in registers. Each warp picks its D best in D rounds of a warp
// arg-max (the winning lane pops its head and, if its cache runs dry while it still has peaks,
// rescans its quads for the next ones below its last selected peak); one warp then merges the
// warps' lists. This realises the shared-memory max-reduction that the paper names as future work
// for Step-6 (Sec. 6). With a cluster the quads are dealt over all its threads and rank 0 merges the
// CTAs' lists through distributed shared memory in the same way: one CTA reads a long spectrum at the
// rate its loads in flight allow (150 us for 360 001 points; the cluster: 45 us), which leaves most of
// the chip idle when the spectra are few, and trails the batch when a few are long.
#include <cooperative_groups.h>

#include <climits>

#include "doa_internal.cuh"
#include "peaks_common.cuh"

namespace doa {
namespace {

using namespace pk;

// Writes the nsel selected peaks in ascending index order (thread 0).
__device__ void write_sel(Cand *sel, int nsel, int *idx, float *val, int *count) {
  if (threadIdx.x == 0) {
    for (int a = 1; a < nsel; ++a) {
      Cand c = sel[a];
      int b = a - 1;
      while (b >= 0 && sel[b].i > c.i) {
        sel[b + 1] = sel[b];
        --b;
      }
      sel[b + 1] = c;
    }
    for (int a = 0; a < nsel; ++a) {
      idx[a] = sel[a].i;
      val[a] = sel[a].v;
    }
    *count = nsel;
  }
}

namespace cg = cooperative_groups;
constexpr int kPeakCluster = 8;
// Points from which a spectrum takes a cluster, one CTA / cluster: smooth spectra the same from here to 16384
// (13 us); rough ones (a peak in most quads) 20 / 12 us at 4096, 24 / 7 at 8192, 35 / 8 at 16383.
constexpr int kClusterPoints = 4096;

// This CTA's share of a spectrum's quads: rank of kCs CTAs of T threads.
template <int kCs, int T>
struct Share {
  int first, stride, rank;
  __device__ Share() {
    rank = kCs > 1 ? (int)cg::this_cluster().block_rank() : 0;
    first = rank * T + (int)threadIdx.x;
    stride = kCs * T;
  }
};

// Merges the cluster's lists (sel, n per CTA, best first) into rank 0's out; every CTA calls it. Returns
// the count (rank 0).
template <int kCs>
__device__ int merge_lists(int want, const Cand *sel, int n, Cand *out) {
  __shared__ int s_n, s_total;
  cg::cluster_group cl = cg::this_cluster();
  if (threadIdx.x == 0) s_n = n;
  cl.sync();
  if (cl.block_rank() == 0 && threadIdx.x < 32) {
    const int lane = threadIdx.x, src = min(lane, kCs - 1);
    const Cand *rs = cl.map_shared_rank(sel, src);
    const int rn = lane < kCs ? *cl.map_shared_rank(&s_n, src) : 0;
    const Cand none{0.f, INT_MAX};
    int pos = 0, total = 0;
    for (int r = 0; r < want; ++r) {
      const Cand mine = pos < rn ? rs[pos] : none;
      const Cand w = warp_best(mine);
      if (w.i == INT_MAX) break;
      if (lane == 0) out[total] = w;
      ++total;
      if (mine.i == w.i) ++pos;
    }
    if (lane == 0) s_total = total;
  }
  cl.sync();   // the lists stay in place until rank 0 has read them
  return s_total;
}

// next (nullable): receives the value of the (d+1)-th best peak (-inf if there is none).
template <int kCs, int T>
__device__ void peaks_block(const float *__restrict__ P, int L, int d, int *idx, float *val, int *count,
                            float *next = nullptr) {
  __shared__ Cand sel[kMaxM + 1], all[kCs > 1 ? kMaxM + 1 : 1];
  const int want = next ? d + 1 : d;
  const Share<kCs, T> sh;
  int nsel = select_rounds<T>(want, sel, [&](const Cand &thr, Cand (&cache)[kCache], int &n) {
    return fill(P, L, sh.first, sh.stride, thr, cache, n);
  });
  Cand *best = sel;
  if (kCs > 1) {
    nsel = merge_lists<kCs>(want, sel, nsel, all);
    best = all;
    if (sh.rank != 0) return;
  }
  if (next) {
    if (threadIdx.x == 0) *next = nsel > d ? best[d].v : -INFINITY;
    nsel = min(nsel, d);
  }
  write_sel(best, nsel, idx, val, count);
}

template <int kCs>
__device__ void peaks2d_block(const float *__restrict__ P, int La, int Le, bool wrap, int d, int *idx, float *val,
                              int *count) {
  __shared__ Cand sel[kMaxM], all[kCs > 1 ? kMaxM : 1];
  const Share<kCs, kPeakThreads> sh;
  int nsel = select_rounds(d, sel, [&](const Cand &thr, Cand (&cache)[kCache], int &n) {
    return fill2d(P, La, Le, wrap, sh.first, sh.stride, thr, cache, n);
  });
  Cand *best = sel;
  if (kCs > 1) {
    nsel = merge_lists<kCs>(d, sel, nsel, all);
    best = all;
    if (sh.rank != 0) return;
  }
  write_sel(best, nsel, idx, val, count);
}

template <int kCs>
__global__ void __launch_bounds__(kPeakThreads) peaks2d_single_kernel(const float *P, int La, int Le, int wrap, int d,
                                                                      int *idx, float *val, int *count) {
  start_after_previous();
  let_next_start();
  peaks2d_block<kCs>(P, La, Le, wrap != 0, d, idx, val, count);
}

template <int kCs>
__global__ void __launch_bounds__(kPeakThreads) peaks_single_kernel(const float *P, int L, int d, int *idx, float *val,
                                                                    int *count) {
  start_after_previous();
  let_next_start();
  peaks_block<kCs, kPeakThreads>(P, L, d, idx, val, count);
}

// Threads per SM of the 1-D batch kernel, and the threads of a job's CTA in a batch of spectra that are many
// but not long (kSmallPoints): the barriers of a job and the merge of its lists by one warp leave a CTA
// of 256 threads idle for a third of its time, while two warps per job wait little and 20 jobs per SM
// overlap. 4096 x 4 spectra of 18 001 points: 32 threads 0.246, 64 0.227, 128 0.243, 256 0.303 ms. A long
// spectrum keeps 256 threads, so that it does not outlast the batch.
// (2-D: 256 threads measured best, 0.22 against 0.28 ms with 64, and four quads per thread in 64
// registers, 0.18 ms against 0.21 with two in 48.)
constexpr int kBatchThreads = 1280;
constexpr int kSmallThreads = 64, kSmallPoints = 65536;

// One CTA (or cluster) per (problem, algorithm) job; the 1-D and 2-D rules run as separate kernels (each skips
// the other kind's jobs) so that each keeps its own register budget.
// repick: the pick after the peak polish, only for the jobs the polish marked (NaN next value).
template <int kCs, int T>
__global__ void __launch_bounds__(T, kBatchThreads / T) peaks_batch_kernel(const uint8_t *plan, uint8_t *ws, int repick) {
  start_after_previous();
  let_next_start();
  const int job = blockIdx.x / kCs;
  const PlanHeader *h = reinterpret_cast<const PlanHeader *>(plan);
  const PlanJob &jb = reinterpret_cast<const PlanJob *>(plan + h->off_job)[job];
  const PlanProblem &pp = reinterpret_cast<const PlanProblem *>(plan + h->off_prob)[jb.prob];
  if (pp.p.geom.pos) return;
  const int L = pp.npts, d = pp.p.d;
  const bool polish = (pp.p.flags & DOA_FLAG_POLISH_PEAKS) && h->next_val_off >= 0;
  float *next = polish ? reinterpret_cast<float *>(ws + h->next_val_off) + job : nullptr;
  if (repick) {
    if (!polish || !isnan(*next)) return;
    next = nullptr;
  }
  peaks_block<kCs, T>(pp.p.P + (size_t)jb.slot * L, L, d, pp.p.peak_idx + (size_t)jb.slot * d,
                   pp.p.peak_val + (size_t)jb.slot * d, pp.p.peak_count + jb.slot, next);
}

template <int kCs>
__global__ void __launch_bounds__(kPeakThreads, 4) peaks2d_batch_kernel(const uint8_t *plan) {
  start_after_previous();
  let_next_start();
  const PlanHeader *h = reinterpret_cast<const PlanHeader *>(plan);
  const PlanJob &jb = reinterpret_cast<const PlanJob *>(plan + h->off_job)[blockIdx.x / kCs];
  const PlanProblem &pp = reinterpret_cast<const PlanProblem *>(plan + h->off_prob)[jb.prob];
  if (!pp.p.geom.pos) return;
  const int L = pp.npts, d = pp.p.d;
  peaks2d_block<kCs>(pp.p.P + (size_t)jb.slot * L, pp.p.grid.L, pp.p.geom.Le, pp.p.geom.wrap_az != 0, d,
                pp.p.peak_idx + (size_t)jb.slot * d, pp.p.peak_val + (size_t)jb.slot * d, pp.p.peak_count + jb.slot);
}

// ---- grid slices ---------------------------------------------------------------------------
// Value at global index k of a slice buffer that starts at global index b0.
struct SliceView {
  const float *buf;
  int b0;
  __device__ float operator()(int k) const { return buf[k - b0]; }
};

// 0: not a peak, 1: decided peak, 2: run still equal at `limit` (< L - 1), undecided.
__device__ __forceinline__ int slice_peak_state(const SliceView &P, int i, float v, int limit, int L) {
  if (!(P(i - 1) < v)) return 0;
  int j = i;
  while (j + 1 <= limit && P(j + 1) == v) ++j;
  if (j + 1 <= limit) return P(j + 1) < v ? 1 : 0;
  return limit < L - 1 ? 2 : 0;
}

// Best decided peaks among the thread's points (i = c0, c0 + T, ... < c1) worse than thr.
__device__ bool slice_fill(const SliceView &P, int c0, int c1, int limit, int L, const Cand &thr,
                           Cand (&cache)[kCache], int &n, int *open_idx, float *open_val) {
  n = 0;
  bool more = false;
  for (int i = c0; i < c1; i += kPeakThreads) {
    const float v = P(i);
    const int st = slice_peak_state(P, i, v, limit, L);
    if (st == 2) {
      *open_idx = i;   // the unique run that reaches the end of the slice's data
      *open_val = v;
    }
    if (st != 1) continue;
    cache_insert(Cand{v, i}, thr, cache, n, more);
  }
  return more;
}

__global__ void __launch_bounds__(kPeakThreads) slice_peaks_kernel(const float *Pbuf, int b0, int k0, int k1, int L,
                                                                    int d, doa_slice_summary *out) {
  __shared__ Cand red[kPeakThreads / 32 + 1];
  __shared__ int s_open_idx;
  __shared__ float s_open_val;
  const SliceView P{Pbuf, b0};
  const int limit = min(k1 + 1, L) - 1;              // last readable global index
  const int c0 = max(k0, 1) + threadIdx.x, c1 = min(k1, L - 1);
  if (threadIdx.x == 0) s_open_idx = -1;
  __syncthreads();
  int oi = -1;
  float ov = 0.f;
  Cand cache[kCache];
  int n = 0, head = 0;
  const Cand none{0.f, INT_MAX};
  bool more = slice_fill(P, c0, c1, limit, L, none, cache, n, &oi, &ov);
  if (oi >= 0) {
    s_open_idx = oi;
    s_open_val = ov;
  }
  int nsel = 0;
  for (int r = 0; r < d; ++r) {
    Cand mine = head < n ? cache[head] : none;
    Cand w = block_best(mine, red);
    if (w.i == INT_MAX) break;
    if (threadIdx.x == 0) {
      out->idx[nsel] = w.i;
      out->val[nsel] = w.v;
    }
    ++nsel;
    if (mine.i == w.i) {
      ++head;
      if (head == n && more) {
        int dummy_i;
        float dummy_v;
        more = slice_fill(P, c0, c1, limit, L, w, cache, n, &dummy_i, &dummy_v);
        head = 0;
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    out->count = nsel;
    out->open_idx = s_open_idx;
    out->open_val = s_open_idx >= 0 ? s_open_val : 0.f;
    const float v0 = P(k0);
    int k = k0;
    while (k + 1 <= limit && P(k + 1) == v0) ++k;
    out->first_val = v0;
    out->first_run_to_end = k + 1 > limit ? 1 : 0;
    out->first_next_val = k + 1 <= limit ? P(k + 1) : 0.f;
  }
}

}  // namespace

cudaError_t launch_slice_peaks(const float *Pbuf, int b0, int k0, int k1, int L, int d, doa_slice_summary *out,
                               cudaStream_t s) {
  slice_peaks_kernel<<<1, kPeakThreads, 0, s>>>(Pbuf, b0, k0, k1, L, d, out);
  return cudaGetLastError();
}

// Launches `kernel` on `jobs` spectra, kCs CTAs each.
template <int kCs, int T, class... Args>
cudaError_t launch_jobs(void (*kernel)(Args...), int jobs, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)jobs * kCs);
  cfg.blockDim = dim3(T);
  cfg.stream = s;
  cudaLaunchAttribute attr[2] = {};
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = kCs;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  const bool chained = chained_grid((int64_t)jobs * kCs);
  cfg.attrs = chained ? attr : attr + 1;
  cfg.numAttrs = (chained ? 1 : 0) + (kCs > 1 ? 1 : 0);
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

cudaError_t launch_peaks_single(const float *P, int L, int d, int *idx, float *val, int *count, cudaStream_t s) {
  return L >= kClusterPoints ? launch_jobs<kPeakCluster, kPeakThreads>(peaks_single_kernel<kPeakCluster>, 1, s, P, L, d, idx, val, count)
                             : launch_jobs<1, kPeakThreads>(peaks_single_kernel<1>, 1, s, P, L, d, idx, val, count);
}

cudaError_t launch_peaks2d_single(const float *P, int La, int Le, int wrap_az, int d, int *idx, float *val,
                                  int *count, cudaStream_t s) {
  return (int64_t)La * Le >= kClusterPoints
             ? launch_jobs<kPeakCluster, kPeakThreads>(peaks2d_single_kernel<kPeakCluster>, 1, s, P, La, Le, wrap_az, d, idx, val, count)
             : launch_jobs<1, kPeakThreads>(peaks2d_single_kernel<1>, 1, s, P, La, Le, wrap_az, d, idx, val, count);
}

// A batch takes clusters when its jobs do not fill the SMs (five CTAs each) and some spectrum is long
// enough. For 1024 mixed jobs of up to 180 001 points clusters gain nothing (0.16 against 0.15 ms, 0.11
// of it the launching of 8192 clustered CTAs).
cudaError_t launch_peaks_batch(const uint8_t *plan_dev, const PlanHeader &h, uint8_t *ws, bool ula, bool geo,
                               cudaStream_t s) {
  int ngeo = 0;
  for (int b = 0; b < kNumBuckets; ++b) ngeo += h.geo_jobs[b];
  const int repick = ula && !geo;   // the call after the polish
  const bool few = (int64_t)h.njobs * kPeakCluster <= 5 * (int64_t)device_sm_count();
  const bool cl = few && h.max_points >= kClusterPoints;
  const bool small = h.max_points <= kSmallPoints &&
                     (int64_t)h.njobs * kSmallThreads >= kBatchThreads * (int64_t)device_sm_count();
  cudaError_t e = cudaSuccess;
  if (h.njobs > 0 && ula && ngeo < h.nprob)
    e = cl ? launch_jobs<kPeakCluster, kPeakThreads>(peaks_batch_kernel<kPeakCluster, kPeakThreads>, h.njobs, s, plan_dev, ws, repick)
        : small ? launch_jobs<1, kSmallThreads>(peaks_batch_kernel<1, kSmallThreads>, h.njobs, s, plan_dev, ws, repick)
                : launch_jobs<1, kPeakThreads>(peaks_batch_kernel<1, kPeakThreads>, h.njobs, s, plan_dev, ws, repick);
  if (e == cudaSuccess && h.njobs > 0 && geo && ngeo > 0)
    e = cl ? launch_jobs<kPeakCluster, kPeakThreads>(peaks2d_batch_kernel<kPeakCluster>, h.njobs, s, plan_dev)
           : launch_jobs<1, kPeakThreads>(peaks2d_batch_kernel<1>, h.njobs, s, plan_dev);
  return e;
}

}  // namespace doa
