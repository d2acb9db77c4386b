// Tensor-core kernels of the learned-proposal network (272 -> 256 -> 256 -> 256 -> 181).
//
// mlp_rows_kernel: persistent CTAs take 128 rows at a time through the whole network. A layer's input
// stays in shared memory as the BF16 K-major operand (128B swizzle), its weights are streamed by TMA
// through a ring of 64-wide K tiles, one thread issues the tcgen05 MMAs (128 x N x 16, FP32 accumulation
// in one of two TMEM buffers), and sixteen warps turn the accumulator into the next layer's operand
// (bias, ReLU, BF16). While the MMAs of a layer run, in a forward pass those warps fetch a quarter of the
// next tile's features into the second operand buffer. In training the same CTA goes on backward:
// dZ4 = (sigmoid(z) - y) / B, then dZ_l = (dZ_{l+1} W_{l+1}) [A_l > 0] with the ReLU masks kept in
// registers; every operand also leaves by a TMA store (row-major BF16, for the weight gradients), with
// partial sums of the bias gradients and the loss.
// mlp_dw_kernel: all four weight gradients dW_l = dZ_l^T A_{l-1} in one launch, a CTA per 128 x 64 tile
// over the whole batch; both operands are read batch-major, as they were stored (the MMA's MN-major
// form), so no transposed copies exist. Blocks beside them add the partial sums of the bias gradients and
// the loss in a fixed order.
//
// Why: one GEMM per launch moved every activation through memory twice, and its epilogue stored
// two-byte elements one at a time (180 us for a 65536 x 256 layer); a weight gradient ran on two CTAs.
// A tile's weights (0.5 MB a pass over the network) come from L2 through two 32 KB stages, which bounds a
// layer's MMAs (5300 cycles against 2050 of tensor work); the epilogue of a hidden layer takes 2300 cycles,
// that of the outputs 16000, half of it the burst of stores that all SMs make at once.
// Measured: forward of 65536 rows 0.740 -> 0.086 ms (167 MB read and written: 1.9 TB/s); a training step of
// 4096 rows 0.50 -> 0.077 ms (32 tiles on as many SMs: 50 us, half of it the loss; weight gradients 20 us).
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>

#include "doa_internal.cuh"
#include "mlp_tc.cuh"
#include "tc_common.cuh"

namespace doa {
namespace {

using namespace tc;

constexpr int kEpiWarps = 16;
constexpr int kEpiThreads = 32 * kEpiWarps;
constexpr int kRowsThreads = kEpiThreads + 64;          // + the TMA warp and the MMA warp
constexpr int kRing = 2;
constexpr int kRingBytes = 256 * 128;                   // 256 weight rows x 64 BF16
constexpr int kATile = kTcRows * 128;                   // 128 rows x 64 BF16
constexpr int kABytes = 5 * kATile;                     // up to 272 wide
constexpr int kRowsSmem = 2 * kABytes + kRing * kRingBytes + 1024;
constexpr int kStageBytes = 32 * 16 * 4;                // a warp's staging tile: 32 rows x 16 FP32 columns
static_assert(64 * DOA_MLP_OUT * 4 <= kABytes, "half a tile of outputs is staged in the operand buffer");
static_assert(3 * kATile + kEpiWarps * kStageBytes <= kABytes, "dZ4 and the staging tiles share an operand buffer");
constexpr int kChunks = kTcRows * (DOA_MLP_IN / 8);     // input steps of eight columns
constexpr int kFetch = (kChunks / 4 + kEpiThreads - 1) / kEpiThreads;   // a thread's steps in a quarter
static_assert(kEpiWarps == kMlpLossParts, "one loss partial per warp");
static_assert(kChunks % 4 == 0, "the input is fetched in quarters");

__device__ __forceinline__ void tma_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t mbar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(mbar)
      : "memory");
}
__device__ __forceinline__ void expect_tx(uint32_t mbar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}
__device__ __forceinline__ void commit(uint32_t mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar) : "memory");
}
// smem tile (box of the map) -> global, clipped to the tensor
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *map, int x, int y, uint32_t src) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(x), "r"(y), "r"(src)
               : "memory");
}
// 16 or 32 accumulator columns of this warp's 32 TMEM lanes
__device__ __forceinline__ void tmem_ld16(uint32_t addr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(addr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}
__device__ __forceinline__ void tmem_ld32(uint32_t addr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,"
      "%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(addr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}
__device__ __forceinline__ uint32_t pack2(float a, float b) {
  const __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t *>(&p);
}
// Sums of N columns over the warp's 32 rows (v[j]: this lane's value of column j); lanes j (mod N)
// receive column j's sum. A butterfly that halves the columns a lane keeps at each step.
template <int N>
__device__ __forceinline__ float column_sums(float (&v)[N]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int off = 16; off >= N; off >>= 1)
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] += __shfl_xor_sync(0xffffffffu, v[j], off);
#pragma unroll
  for (int off = N / 2; off > 0; off >>= 1) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int j = 0; j < off; ++j) {
      const float give = up ? v[j] : v[j + off], keep = up ? v[j + off] : v[j];
      v[j] = keep + __shfl_xor_sync(0xffffffffu, give, off);
    }
  }
  return v[0];
}

// Barrier 1 of the epilogue warps: true if p holds in all of their threads (a wait that ran out ends their loop
// over the tiles for all of them or for none, since they meet at barriers in it).
__device__ __forceinline__ bool all_ok(bool p) {
  uint32_t r;
  asm volatile("{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbarrier.cta.red.and.pred q, 1, %2, p;\nselp.b32 %0, 1, 0, q;\n}\n"
               : "=r"(r)
               : "r"((uint32_t)p), "r"(kEpiThreads)
               : "memory");
  return r != 0;
}

// One layer pass of the row kernel: its weights' tensor map, MMA N and K steps of 16.
struct RowPass {
  int map, n, k16;
};
__device__ __forceinline__ RowPass row_pass(int p) {
  switch (p) {
    case 0: return {0, 256, 17};    // K = 272
    case 1: return {1, 256, 16};
    case 2: return {2, 256, 16};
    case 3: return {3, 192, 16};    // 181 outputs
    case 4: return {4, 256, 12};    // dZ4 W4, K = 181 (zero-filled)
    case 5: return {5, 256, 16};    // dZ3 W3
    default: return {6, 256, 16};   // dZ2 W2
  }
}

template <bool kTrain>
__global__ void __launch_bounds__(kRowsThreads, 1) mlp_rows_kernel(const __grid_constant__ MlpMaps maps,
                                                                   const __grid_constant__ MlpRowArgs g) {
  start_after_previous();
  let_next_start();
  constexpr int kPasses = kTrain ? 7 : 4;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t *sm = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t *ring = sm + 2 * kABytes;
  __shared__ __align__(8) uint64_t full_bar[kRing], empty_bar[kRing], a_bar, acc_bar;
  __shared__ uint32_t tmem_base;
  __shared__ int s_fail, s_issued, s_consumed;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tiles = (g.B + kTcRows - 1) / kTcRows;
  if (tid == 0) {
    for (int s = 0; s < kRing; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    mbar_init(&a_bar, kEpiThreads);
    mbar_init(&acc_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_fail = s_issued = s_consumed = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;

  if (warp == kEpiWarps) {
    if (lane == 0) {   // weights, K tile by K tile of every pass
      int t = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x)
        for (int p = 0; p < kPasses && ok; ++p) {
          const RowPass rp = row_pass(p);
          for (int kt = 0; kt * 4 < rp.k16; ++kt, ++t) {
            const int s = t % kRing;
            ok = t < kRing || mbar_wait(smem_u32(&empty_bar[s]), (uint32_t)((t / kRing - 1) & 1));
            if (!ok) {
              s_fail = 1;
              break;
            }
            expect_tx(smem_u32(&full_bar[s]), (uint32_t)(rp.n * 128));
            tma_2d(smem_u32(ring + s * kRingBytes), &maps.m[rp.map], kt * 64, 0, smem_u32(&full_bar[s]));
            s_issued = t + 1;
          }
        }
    }
  } else if (warp == kEpiWarps + 1) {
    if (lane == 0) {   // MMAs, and in training the stores of their operands
      int t = 0, n = 0;   // K tiles and passes so far
      bool ok = true;
      uint8_t *abuf = sm;
      for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
        for (int p = 0; p < kPasses && ok; ++p, ++n) {
          const RowPass rp = row_pass(p);
          const uint32_t idesc = inst_desc(1, rp.n), acc = tmem + (uint32_t)((n & 1) * 256);
          // the operand is written, and this TMEM buffer was read out a pass ago
          ok = mbar_wait(smem_u32(&a_bar), (uint32_t)((n + (kTrain ? tile / gridDim.x : 0)) & 1));
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          if (kTrain && ok) {
            for (int kt = 0; kt * 4 < rp.k16; ++kt)
              tma_store_2d(&maps.store[p], kt * 64, tile * kTcRows, smem_u32(abuf + kt * kATile));
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
          }
          for (int kt = 0; ok && kt * 4 < rp.k16; ++kt, ++t) {
            const int s = t % kRing;
            ok = mbar_wait(smem_u32(&full_bar[s]), (uint32_t)((t / kRing) & 1));
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t pa = smem_u32(abuf + kt * kATile), pb = smem_u32(ring + s * kRingBytes);
            for (int kk = 0; kk < 4 && kt * 4 + kk < rp.k16; ++kk)
              mma(acc, smem_desc(pa + kk * 32), smem_desc(pb + kk * 32), idesc, (kt > 0 || kk > 0) ? 1u : 0u);
            commit(smem_u32(&empty_bar[s]));
            s_consumed = t + 1;
          }
          // the operand may be overwritten once the MMAs and the store have read it
          if (kTrain) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
          commit(smem_u32(&acc_bar));
        }
        if (kTrain && ok) {   // dZ_1 has no MMA of this tile's chain: store it
          ok = mbar_wait(smem_u32(&a_bar), (uint32_t)((n + tile / gridDim.x) & 1));
          for (int kt = 0; kt < 4 && ok; ++kt)
            tma_store_2d(&maps.store[7], kt * 64, tile * kTcRows, smem_u32(abuf + kt * kATile));
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
          asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
          mbar_arrive(smem_u32(&acc_bar));
        }
        abuf = abuf == sm ? sm + kABytes : sm;
      }
      if (!ok) s_fail = 1;
      if (kTrain) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
  } else {
    const int q = warp & 3, h = warp >> 2;          // TMEM lanes 32 q .., column quarter h
    const int rl = q * 32 + lane;                   // this thread's row of the tile
    const uint32_t tl = tmem + ((uint32_t)(q * 32) << 16);
    uint8_t *abuf = sm;
    int n = 0, na = 0;                              // passes so far, waits on acc_bar
    bool ok = true;
    // input steps: FP32 features -> BF16 operand, eight columns each; quarter by quarter
    auto fetch = [&](int tile, int quarter, int k, float4 &a, float4 &b) {
      const int e = quarter * (kChunks / 4) + k * kEpiThreads + tid;
      const int i = e / (DOA_MLP_IN / 8), c = (e - i * (DOA_MLP_IN / 8)) * 8, r = tile * kTcRows + i;
      a = b = make_float4(0.f, 0.f, 0.f, 0.f);
      if (k * kEpiThreads + tid >= kChunks / 4 || r >= g.B) return;
      const float *x = g.X + (size_t)r * DOA_MLP_IN + c;
      if (g.x_vec) {
        a = __ldcs(reinterpret_cast<const float4 *>(x));
        b = __ldcs(reinterpret_cast<const float4 *>(x) + 1);
      } else {
        a = make_float4(x[0], x[1], x[2], x[3]);
        b = make_float4(x[4], x[5], x[6], x[7]);
      }
    };
    auto place = [&](uint8_t *buf, int quarter, int k, const float4 &a, const float4 &b) {
      const int e = quarter * (kChunks / 4) + k * kEpiThreads + tid;
      const int i = e / (DOA_MLP_IN / 8), c = (e - i * (DOA_MLP_IN / 8)) * 8;
      if (k * kEpiThreads + tid >= kChunks / 4) return;
      *reinterpret_cast<uint4 *>(buf + (c >> 6) * kATile + sw128(i, c & 63)) =
          make_uint4(pack2(a.x, a.y), pack2(a.z, a.w), pack2(b.x, b.y), pack2(b.z, b.w));
    };
    auto publish = [&]() {   // the operand (generic proxy) and the TMEM reads, before the next MMAs
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      mbar_arrive(smem_u32(&a_bar));
    };
    auto wait_acc = [&]() {
      ok = __all_sync(0xffffffffu, ok && mbar_wait(smem_u32(&acc_bar), (uint32_t)(na & 1)));
      ++na;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    };
    auto put8 = [&](const float *v, int c) {   // eight columns of this thread's row into the operand
      *reinterpret_cast<uint4 *>(abuf + (c >> 6) * kATile + sw128(rl, c & 63)) =
          make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
    };
    auto load = [&](int tile, uint8_t *buf) {
#pragma unroll
      for (int quarter = 0; quarter < 4; ++quarter) {
        float4 fa[kFetch], fb[kFetch];
#pragma unroll
        for (int k = 0; k < kFetch; ++k) fetch(tile, quarter, k, fa[k], fb[k]);
#pragma unroll
        for (int k = 0; k < kFetch; ++k) place(buf, quarter, k, fa[k], fb[k]);
      }
      publish();
    };
    if (blockIdx.x < tiles) load(blockIdx.x, abuf);
    for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
      const int row = tile * kTcRows + rl;
      const bool live = row < g.B;
      const int next = tile + gridDim.x;
      uint8_t *nbuf = abuf == sm ? sm + kABytes : sm;
      // waits for the MMAs of pass p, with a quarter of the next tile's input fetched meanwhile
      auto wait_fetch = [&](int quarter) {
        float4 fa[kFetch], fb[kFetch];
        if (!kTrain && next < tiles) {
#pragma unroll
          for (int k = 0; k < kFetch; ++k) fetch(next, quarter, k, fa[k], fb[k]);
        }
        wait_acc();
        if (!kTrain && next < tiles) {
#pragma unroll
          for (int k = 0; k < kFetch; ++k) place(nbuf, quarter, k, fa[k], fb[k]);
        }
      };
      uint32_t relu[3][2];   // [A_l > 0] of this thread's row and columns
      // hidden layers
#pragma unroll
      for (int p = 0; p < 3; ++p, ++n) {
        wait_fetch(p);
        const uint32_t acc = tl + (uint32_t)((n & 1) * 256);
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
          const int c0 = h * 64 + cc * 32;
          float v[32];
          tmem_ld32(acc + (uint32_t)c0, v);
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = fmaxf(v[j] + __ldg(g.bias[p] + c0 + j), 0.f);
#pragma unroll
          for (int j = 0; j < 32; j += 8) put8(v + j, c0 + j);
          if (kTrain) {   // the mask of the BF16 activations: a value rounds to zero up to 2^-134
            uint32_t m = 0u;
#pragma unroll
            for (int j = 0; j < 32; ++j) m |= (v[j] > 4.5917748e-41f ? 1u : 0u) << j;   // 2^-134
            relu[p][cc] = m;
          }
        }
        publish();
      }
      // output layer
      wait_fetch(3);
      const uint32_t acc4 = tl + (uint32_t)((n & 1) * 256);
      ++n;
      float *stage = reinterpret_cast<float *>(abuf + 3 * kATile + warp * kStageBytes);   // 32 rows x 16, swizzled
      auto at = [&](int r, int c) { return r * 16 + (c ^ ((r >> 1) & 15)); };
      if constexpr (!kTrain) {
        if (next < tiles) publish();   // the next tile's first MMAs run beside this epilogue
        // z + bias through shared memory, 64 rows at a time, and out in the tile's memory order
        float *Z = reinterpret_cast<float *>(abuf);
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
          if ((q >> 1) == half) {
            float *z = Z + (rl & 63) * DOA_MLP_OUT;
#pragma unroll 1
            for (int cc = 0; cc < 3; ++cc) {
              const int c0 = h * 48 + cc * 16;
              float v[16];
              tmem_ld16(acc4 + (uint32_t)c0, v);
#pragma unroll
              for (int j = 0; j < 16; ++j)
                if (c0 + j < DOA_MLP_OUT) z[c0 + j] = v[j] + __ldg(g.bias[3] + c0 + j);
            }
          }
          asm volatile("bar.sync 1, %0;" ::"r"(kEpiThreads) : "memory");
          const int r0 = tile * kTcRows + half * 64, cnt = max(0, min(64, g.B - r0)) * DOA_MLP_OUT;
          const size_t o0 = (size_t)r0 * DOA_MLP_OUT;
          if (g.out_vec) {      // rows come in eights: cnt is a multiple of four
            for (int e = tid * 4; e < cnt; e += kEpiThreads * 4) {
              const float4 x = *reinterpret_cast<const float4 *>(Z + e);
              if (g.logits) __stcs(reinterpret_cast<float4 *>(g.logits + o0 + e), x);
              if (g.probs)
                __stcs(reinterpret_cast<float4 *>(g.probs + o0 + e),
                       make_float4(1.f / (1.f + __expf(-x.x)), 1.f / (1.f + __expf(-x.y)), 1.f / (1.f + __expf(-x.z)),
                                   1.f / (1.f + __expf(-x.w))));
            }
          } else {
            for (int e = tid; e < cnt; e += kEpiThreads) {
              const float x = Z[e];
              if (g.logits) g.logits[o0 + e] = x;
              if (g.probs) g.probs[o0 + e] = 1.f / (1.f + __expf(-x));
            }
          }
          // the staged rows are read before they (or the buffer's next input) are written again
          ok = all_ok(ok);
        }
      } else {
        const float invB = 1.f / (float)g.B;
        float *gbp = g.gb_part + (size_t)(tile * 4 + q) * kMlpGbCols;
        float loss = 0.f;
#pragma unroll 1
        for (int cc = 0; cc < 3; ++cc) {
          const int c0 = h * 48 + cc * 16, c = c0 + (lane & 15);
          float y[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const int r = tile * kTcRows + q * 32 + 2 * i + (lane >> 4);
            y[i] = (r < g.B && c < DOA_MLP_OUT) ? __ldcs(g.Y + (size_t)r * DOA_MLP_OUT + c) : 0.f;
          }
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 16; ++i) stage[at(2 * i + (lane >> 4), lane & 15)] = y[i];
          __syncwarp();
          float v[16];
          tmem_ld16(acc4 + (uint32_t)c0, v);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            float d = 0.f;
            if (live && c0 + j < DOA_MLP_OUT) {
              const float z = v[j] + __ldg(g.bias[3] + c0 + j), lab = stage[at(lane, j)];
              const float sg = 1.f / (1.f + __expf(-z));
              d = (sg - lab) * invB;
              loss += (fmaxf(z, 0.f) - lab * z + log1pf(__expf(-fabsf(z)))) * invB;
            }
            v[j] = d;
          }
          put8(v, c0);
          put8(v + 8, c0 + 8);
          const float sum = column_sums(v);
          if (lane < 16) gbp[3 * DOA_MLP_HIDDEN + c0 + lane] = sum;
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, off);
        if (lane == 0) g.loss_part[tile * kEpiWarps + warp] = loss;
        publish();
        // back through the hidden layers
#pragma unroll
        for (int l = 2; l >= 0; --l, ++n) {
          wait_acc();
          const uint32_t acc = tl + (uint32_t)((n & 1) * 256);
#pragma unroll
          for (int cc = 0; cc < 2; ++cc) {
            const int c0 = h * 64 + cc * 32;
            float v[32];
            tmem_ld32(acc + (uint32_t)c0, v);
            const uint32_t m = live ? relu[l][cc] : 0u;
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = (m >> j) & 1u ? v[j] : 0.f;
#pragma unroll
            for (int j = 0; j < 32; j += 8) put8(v + j, c0 + j);
            gbp[l * DOA_MLP_HIDDEN + c0 + lane] = column_sums(v);
          }
          publish();
        }
        wait_acc();                          // dZ_1 is stored
        if (next < tiles) {
          load(next, nbuf);
          ok = all_ok(ok);
        }
      }
      abuf = nbuf;
    }
    if (!ok) s_fail = 1;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (s_fail && tid == 0) {
    if (g.err) atomicExch(g.err, 1);
    // let the copies still in flight land before the CTA exits (bounded waits)
    for (int t = s_consumed; t < s_issued; ++t) mbar_wait(smem_u32(&full_bar[t % kRing]), (uint32_t)((t / kRing) & 1));
  }
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// ---- weight gradients -----------------------------------------------------------------------------
constexpr int kDwStages = 8;   // the loads in flight bound a tile: 192 KB a CTA
constexpr int kDwStage = kATile + 64 * 128;
constexpr int kDwSmem = kDwStages * kDwStage + 1024;
constexpr int kDwThreads = 256;
constexpr int kDwBox = 64 * 128;   // 64 batch rows x 64 features

// MN-major forms of the descriptors: features contiguous in 128-byte swizzled rows, one row per batch
// index; groups of 8 rows 1024 bytes apart, the next 64 features kDwBox bytes apart.
__device__ __forceinline__ uint64_t mn_desc(uint32_t addr) {
  uint64_t d = (uint64_t)((addr >> 4) & 0x3FFF);
  d |= (uint64_t)(kDwBox >> 4) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
constexpr uint32_t kMnMajor = (1u << 15) | (1u << 16);   // both operands

// Output tiles: 128 rows x 64 columns of dW_l (layer 0's last: 16 columns).
struct DwTile {
  int layer, m0, n0, bn;
};
__host__ __device__ inline DwTile dw_tile(int i) {
  if (i < 10) return {0, (i & 1) * 128, (i >> 1) * 64, i < 8 ? 64 : 16};
  i -= 10;
  return {1 + (i >> 3), (i & 1) * 128, ((i & 7) >> 1) * 64, 64};
}
static_assert(kMlpDwTiles == 10 + 3 * 8, "tiles of the four layers");

// Adds the partial sums of 32 bias gradients (block b of kMlpGbCols / 32), or of the loss (the block after).
__device__ void add_partials(int b, int tiles, const float *gb_part, const float *loss_part, const MlpGrads &o) {
  __shared__ float red[8][33];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  float a = 0.f;
  if (b < kMlpGbCols / 32) {
    const int col = b * 32 + lane;
    for (int r = w; r < tiles * 4; r += 8) a += gb_part[(size_t)r * kMlpGbCols + col];
  } else {
    for (int r = tid; r < tiles * kEpiWarps; r += 256) a += loss_part[r];
  }
  red[w][lane] = a;
  __syncthreads();
  if (w == 0) {
    a = red[0][lane];
    for (int k = 1; k < 8; ++k) a += red[k][lane];
    if (b < kMlpGbCols / 32) {
      const int col = b * 32 + lane, layer = min(col / DOA_MLP_HIDDEN, 3), c = col - layer * DOA_MLP_HIDDEN;
      if (c < (layer == 3 ? DOA_MLP_OUT : DOA_MLP_HIDDEN)) o.gb[layer][c] = a;
    } else {
      for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
      if (lane == 0 && o.loss) *o.loss = a;
    }
  }
}

// A tile's batch is not split over CTAs. The tensor cores' FP32 accumulation truncates, so split sums differ
// from the whole sum by 9e-6 of the norm (4096 rows), and one Adam step later a BF16 weight or a ReLU mask
// may fall the other way (1.9e-4). The whole sum in the order it always had costs 7 us a step.
__global__ void __launch_bounds__(kDwThreads) mlp_dw_kernel(const __grid_constant__ MlpDwMaps maps,
                                                               const __grid_constant__ MlpGrads o, int B, int tiles,
                                                               const float *gb_part, const float *loss_part, int *err) {
  start_after_previous();
  let_next_start();
  if (blockIdx.x >= kMlpDwTiles) {
    add_partials(blockIdx.x - kMlpDwTiles, tiles, gb_part, loss_part, o);
    return;
  }
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t *sm = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t full_bar[kDwStages], empty_bar[kDwStages], done_bar;
  __shared__ uint32_t tmem_base;
  __shared__ int s_fail, s_issued, s_consumed;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const DwTile tl = dw_tile(blockIdx.x);
  const int nk = (B + 63) / 64;
  if (tid == 0) {
    for (int s = 0; s < kDwStages; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    mbar_init(&done_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_fail = s_issued = s_consumed = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                 "r"(64));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;
  if (warp == 0 && lane == 0) {
    for (int t = 0; t < nk; ++t) {
      const int s = t % kDwStages;
      if (t >= kDwStages && !mbar_wait(smem_u32(&empty_bar[s]), (uint32_t)((t / kDwStages - 1) & 1))) {
        s_fail = 1;
        break;
      }
      uint8_t *st = sm + s * kDwStage;
      expect_tx(smem_u32(&full_bar[s]), (uint32_t)(3 * kDwBox));
      for (int i = 0; i < 2; ++i)
        tma_2d(smem_u32(st + i * kDwBox), &maps.a[tl.layer], tl.m0 + i * 64, t * 64, smem_u32(&full_bar[s]));
      tma_2d(smem_u32(st + 2 * kDwBox), &maps.b[tl.layer], tl.n0, t * 64, smem_u32(&full_bar[s]));
      s_issued = t + 1;
    }
  } else if (warp == 1 && lane == 0) {
    const uint32_t idesc = inst_desc(1, tl.bn) | kMnMajor;
    for (int t = 0; t < nk; ++t) {
      const int s = t % kDwStages;
      if (!mbar_wait(smem_u32(&full_bar[s]), (uint32_t)((t / kDwStages) & 1))) {
        s_fail = 1;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t pa = smem_u32(sm + s * kDwStage), pb = pa + 2 * kDwBox;
      for (int kk = 0; kk < 4; ++kk)   // 16 batch rows: two groups of 8
        mma(tmem, mn_desc(pa + kk * 2048), mn_desc(pb + kk * 2048), idesc, (t > 0 || kk > 0) ? 1u : 0u);
      commit(smem_u32(&empty_bar[s]));
      s_consumed = t + 1;
    }
    commit(smem_u32(&done_bar));
  }
  __syncwarp();
  bool ok = mbar_wait(smem_u32(&done_bar), 0u);
  ok = __syncthreads_and(ok && !s_fail) != 0;
  if (!ok && tid == 0) {
    if (err) atomicExch(err, 1);
    for (int t = s_consumed; t < s_issued; ++t)
      mbar_wait(smem_u32(&full_bar[t % kDwStages]), (uint32_t)((t / kDwStages) & 1));
  }
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  // the tile through shared memory (every copy has landed and every MMA has read), rows out coalesced
  float *stage = reinterpret_cast<float *>(sm);
  constexpr int kPitch = 65;
  const int q = warp & 3, rl = q * 32 + lane, c0 = (warp >> 2) * 32;
  if (c0 < tl.bn && ok) {
    float v[32];
    tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c0, v);
#pragma unroll
    for (int j = 0; j < 32; ++j) stage[rl * kPitch + c0 + j] = v[j];
  }
  __syncthreads();
  const int out = tl.layer == 3 ? DOA_MLP_OUT : DOA_MLP_HIDDEN, in = tl.layer == 0 ? DOA_MLP_IN : DOA_MLP_HIDDEN;
  for (int r = warp; r < kTcRows && tl.m0 + r < out && ok; r += kDwThreads / 32) {
    float *d = o.gW[tl.layer] + (size_t)(tl.m0 + r) * in + tl.n0;
    for (int cidx = lane; cidx < tl.bn; cidx += 32) d[cidx] = stage[r * kPitch + cidx];
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(64));
}

PFN_cuTensorMapEncodeTiled_v12000 encoder() {
  static const PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
    cudaDriverEntryPointQueryResult q;
    void *f = nullptr;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q);
    return e == cudaSuccess && q == cudaDriverEntryPointSuccess ? reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f)
                                                                : nullptr;
  }();
  return fn;
}

// rows x cols BF16 (row pitch ld), boxes of box_rows x 64, 128B swizzle, zero fill outside
cudaError_t encode_bf16(CUtensorMap *map, const void *base, int rows, int cols, int ld, int box_rows) {
  const PFN_cuTensorMapEncodeTiled_v12000 fn = encoder();
  if (!fn) return cudaErrorNotSupported;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

constexpr int kNetDims[5] = {DOA_MLP_IN, DOA_MLP_HIDDEN, DOA_MLP_HIDDEN, DOA_MLP_HIDDEN, DOA_MLP_OUT};

}  // namespace

cudaError_t launch_mlp_rows(const doa_mlp *net, const MlpRowArgs &g, bool train, cudaStream_t s) {
  MlpMaps maps;
  cudaError_t e;
  for (int l = 0; l < 4; ++l)
    if ((e = encode_bf16(&maps.m[l], net->Wh[l], kNetDims[l + 1], kNetDims[l], kNetDims[l], l == 3 ? 192 : 256)) !=
        cudaSuccess)
      return e;
  for (int l = 3; l >= 1 && train; --l) {   // W_l^T: in rows, K = out
    const int out = kNetDims[l + 1];
    if ((e = encode_bf16(&maps.m[4 + 3 - l], net->WhT[l], kNetDims[l], out, (out + 7) / 8 * 8, 256)) != cudaSuccess)
      return e;
  }
  for (int p = 0; p < 8 && train; ++p) {    // the passes' operands, boxes of 128 rows x 64
    const __nv_bfloat16 *base = p == 0 ? g.X0 : (p < 4 ? g.A[p - 1] : g.dZ[7 - p]);
    const int cols = p == 0 ? DOA_MLP_IN : (p == 4 ? kMlpOutPitch : DOA_MLP_HIDDEN);
    if ((e = encode_bf16(&maps.store[p], base, g.B, cols, cols, kTcRows)) != cudaSuccess) return e;
  }
  const void *k = train ? (const void *)mlp_rows_kernel<true> : (const void *)mlp_rows_kernel<false>;
  if ((e = ensure_smem_attr(k, kRowsSmem)) != cudaSuccess) return e;
  const int tiles = (g.B + kTcRows - 1) / kTcRows, ctas = std::min(tiles, device_sm_count());
  return train ? launch_chained(mlp_rows_kernel<true>, ctas, kRowsThreads, kRowsSmem, s, maps, g)
               : launch_chained(mlp_rows_kernel<false>, ctas, kRowsThreads, kRowsSmem, s, maps, g);
}

cudaError_t launch_mlp_dw(const MlpRowArgs &g, const MlpGrads &o, cudaStream_t s) {
  MlpDwMaps maps;
  cudaError_t e;
  for (int l = 0; l < 4; ++l) {   // boxes of 64 batch rows x 64 features
    const int out = l == 3 ? kMlpOutPitch : DOA_MLP_HIDDEN, in = l == 0 ? DOA_MLP_IN : DOA_MLP_HIDDEN;
    if ((e = encode_bf16(&maps.a[l], g.dZ[l], g.B, out, out, 64)) != cudaSuccess) return e;
    if ((e = encode_bf16(&maps.b[l], l == 0 ? g.X0 : g.A[l - 1], g.B, in, in, 64)) != cudaSuccess) return e;
  }
  if ((e = ensure_smem_attr((const void *)mlp_dw_kernel, kDwSmem)) != cudaSuccess) return e;
  const int tiles = (g.B + kTcRows - 1) / kTcRows;
  // the step's kernels and Adam queue behind each other (5 us of a step of 4096 rows)
  return launch_chained(mlp_dw_kernel, kMlpDwTiles + kMlpGbCols / 32 + 1, kDwThreads, kDwSmem, s, maps, o, g.B, tiles,
                        g.gb_part, g.loss_part, g.err);
}

}  // namespace doa
