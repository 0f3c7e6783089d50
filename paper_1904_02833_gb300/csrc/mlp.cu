// Warm-start network on the 5th-generation tensor cores: 24 features -> 128 -> 128 -> 1
// with SiLU, BF16 operands, FP32 accumulation in tensor memory.
//
// Inference (mlp_infer_kernel) and training (mlp_train_kernel: forward, MSE loss,
// backward, weight-gradient accumulation across tiles in tensor memory) process tiles
// of 128 constraint rows.  Every GEMM is one or more tcgen05.mma of M = 128 issued by one
// thread; operands are staged in shared memory in the canonical no-swizzle K-major
// layout (tc.cuh), and the products that need an operand transposed read the same tile
// MN-major.  The blocks' partial gradients are added, and Adam runs on FP32 master
// weights and refreshes the BF16 copies the GEMMs read, in mlp_reduce_kernel.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "internal.h"
#include "snakesim.h"
#include "tc.cuh"

using namespace snakesim;

namespace {

constexpr int kIn = 24;      // features
constexpr int kInPad = 32;   // K of the first GEMM (two K = 16 steps)
constexpr int kHid = 128;
constexpr int kTile = 128;   // rows per tile (M of every MMA)
constexpr uint32_t kWaitLimit = 1u << 26;

// parameter vector (FP32): W1 [128][24], b1 [128], W2 [128][128], b2 [128], w3 [128], b3
constexpr int kOffW1 = 0;
constexpr int kOffB1 = kOffW1 + kHid * kIn;
constexpr int kOffW2 = kOffB1 + kHid;
constexpr int kOffB2 = kOffW2 + kHid * kHid;
constexpr int kOffW3 = kOffB2 + kHid;
constexpr int kOffB3 = kOffW3 + kHid;
constexpr int kNumParams = kOffB3 + 1;  // 19841
static_assert(kNumParams == MLP_NUM_PARAMS, "parameter count");

// After a timed-out wait on an MMA: thread 0, the only thread that issues MMAs, commits
// once more to a barrier of its own, which arrives only when every MMA the thread issued
// before has completed (tcgen05.commit tracks all of the issuing thread's earlier
// tensor-core operations, not one group), and the block waits for that arrival before
// its TMEM columns are freed.  Like every wait it is bounded: an MMA completes in
// microseconds, so a drain that runs out means no completion will ever arrive (the
// columns are not being written) and the block still frees them, which it must do
// before it exits.
__device__ __forceinline__ void drain_mma(uint64_t* drain, int t) {
  if (t == 0) tc::mma_commit(drain);
  tc::mbar_wait(drain, 0, kWaitLimit);
}

struct MlpDev {
  const __nv_bfloat16* w1;  // [128][32] row-major (out x in, zero-padded in 24..31)
  const __nv_bfloat16* w2;  // [128][128] (out x in)
  const float* b1;
  const float* b2;
  const float* w3;
  const float* b3;
};

__device__ __forceinline__ float tanh_approx(float x) {
  float t;
  asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(x));
  return t;
}
__device__ __forceinline__ float sigmoid(float z) { return fmaf(0.5f, tanh_approx(0.5f * z), 0.5f); }
__device__ __forceinline__ float silu(float z) { return z * sigmoid(z); }
__device__ __forceinline__ float silu_grad(float z) {
  const float s = sigmoid(z);
  return s * (1.f + z * (1.f - s));
}

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}
// silu of two values z = 2 hz, evaluated in bfloat16 pairs (the result feeds a bfloat16
// operand anyway): silu(z) = hz + hz tanh(hz), one packed tanh for two values.
__device__ __forceinline__ uint32_t silu_half_bf16x2(float hz0, float hz1) {
  const uint32_t hz = pack_bf16x2(hz0, hz1);
  uint32_t th, r;
  asm("tanh.approx.bf16x2 %0, %1;" : "=r"(th) : "r"(hz));
  asm("fma.rn.bf16x2 %0, %1, %2, %1;" : "=r"(r) : "r"(hz), "r"(th));
  return r;
}
__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d)
               : "memory");
}

// Copies a row-major bf16 matrix [rows][K] into the canonical K-major smem layout.
__device__ void stage_kmajor(uint8_t* dst, const __nv_bfloat16* src, int rows, int K) {
  const int chunks = rows * (K / 8);
  const uint32_t base = tc::smem_u32(dst);
  for (int c = threadIdx.x; c < chunks; c += blockDim.x) {
    const int m = c / (K / 8), kc = (c % (K / 8)) * 8;
    const uint4 v = *reinterpret_cast<const uint4*>(src + (size_t)m * K + kc);
    st_shared_v4(base + tc::kmajor_off(m, kc, K), v.x, v.y, v.z, v.w);
  }
}
struct InferSmem {
  uint8_t w1[kHid * kInPad * 2];
  uint8_t w2[kHid * kHid * 2];
  uint8_t h[2][kTile * kHid * 2];  // per group: X of the tile (first 8 KB), then H
  alignas(16) float hb1[kHid], hb2[kHid], w3[kHid];  // hb: half the bias
  uint64_t mbar[2];
  uint64_t drain[2];  // drain_mma: arrives once every MMA issued so far has completed
  uint32_t tmem;
};
constexpr int kInferThreads = 256;

}  // namespace

// The rows the network runs on, in the solver's six-rows-per-node order: sel = 0 all rows;
// sel = 1 the stretch, yaw and pitch rows (row r is row 6 (r / 3) + r % 3 of feat and out);
// sel = 2 the stretch rows (row r is row 6 r).
__device__ __forceinline__ long long infer_row(long long r, int sel) {
  return sel == 1 ? 6 * (r / 3) + r % 3 : (sel == 2 ? 6 * r : r);
}
// Barrier of one 128-thread group (hardware barrier 1 + group); the _or form returns whether
// any of its threads passed true.
__device__ __forceinline__ void group_sync(int group) {
  asm volatile("bar.sync %0, 128;\n" ::"r"(1 + group) : "memory");
}
__device__ __forceinline__ bool group_or(int group, bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\t"
      "bar.red.or.pred p, %2, 128, q;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(r)
      : "r"((uint32_t)v), "r"(1 + group)
      : "memory");
  return r != 0;
}

// y[r] = w3 . silu(W2 silu(W1 x_r + b1) + b2) + b3 for feat [rows][32] bf16.
// Two groups of four warps per block, two blocks per SM, every group with a tile of its own
// and a thread per row: the MMA waits and barriers of one group are covered by the epilogues
// of the other three.  A group needs one 128-column accumulator (Z2 replaces Z1 once the
// first epilogue has read it) and one 32 KB tile (H replaces X), which is what lets four
// groups share an SM with two copies of the weights; its next features are loaded into
// registers while it works.  The epilogues carry half of z: silu(z) = hz + hz tanh(hz) with
// hz = z / 2 = fma(0.5, acc, b / 2), two columns per packed FP32 instruction, so that a SiLU
// costs two to four instructions beside its tanh.
// What bounds it: the tanh unit (192 evaluations per row keep it busy 60 % of the kernel) and
// the queue in front of it; the epilogues' issue slots are 1215 thread instructions per row
// (1827 before); DRAM moves 68 bytes per row, a quarter of the time.  Measured, a call on
// 1,261,356 rows: 146 us with one tile per eight-warp block and two threads per row, 135 us
// now; outputs bit for bit the same.  Kernel alone (us before / now): 128 rows 8.9 / 9.0, 16384
// 8.9 / 9.0, 38912 (a tile per block) 11.1 / 11.2, 77952 16.4 / 14.9, 400000 43.5 / 41.2.
__global__ void __launch_bounds__(kInferThreads, 2) mlp_infer_kernel(const __nv_bfloat16* __restrict__ feat,
                                                                    long long rows, MlpDev w,
                                                                    float* __restrict__ out, int* err,
                                                                    int sel) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  InferSmem& S = *reinterpret_cast<InferSmem*>(smem_raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, group = warp >> 2, t = threadIdx.x & 127;
  const long long ntiles = (rows + kTile - 1) / kTile;
  // a tile is 128 rows x 4 chunks of 16 bytes: chunks t, t + 128, t + 256 and t + 384
  auto load_tile = [&](long long tile, uint4 (&v)[4]) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int c = t + u * 128;
      const long long r = tile * kTile + (c >> 2);
      v[u] = make_uint4(0u, 0u, 0u, 0u);
      if (tile < ntiles && r < rows) v[u] = reinterpret_cast<const uint4*>(feat + infer_row(r, sel) * kInPad)[c & 3];
    }
  };
  // tiles go to the blocks first, then to their second groups
  const long long stride = 2LL * gridDim.x;
  uint4 nxt[4];
  load_tile((long long)group * gridDim.x + blockIdx.x, nxt);
  if (warp == 0) tc::tmem_alloc(&S.tmem, 256);
  if (t == 0) { tc::mbar_init(&S.mbar[group], 1); tc::mbar_init(&S.drain[group], 1); }
  stage_kmajor(S.w1, w.w1, kHid, kInPad);
  stage_kmajor(S.w2, w.w2, kHid, kHid);
  if (threadIdx.x < kHid) {
    S.hb1[t] = 0.5f * w.b1[t];
    S.hb2[t] = 0.5f * w.b2[t];
    S.w3[t] = w.w3[t];
  }
  const float b3 = w.b3[0];
  tc::fence_proxy_async();
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = S.tmem + 128 * group;
  const uint32_t row_tmem = tmem + ((uint32_t)((warp & 3) * 32) << 16);  // this warp's 32 rows
  const int row = (warp & 3) * 32 + lane;
  const uint32_t idesc = tc::make_idesc_bf16(kTile, kHid);
  const uint32_t sh = tc::smem_u32(S.h[group]);
  const uint32_t sw1 = tc::smem_u32(S.w1), sw2 = tc::smem_u32(S.w2);
  uint32_t phase = 0;
  bool ok = true;
  const float2 half2 = make_float2(0.5f, 0.5f), one2 = make_float2(1.f, 1.f);
  for (long long tile = (long long)group * gridDim.x + blockIdx.x; tile < ntiles; tile += stride) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int c = t + u * 128;
      st_shared_v4(sh + tc::kmajor_off(c >> 2, 8 * (c & 3), kInPad), nxt[u].x, nxt[u].y, nxt[u].z, nxt[u].w);
    }
    tc::fence_proxy_async();
    tc::fence_before_sync();
    group_sync(group);
    tc::fence_after_sync();
    if (t == 0) {
#pragma unroll
      for (int kk = 0; kk < kInPad / 16; ++kk)
        tc::mma_bf16(tmem, tc::make_sdesc(sh + kk * 256, 128, kInPad / 8 * 128),
                     tc::make_sdesc(sw1 + kk * 256, 128, kInPad / 8 * 128), idesc, kk > 0);
      tc::mma_commit(&S.mbar[group]);
    }
    load_tile(tile + stride, nxt);  // in flight while this tile is worked on
    if (group_or(group, (warp & 3) == 0 && !tc::mbar_wait(&S.mbar[group], phase, kWaitLimit))) { ok = false; break; }
    phase ^= 1;
    tc::fence_after_sync();
    // epilogue 1: h = silu(z1 + b1) -> bf16 -> shared (A operand of the second GEMM); the
    // next 32 columns are on their way while 32 are worked on
    {
      uint32_t a[2][32];
      tc::tmem_load(row_tmem, a[0]);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        uint32_t(&z)[32] = a[k & 1];
        tc::tmem_wait(z);
        if (k < 3) tc::tmem_load(row_tmem + 32 * (k + 1), a[(k + 1) & 1]);
        uint32_t p[16];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const float4 hb = *reinterpret_cast<const float4*>(&S.hb1[32 * k + 4 * q]);
          const float2 u = __ffma2_rn(make_float2(__uint_as_float(z[4 * q]), __uint_as_float(z[4 * q + 1])), half2,
                                      make_float2(hb.x, hb.y));
          const float2 v = __ffma2_rn(make_float2(__uint_as_float(z[4 * q + 2]), __uint_as_float(z[4 * q + 3])), half2,
                                      make_float2(hb.z, hb.w));
          p[2 * q] = silu_half_bf16x2(u.x, u.y);
          p[2 * q + 1] = silu_half_bf16x2(v.x, v.y);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
          st_shared_v4(sh + tc::kmajor_off(row, 32 * k + 8 * q, kHid), p[4 * q], p[4 * q + 1], p[4 * q + 2],
                       p[4 * q + 3]);
      }
    }
    tc::fence_proxy_async();
    tc::fence_before_sync();
    group_sync(group);
    tc::fence_after_sync();
    if (t == 0) {
#pragma unroll
      for (int kk = 0; kk < kHid / 16; ++kk)
        tc::mma_bf16(tmem, tc::make_sdesc(sh + kk * 256, 128, kHid / 8 * 128),
                     tc::make_sdesc(sw2 + kk * 256, 128, kHid / 8 * 128), idesc, kk > 0);
      tc::mma_commit(&S.mbar[group]);
    }
    if (group_or(group, (warp & 3) == 0 && !tc::mbar_wait(&S.mbar[group], phase, kWaitLimit))) { ok = false; break; }
    phase ^= 1;
    tc::fence_after_sync();
    // epilogue 2: y = w3 . silu(z2 + b2) + b3, one running sum per 64 columns
    float y[2] = {0.f, 0.f};
    {
      uint32_t a[2][2][16];
      tc::tmem_load(row_tmem, a[0][0]);
      tc::tmem_load(row_tmem + 64, a[0][1]);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        uint32_t(&z)[2][16] = a[k & 1];
        tc::tmem_wait(z[0], z[1]);
        if (k < 3) {
          tc::tmem_load(row_tmem + 16 * (k + 1), a[(k + 1) & 1][0]);
          tc::tmem_load(row_tmem + 64 + 16 * (k + 1), a[(k + 1) & 1][1]);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int c = 64 * u + 16 * k + 4 * q;
            const float4 hb = *reinterpret_cast<const float4*>(&S.hb2[c]);
            const float4 w3 = *reinterpret_cast<const float4*>(&S.w3[c]);
            const float2 h0 = __ffma2_rn(make_float2(__uint_as_float(z[u][4 * q]), __uint_as_float(z[u][4 * q + 1])),
                                         half2, make_float2(hb.x, hb.y));
            const float2 h1 = __ffma2_rn(make_float2(__uint_as_float(z[u][4 * q + 2]), __uint_as_float(z[u][4 * q + 3])),
                                         half2, make_float2(hb.z, hb.w));
            const float2 s0 = __fmul2_rn(h0, __fadd2_rn(make_float2(tanh_approx(h0.x), tanh_approx(h0.y)), one2));
            const float2 s1 = __fmul2_rn(h1, __fadd2_rn(make_float2(tanh_approx(h1.x), tanh_approx(h1.y)), one2));
            y[u] = fmaf(w3.x, s0.x, y[u]);
            y[u] = fmaf(w3.y, s0.y, y[u]);
            y[u] = fmaf(w3.z, s1.x, y[u]);
            y[u] = fmaf(w3.w, s1.y, y[u]);
          }
      }
    }
    const long long r = tile * kTile + row;
    if (r < rows) out[infer_row(r, sel)] = (y[0] + y[1]) + b3;
  }
  if (!ok) {
    if (t == 0) atomicExch(err, 1);
    drain_mma(&S.drain[group], t);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(S.tmem, 256);
}

// Self-test of the bounded tensor-core waits: one block allocates tensor memory, waits
// with a bound of `polls` on an mbarrier that nothing arrives on (so the wait runs out, as
// a lost MMA completion would make the network kernels' waits run out), records the
// timeout in *err and frees its tensor memory before returning, as those kernels do.
__global__ void __launch_bounds__(128) mlp_wait_selftest_kernel(uint32_t polls, int* err) {
  __shared__ uint64_t mbar;
  __shared__ uint32_t tmem_addr;
  const int t = threadIdx.x, warp = t >> 5;
  if (warp == 0) tc::tmem_alloc(&tmem_addr, 32);
  if (t == 0) tc::mbar_init(&mbar, 1);
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (__syncthreads_or(!tc::mbar_wait(&mbar, 0, polls)) && t == 0) atomicExch(err, 1);
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem_addr, 32);
}

// ------------------------------------------------------------------ training
// One tile of 128 rows needs five GEMMs: Z1 = X W1^T, Z2 = H1 W2^T, dH1 = dZ2 W2,
// dW2 = dZ2^T H1, dW1 = dZ1^T X.  Every operand is staged once, as K-major core matrices
// of the row-major matrix; the products that need it transposed read the same bytes as an
// MN-major operand (tc::make_idesc_bf16 and tc::mn_desc), so nothing is stored twice.
// What bounds a block: the chain load -> MMA -> SiLU -> MMA -> SiLU -> MMA -> SiLU' -> MMA
// of its tile (a minibatch of 16384 rows is 128 tiles, one per SM).  Sixteen warps share
// every epilogue, four threads per row with 32 columns each, so that a phase is 32 columns
// long and the SM's tanh unit (3 x 128 evaluations per row) is what it waits for.  The
// column sums (db1, db2, dw3, of the unrounded FP32 values) are taken by a transposing
// butterfly in every warp.  Each block stores its partial gradients as they lie in its
// registers (lanes = rows, 16 bytes each: coalesced), and mlp_reduce_kernel adds the
// blocks' partials in a fixed order: no atomics, and a run is reproducible.
// Measured, one Adam step on 16384 rows: 1481 us with a thread per row, transposed operand
// copies written two bytes at a time, and the column sums and gradients by FP32 atomics
// (shared memory: a compare-and-swap loop with all 128 threads on one address); 22.7
// us now.
namespace {

constexpr int kTrainThreads = 512;
struct TrainSmem {
  uint8_t w1[kHid * kInPad * 2];  // W1 [h1][in]
  uint8_t w2[kHid * kHid * 2];    // W2 [h2][h1]
  uint8_t x[kTile * kInPad * 2];  // X [row][in]
  uint8_t h[kTile * kHid * 2];    // H1 [row][h1]
  uint8_t d[kTile * kHid * 2];    // dZ2 [row][h2], then dZ1 [row][h1]
  float b1[kHid], b2[kHid], w3[kHid];
  float part[4][kTile];           // shares of y per column quarter
  float sums[3][4][kHid];         // db1, db2, dw3 per lane quarter
  float gb3[4], loss[4];
  uint64_t mbar;
  uint64_t drain;  // drain_mma: arrives once every MMA issued so far has completed
  uint32_t tmem;
};

// Partial gradients of one block, in 16-byte units: dW2 as [column / 4][row], dW1 as
// [column / 4][row] (24 columns), then db1, db2, dw3, and (db3, loss, 0, 0).
constexpr int kPartW1 = kHid / 4 * kHid;
constexpr int kPartB1 = kPartW1 + kIn / 4 * kHid;
constexpr int kPartB2 = kPartB1 + kHid / 4;
constexpr int kPartW3 = kPartB2 + kHid / 4;
constexpr int kPartB3 = kPartW3 + kHid / 4;
constexpr int kPart4 = kPartB3 + 1;

// Sum over the warp's lanes of each of 32 values: lane l returns the sum of v[l].
// Recursive halving: 31 shuffles instead of 32 x 5.
__device__ __forceinline__ float column_sum(float (&v)[32], int lane) {
#pragma unroll
  for (int w = 16; w >= 1; w >>= 1) {
    const bool up = (lane & w) != 0;
#pragma unroll
    for (int i = 0; i < w; ++i) {
      const float keep = up ? v[i + w] : v[i], send = up ? v[i] : v[i + w];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, w);
    }
  }
  return v[0];
}

}  // namespace

// Gradient of L = sum_r (y_r - target_r)^2 * scale: block b's share over its tiles goes to
// part[b * kPart4 ..].
__global__ void __launch_bounds__(kTrainThreads, 1) mlp_train_kernel(const __nv_bfloat16* __restrict__ feat,
                                                                    const float* __restrict__ target,
                                                                    long long rows, float scale, MlpDev w,
                                                                    float4* __restrict__ part, int* err) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  TrainSmem& S = *reinterpret_cast<TrainSmem*>(smem_raw);
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int quad = warp & 3, quarter = warp >> 2;
  const int row = quad * 32 + lane;  // the TMEM lane (tile row) this thread reads
  const int col = quarter * 32;      // first of its 32 columns
  if (warp == 0) tc::tmem_alloc(&S.tmem, 512);
  if (t == 0) { tc::mbar_init(&S.mbar, 1); tc::mbar_init(&S.drain, 1); }
  const long long ntiles = (rows + kTile - 1) / kTile;
  // a tile is 128 rows x 4 chunks of 16 bytes, one per thread; row t / 4, chunk t % 4
  auto load_x = [&](long long tile) {
    const long long r = tile * kTile + (t >> 2);
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (tile < ntiles && r < rows) v = reinterpret_cast<const uint4*>(feat + r * kInPad)[t & 3];
    return v;
  };
  uint4 xv = load_x(blockIdx.x);
  stage_kmajor(S.w1, w.w1, kHid, kInPad);
  stage_kmajor(S.w2, w.w2, kHid, kHid);
  if (t < kHid) { S.b1[t] = w.b1[t]; S.b2[t] = w.b2[t]; S.w3[t] = w.w3[t]; }
  const float b3 = w.b3[0];
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  const uint32_t T_Z1 = 0, T_Z2 = 128, T_DW1 = 256, T_DW2 = 384;  // TMEM columns
  const uint32_t id_kk = tc::make_idesc_bf16(kTile, kHid);
  const uint32_t id_kn = tc::make_idesc_bf16(kTile, kHid, false, true);
  const uint32_t id_nn = tc::make_idesc_bf16(kHid, kHid, true, true);
  const uint32_t id_nn32 = tc::make_idesc_bf16(kHid, kInPad, true, true);
  const uint32_t sx = tc::smem_u32(S.x), sh = tc::smem_u32(S.h), sd = tc::smem_u32(S.d);
  const uint32_t sw1 = tc::smem_u32(S.w1), sw2 = tc::smem_u32(S.w2);
  const uint32_t SB32 = kInPad / 8 * 128, SB128 = kHid / 8 * 128;
  uint32_t phase = 0;
  bool ok = true, first = true;
  auto sync_mma = [&]() {
    tc::fence_proxy_async();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
  };
  auto wait_mma = [&]() -> bool {
    if (__syncthreads_or(!tc::mbar_wait(&S.mbar, phase, kWaitLimit))) {
      if (t == 0) atomicExch(err, 1);
      return false;
    }
    phase ^= 1;
    tc::fence_after_sync();
    return true;
  };
  float gb1 = 0.f, gb2 = 0.f, gw3 = 0.f;  // column col + lane, rows of this warp's quarter
  float gb3 = 0.f, loss = 0.f;            // this thread's row (column quarter 0 only)
  st_shared_v4(sx + tc::kmajor_off(t >> 2, 8 * (t & 3), kInPad), xv.x, xv.y, xv.z, xv.w);
  sync_mma();
  const uint32_t tmem = S.tmem;
  const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
  for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    if (t == 0) {
#pragma unroll
      for (int kk = 0; kk < kInPad / 16; ++kk)
        tc::mma_bf16(tmem + T_Z1, tc::make_sdesc(sx + kk * 256, 128, SB32),
                     tc::make_sdesc(sw1 + kk * 256, 128, SB32), id_kk, kk > 0);
      tc::mma_commit(&S.mbar);
    }
    const long long r = tile * kTile + row;
    const bool valid = r < rows;
    const float tg = valid ? target[r] : 0.f;
    xv = load_x(tile + gridDim.x);
    if (!(ok = wait_mma())) break;
    // H1 = silu(Z1 + b1)
    {
      float a[32];
      tc::tmem_ld32(tmem + lane_base + T_Z1 + col, a);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        uint32_t p[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int i = 8 * q + 2 * e;
          p[e] = pack_bf16x2(silu(a[i] + S.b1[col + i]), silu(a[i + 1] + S.b1[col + i + 1]));
        }
        st_shared_v4(sh + tc::kmajor_off(row, col + 8 * q, kHid), p[0], p[1], p[2], p[3]);
      }
    }
    sync_mma();
    if (t == 0) {
#pragma unroll
      for (int kk = 0; kk < kHid / 16; ++kk)
        tc::mma_bf16(tmem + T_Z2, tc::make_sdesc(sh + kk * 256, 128, SB128),
                     tc::make_sdesc(sw2 + kk * 256, 128, SB128), id_kk, kk > 0);
      tc::mma_commit(&S.mbar);
    }
    if (!(ok = wait_mma())) break;
    // y, g = dL/dy, dZ2 = g w3 silu'(Z2) and the column sums dw3, db2
    {
      float z[32], s[32];
      tc::tmem_ld32(tmem + lane_base + T_Z2 + col, z);
      float y = 0.f;
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        z[i] += S.b2[col + i];
        s[i] = sigmoid(z[i]);
        y = fmaf(S.w3[col + i], z[i] * s[i], y);
      }
      S.part[quarter][row] = y;
      __syncthreads();
      y = b3 + ((S.part[0][row] + S.part[1][row]) + (S.part[2][row] + S.part[3][row]));
      const float res = valid ? y - tg : 0.f;
      const float g = 2.f * res * scale;
      if (quarter == 0) { loss += res * res * scale; gb3 += g; }
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const float h2 = z[i] * s[i];
        s[i] = g * S.w3[col + i] * (s[i] * (1.f + z[i] * (1.f - s[i])));
        z[i] = g * h2;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
        st_shared_v4(sd + tc::kmajor_off(row, col + 8 * q, kHid), pack_bf16x2(s[8 * q], s[8 * q + 1]),
                     pack_bf16x2(s[8 * q + 2], s[8 * q + 3]), pack_bf16x2(s[8 * q + 4], s[8 * q + 5]),
                     pack_bf16x2(s[8 * q + 6], s[8 * q + 7]));
      sync_mma();
      if (t == 0) {
        // dH1 = dZ2 W2 (into the Z2 columns, consumed); dW2 += dZ2^T H1
#pragma unroll
        for (int kk = 0; kk < kHid / 16; ++kk)
          tc::mma_bf16(tmem + T_Z2, tc::make_sdesc(sd + kk * 256, 128, SB128),
                       tc::mn_desc(sw2 + kk * 2 * SB128, SB128), id_kn, kk > 0);
#pragma unroll
        for (int kk = 0; kk < kTile / 16; ++kk)
          tc::mma_bf16(tmem + T_DW2, tc::mn_desc(sd + kk * 2 * SB128, SB128),
                       tc::mn_desc(sh + kk * 2 * SB128, SB128), id_nn, (!first || kk > 0) ? 1u : 0u);
        tc::mma_commit(&S.mbar);
      }
      gw3 += column_sum(z, lane);  // while the tensor core works
      gb2 += column_sum(s, lane);
    }
    if (!(ok = wait_mma())) break;
    // dZ1 = dH1 silu'(Z1) and its column sums db1
    {
      float a[32], z[32];
      tc::tmem_ld32(tmem + lane_base + T_Z2 + col, a);
      tc::tmem_ld32(tmem + lane_base + T_Z1 + col, z);
#pragma unroll
      for (int i = 0; i < 32; ++i) a[i] *= silu_grad(z[i] + S.b1[col + i]);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        st_shared_v4(sd + tc::kmajor_off(row, col + 8 * q, kHid), pack_bf16x2(a[8 * q], a[8 * q + 1]),
                     pack_bf16x2(a[8 * q + 2], a[8 * q + 3]), pack_bf16x2(a[8 * q + 4], a[8 * q + 5]),
                     pack_bf16x2(a[8 * q + 6], a[8 * q + 7]));
      sync_mma();
      if (t == 0) {
        // dW1 += dZ1^T X
#pragma unroll
        for (int kk = 0; kk < kTile / 16; ++kk)
          tc::mma_bf16(tmem + T_DW1, tc::mn_desc(sd + kk * 2 * SB128, SB128),
                       tc::mn_desc(sx + kk * 2 * SB32, SB32), id_nn32, (!first || kk > 0) ? 1u : 0u);
        tc::mma_commit(&S.mbar);
      }
      gb1 += column_sum(a, lane);
    }
    if (!(ok = wait_mma())) break;
    first = false;
    st_shared_v4(sx + tc::kmajor_off(t >> 2, 8 * (t & 3), kInPad), xv.x, xv.y, xv.z, xv.w);
    sync_mma();
  }
  if (!ok) drain_mma(&S.drain, t);
  // this block's partial gradients (zeros after a timed-out wait, which is reported)
  part += (size_t)blockIdx.x * kPart4;
  const float on = ok ? 1.f : 0.f;
  {
    float a[32];
    tc::tmem_ld32(tmem + lane_base + T_DW2 + col, a);
#pragma unroll
    for (int q = 0; q < 8; ++q)
      part[(col / 4 + q) * kHid + row] =
          ok ? make_float4(a[4 * q], a[4 * q + 1], a[4 * q + 2], a[4 * q + 3]) : make_float4(0.f, 0.f, 0.f, 0.f);
    if (quarter == 0) {
      tc::tmem_ld32(tmem + lane_base + T_DW1, a);
#pragma unroll
      for (int q = 0; q < kIn / 4; ++q)
        part[kPartW1 + q * kHid + row] =
            ok ? make_float4(a[4 * q], a[4 * q + 1], a[4 * q + 2], a[4 * q + 3]) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) {
        gb3 += __shfl_xor_sync(0xffffffffu, gb3, o);
        loss += __shfl_xor_sync(0xffffffffu, loss, o);
      }
      if (lane == 0) { S.gb3[quad] = gb3; S.loss[quad] = loss; }
    }
  }
  S.sums[0][quad][col + lane] = gb1;
  S.sums[1][quad][col + lane] = gb2;
  S.sums[2][quad][col + lane] = gw3;
  tc::fence_before_sync();
  __syncthreads();
  if (t < 3 * kHid) {
    const int k = t / kHid, c = t % kHid;
    reinterpret_cast<float*>(part + kPartB1)[t] =
        on * ((S.sums[k][0][c] + S.sums[k][1][c]) + (S.sums[k][2][c] + S.sums[k][3][c]));
  } else if (t == 3 * kHid) {
    part[kPartB3] = make_float4(on * ((S.gb3[0] + S.gb3[1]) + (S.gb3[2] + S.gb3[3])),
                                on * ((S.loss[0] + S.loss[1]) + (S.loss[2] + S.loss[3])), 0.f, 0.f);
  }
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

// Adds the training blocks' partial gradients and writes the gradient (out, may be null) and
// the loss (may be null); with p, one Adam step on the FP32 master parameters with it, which
// refreshes the BF16 weight copies.  A block takes 32 of the kPart4 16-byte units: eight
// warps add every eighth block's share (independent loads), the first four combine them.
__global__ void __launch_bounds__(256) mlp_reduce_kernel(const float4* __restrict__ part, int n_part,
                                                         float* __restrict__ out, float* __restrict__ loss,
                                                         float* __restrict__ p, float* __restrict__ m,
                                                         float* __restrict__ v, float lr, float b1, float b2,
                                                         float eps, float c1, float c2,
                                                         __nv_bfloat16* __restrict__ w1b,
                                                         __nv_bfloat16* __restrict__ w2b) {
  __shared__ float4 sums[8][32];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  {
    const int u = blockIdx.x * 32 + lane;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    if (u < kPart4)
#pragma unroll 4
      for (int b = warp; b < n_part; b += 8) {
        const float4 q = part[(size_t)b * kPart4 + u];
        a.x += q.x; a.y += q.y; a.z += q.z; a.w += q.w;
      }
    sums[warp][lane] = a;
  }
  __syncthreads();
  if (t >= 128) return;
  const int u = blockIdx.x * 32 + (t >> 2), k = t & 3;
  if (u >= kPart4) return;
  float g = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) g += reinterpret_cast<const float*>(&sums[w][t >> 2])[k];
  int i;  // index in the parameter vector
  if (u < kPartW1) i = kOffW2 + (u % kHid) * kHid + 4 * (u / kHid) + k;
  else if (u < kPartB1) i = kOffW1 + ((u - kPartW1) % kHid) * kIn + 4 * ((u - kPartW1) / kHid) + k;
  else if (u < kPartB2) i = kOffB1 + 4 * (u - kPartB1) + k;
  else if (u < kPartW3) i = kOffB2 + 4 * (u - kPartB2) + k;
  else if (u < kPartB3) i = kOffW3 + 4 * (u - kPartW3) + k;
  else {
    if (k == 1 && loss) *loss = g;
    if (k != 0) return;
    i = kOffB3;
  }
  if (out) out[i] = g;
  if (!p) return;
  const float mi = b1 * m[i] + (1.f - b1) * g;
  const float vi = b2 * v[i] + (1.f - b2) * g * g;
  m[i] = mi; v[i] = vi;
  const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  p[i] = pi;
  if (i < kOffB1) {
    const int o = i / kIn, c = i % kIn;
    w1b[o * kInPad + c] = __float2bfloat16_rn(pi);
  } else if (i >= kOffW2 && i < kOffB2) {
    w2b[i - kOffW2] = __float2bfloat16_rn(pi);
  }
}

__global__ void mlp_pack_kernel(const float* __restrict__ p, __nv_bfloat16* __restrict__ w1b,
                                __nv_bfloat16* __restrict__ w2b) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < kHid * kInPad) {
    const int o = i / kInPad, k = i % kInPad;
    w1b[i] = __float2bfloat16_rn(k < kIn ? p[kOffW1 + o * kIn + k] : 0.f);
  }
  if (i < kHid * kHid) w2b[i] = __float2bfloat16_rn(p[kOffW2 + i]);
}

// ------------------------------------------------------------------ host
struct MlpHandle;
namespace snakesim {
SimStatus mlp_forward_launch(MlpHandle* h, const void* feat, long long rows, float* out, cudaStream_t st,
                             int sel);
}
struct MlpHandle {
  cudaStream_t stream = nullptr;
  uint8_t* mem = nullptr;  // owns the device buffers below
  float *p = nullptr, *m = nullptr, *v = nullptr;
  float4* part = nullptr;  // [sms][kPart4] partial gradients of the training blocks
  __nv_bfloat16 *w1b = nullptr, *w2b = nullptr;
  int* err = nullptr;
  long long adam_t = 0;
  int sms = 0;
};

namespace {
SimStatus mfail(SimStatus s, const std::string& m) { set_last_error(m.c_str()); return s; }
#define MCU(call)                                                                     \
  do {                                                                                \
    cudaError_t e_ = (call);                                                          \
    if (e_ != cudaSuccess)                                                            \
      return mfail(e_ == cudaErrorMemoryAllocation ? SIM_ENOMEM : SIM_ECUDA,          \
                   std::string(#call) + ": " + cudaGetErrorString(e_));               \
  } while (0)

MlpDev dev_of(MlpHandle* h) {
  MlpDev d;
  d.w1 = h->w1b; d.w2 = h->w2b; d.b1 = h->p + kOffB1; d.b2 = h->p + kOffB2; d.w3 = h->p + kOffW3;
  d.b3 = h->p + kOffB3;
  return d;
}

SimStatus check_err(MlpHandle* h) {
  int e = 0;
  MCU(cudaMemcpyAsync(&e, h->err, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
  MCU(cudaStreamSynchronize(h->stream));
  if (e) return mfail(SIM_ECUDA, "tensor-core wait timed out");
  return SIM_OK;
}

// Partial gradients of `rows` rows (0: no blocks) into h->part; *grid receives the blocks.
SimStatus train_launch(MlpHandle* h, const void* feat, const float* target, long long rows, float scale, int* grid) {
  const long long tiles = (rows + kTile - 1) / kTile;
  *grid = (int)std::min<long long>(tiles, h->sms);
  if (*grid == 0) return SIM_OK;
  mlp_train_kernel<<<*grid, kTrainThreads, sizeof(TrainSmem), h->stream>>>((const __nv_bfloat16*)feat, target, rows,
                                                                          scale, dev_of(h), h->part, h->err);
  MCU(cudaGetLastError());
  return SIM_OK;
}
}  // namespace

SimStatus snakesim::mlp_forward_launch(MlpHandle* h, const void* feat, long long rows, float* out,
                                       cudaStream_t st, int sel) {
  if (rows <= 0) return SIM_OK;
  const long long tiles = (rows + kTile - 1) / kTile;
  const int grid = (int)std::min<long long>(tiles, 2LL * h->sms);
  mlp_infer_kernel<<<grid, kInferThreads, sizeof(InferSmem), st>>>((const __nv_bfloat16*)feat, rows, dev_of(h),
                                                                  out, h->err, sel);
  MCU(cudaGetLastError());
  return SIM_OK;
}

extern "C" {

SimStatus mlp_create(void* stream, MlpHandle** out) {
  if (!out) return mfail(SIM_EINVAL, "null output");
  *out = nullptr;
  MlpHandle* h = new MlpHandle();
  h->stream = (cudaStream_t)stream;
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&h->sms, cudaDevAttrMultiProcessorCount, dev);
  // one allocation: the parameters, moments, weight copies and the flag (zeroed), then the
  // training blocks' partial gradients (written before they are read)
  size_t at = 0;
  auto take = [&](size_t bytes) { const size_t o = at; at += (bytes + 255) & ~(size_t)255; return o; };
  const size_t o_p = take(kNumParams * sizeof(float)), o_m = take(kNumParams * sizeof(float));
  const size_t o_v = take(kNumParams * sizeof(float)), o_w1 = take(kHid * kInPad * sizeof(__nv_bfloat16));
  const size_t o_w2 = take(kHid * kHid * sizeof(__nv_bfloat16)), o_err = take(sizeof(int));
  const size_t zeroed = at, o_part = take((size_t)std::max(1, h->sms) * kPart4 * sizeof(float4));
  cudaError_t e = cudaMalloc((void**)&h->mem, at);
  if (e != cudaSuccess) { h->mem = nullptr; mlp_destroy(h); return mfail(SIM_ENOMEM, cudaGetErrorString(e)); }
  h->p = (float*)(h->mem + o_p);
  h->m = (float*)(h->mem + o_m);
  h->v = (float*)(h->mem + o_v);
  h->w1b = (__nv_bfloat16*)(h->mem + o_w1);
  h->w2b = (__nv_bfloat16*)(h->mem + o_w2);
  h->err = (int*)(h->mem + o_err);
  h->part = (float4*)(h->mem + o_part);
  cudaMemset(h->mem, 0, zeroed);
  e = cudaFuncSetAttribute(mlp_infer_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(InferSmem));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(mlp_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem));
  if (e != cudaSuccess) { mlp_destroy(h); return mfail(SIM_ECUDA, cudaGetErrorString(e)); }
  *out = h;
  return SIM_OK;
}

SimStatus mlp_set_params(MlpHandle* h, const float* params, int is_device) {
  if (!h || !params) return mfail(SIM_EINVAL, "null handle or params");
  MCU(cudaMemcpyAsync(h->p, params, kNumParams * sizeof(float),
                      is_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, h->stream));
  mlp_pack_kernel<<<(kHid * kHid + 255) / 256, 256, 0, h->stream>>>(h->p, h->w1b, h->w2b);
  MCU(cudaGetLastError());
  MCU(cudaMemsetAsync(h->m, 0, kNumParams * sizeof(float), h->stream));
  MCU(cudaMemsetAsync(h->v, 0, kNumParams * sizeof(float), h->stream));
  h->adam_t = 0;
  if (!is_device) MCU(cudaStreamSynchronize(h->stream));
  return SIM_OK;
}

SimStatus mlp_get_params(MlpHandle* h, float* params, int is_device) {
  if (!h || !params) return mfail(SIM_EINVAL, "null handle or params");
  MCU(cudaMemcpyAsync(params, h->p, kNumParams * sizeof(float),
                      is_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, h->stream));
  if (!is_device) MCU(cudaStreamSynchronize(h->stream));
  return SIM_OK;
}

SimStatus mlp_forward(MlpHandle* h, const void* feat, int64_t rows, float* out) {
  if (!h || !feat || !out || rows < 0) return mfail(SIM_EINVAL, "bad arguments");
  if (((uintptr_t)feat & 15u) != 0) return mfail(SIM_EINVAL, "feat is not 16-byte aligned");
  SimStatus s = snakesim::mlp_forward_launch(h, feat, rows, out, h->stream, 0);
  if (s != SIM_OK) return s;
  return check_err(h);
}

SimStatus mlp_grad(MlpHandle* h, const void* feat, const float* target, int64_t rows, float scale,
                   float* grad, float* loss) {
  if (!h || !feat || !target || rows < 0) return mfail(SIM_EINVAL, "bad arguments");
  if (((uintptr_t)feat & 15u) != 0) return mfail(SIM_EINVAL, "feat is not 16-byte aligned");
  int grid = 0;
  SimStatus s = train_launch(h, feat, target, rows, scale, &grid);
  if (s != SIM_OK) return s;
  mlp_reduce_kernel<<<(kPart4 + 31) / 32, 256, 0, h->stream>>>(h->part, grid, grad, loss, nullptr, nullptr, nullptr,
                                                               0.f, 0.f, 0.f, 0.f, 1.f, 1.f, nullptr, nullptr);
  MCU(cudaGetLastError());
  return check_err(h);
}

SimStatus mlp_train_step(MlpHandle* h, const void* feat, const float* target, int64_t rows, float lr,
                         float* loss) {
  if (!h || !feat || !target || rows <= 0 || !(lr > 0.f)) return mfail(SIM_EINVAL, "bad arguments");
  if (((uintptr_t)feat & 15u) != 0) return mfail(SIM_EINVAL, "feat is not 16-byte aligned");
  int grid = 0;
  SimStatus s = train_launch(h, feat, target, rows, 1.0f / (float)rows, &grid);
  if (s != SIM_OK) return s;
  h->adam_t += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)h->adam_t), c2 = 1.f - powf(b2, (float)h->adam_t);
  mlp_reduce_kernel<<<(kPart4 + 31) / 32, 256, 0, h->stream>>>(h->part, grid, nullptr, loss, h->p, h->m, h->v, lr, b1,
                                                               b2, 1e-8f, c1, c2, h->w1b, h->w2b);
  MCU(cudaGetLastError());
  return SIM_OK;
}

SimStatus mlp_check(MlpHandle* h) {
  if (!h) return mfail(SIM_EINVAL, "null handle");
  return check_err(h);
}

SimStatus mlp_wait_selftest(uint32_t polls, void* stream, int32_t* timed_out) {
  if (polls < 1 || !timed_out) return mfail(SIM_EINVAL, "polls >= 1 and a result pointer");
  cudaStream_t st = (cudaStream_t)stream;
  int* flag = nullptr;
  MCU(cudaMalloc(&flag, sizeof(int)));
  int e = 0;
  cudaError_t c = cudaMemsetAsync(flag, 0, sizeof(int), st);
  if (c == cudaSuccess) {
    mlp_wait_selftest_kernel<<<1, 128, 0, st>>>(polls, flag);
    c = cudaGetLastError();
  }
  if (c == cudaSuccess) c = cudaMemcpyAsync(&e, flag, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (c == cudaSuccess) c = cudaStreamSynchronize(st);
  cudaFree(flag);
  if (c != cudaSuccess) return mfail(SIM_ECUDA, std::string("mlp_wait_selftest: ") + cudaGetErrorString(c));
  *timed_out = e;
  return SIM_OK;
}

SimStatus mlp_destroy(MlpHandle* h) {
  if (!h) return SIM_OK;
  cudaStreamSynchronize(h->stream);
  if (h->mem) cudaFree(h->mem);
  delete h;
  return SIM_OK;
}

}  // extern "C"

// ------------------------------------------------------------------ allocation-free forward
// Some callers cannot allocate device memory: a control loop with a hard real-time
// budget must not stall on the CUDA allocator, and a host application that gives this
// library a fixed device budget owned by its own allocator has no cudaMalloc to offer.
// For them, mlp_forward_noalloc runs the network from a parameter vector they own; the
// only working memory it needs -- the bfloat16 copies of W1 and W2 the tensor cores read,
// and the wait-timeout flag -- lives in the file-scope array below, which every GPU that
// loads the library holds until the process exits.
namespace {
constexpr size_t kNoallocW1 = (size_t)kHid * kInPad * 2;   // 8 KB
constexpr size_t kNoallocW2 = (size_t)kHid * kHid * 2;     // 32 KB
constexpr size_t kNoallocBytes = kNoallocW1 + kNoallocW2 + 256;  // + timeout flag
static_assert(kNoallocBytes == MLP_NOALLOC_SCRATCH_BYTES, "documented size");
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocBytes];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
unsigned char* g_noalloc_addr[kMaxDevices] = {};  // device address of the array, per device
unsigned long long g_noalloc_ctx[kMaxDevices] = {};  // id of the context it belongs to
int g_noalloc_sms[kMaxDevices] = {};

// The id of the calling thread's current CUDA context (0 if none yet), from the driver's
// cuCtxGetCurrent / cuCtxGetId, reached through the runtime's driver entry points (no
// link-time dependency on the driver library).  The driver never reuses an id, so a
// primary context destroyed by cudaDeviceReset and created again has a new one.
SimStatus current_context_id(unsigned long long* id) {
  typedef CUresult (*GetCur)(CUcontext*);
  typedef CUresult (*GetId)(CUcontext, unsigned long long*);
  static GetCur get_cur = nullptr;
  static GetId get_id = nullptr;
  if (!get_cur || !get_id) {
    cudaDriverEntryPointQueryResult q1 = cudaDriverEntryPointSymbolNotFound, q2 = q1;
    void *f1 = nullptr, *f2 = nullptr;
    cudaError_t e1 = cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f1, 12000, cudaEnableDefault, &q1);
    cudaError_t e2 = cudaGetDriverEntryPointByVersion("cuCtxGetId", &f2, 12000, cudaEnableDefault, &q2);
    if (e1 != cudaSuccess || e2 != cudaSuccess || q1 != cudaDriverEntryPointSuccess ||
        q2 != cudaDriverEntryPointSuccess || !f1 || !f2)
      return mfail(SIM_ECUDA, "cuCtxGetCurrent / cuCtxGetId entry points not available");
    get_cur = reinterpret_cast<GetCur>(f1);
    get_id = reinterpret_cast<GetId>(f2);
  }
  CUcontext c = nullptr;
  if (get_cur(&c) != CUDA_SUCCESS) return mfail(SIM_ECUDA, "cuCtxGetCurrent failed");
  *id = 0;
  if (c && get_id(c, id) != CUDA_SUCCESS) return mfail(SIM_ECUDA, "cuCtxGetId failed");
  return SIM_OK;
}

// Set-up, once per device and context, with that device current: the array's device
// address (the name g_noalloc_scratch in host code is only a host-side stand-in) and the
// kernel's shared-memory opt-in.  A later context on the device (after cudaDeviceReset)
// is set up again.
SimStatus noalloc_setup(int dev, unsigned char** addr, int* sms) {
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  unsigned long long ctx = 0;
  SimStatus s = current_context_id(&ctx);
  if (s != SIM_OK) return s;
  if (!g_noalloc_addr[dev] || ctx == 0 || ctx != g_noalloc_ctx[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);  // creates the context if needed
    if (e != cudaSuccess) return mfail(SIM_ECUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
    e = cudaFuncSetAttribute(mlp_infer_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(InferSmem));
    if (e != cudaSuccess) return mfail(SIM_ECUDA, std::string("cudaFuncSetAttribute: ") + cudaGetErrorString(e));
    int n = 0;
    e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return mfail(SIM_ECUDA, std::string("cudaDeviceGetAttribute: ") + cudaGetErrorString(e));
    if (ctx == 0 && (s = current_context_id(&ctx)) != SIM_OK) return s;
    g_noalloc_sms[dev] = n;
    g_noalloc_addr[dev] = static_cast<unsigned char*>(p);
    g_noalloc_ctx[dev] = ctx;
  }
  *addr = g_noalloc_addr[dev];
  *sms = g_noalloc_sms[dev];
  return SIM_OK;
}
}  // namespace

extern "C" SimStatus mlp_forward_noalloc(const float* params, int32_t n_params, const void* feat,
                                         int64_t rows, float* out, void* stream) {
  if (!params || !feat || !out || rows < 0) return mfail(SIM_EINVAL, "null pointer or rows < 0");
  if (((uintptr_t)feat & 15u) != 0) return mfail(SIM_EINVAL, "feat is not 16-byte aligned");
  if (n_params != kNumParams)
    return mfail(SIM_EINVAL, "mlp_forward_noalloc: its static working array holds the bfloat16 weights of "
                             "exactly one 24-128-128-1 network (" + std::to_string(kNumParams) +
                             " parameters, " + std::to_string(kNoallocBytes) + " bytes); got " +
                             std::to_string(n_params) + " parameters");
  int dev = 0;
  MCU(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return mfail(SIM_EINVAL, "device index out of range");
  unsigned char* base = nullptr;
  int sms = 0;
  SimStatus s = noalloc_setup(dev, &base, &sms);
  if (s != SIM_OK) return s;
  if (rows == 0) return SIM_OK;
  cudaStream_t st = (cudaStream_t)stream;
  __nv_bfloat16* w1b = reinterpret_cast<__nv_bfloat16*>(base);
  __nv_bfloat16* w2b = reinterpret_cast<__nv_bfloat16*>(base + kNoallocW1);
  int* err = reinterpret_cast<int*>(base + kNoallocW1 + kNoallocW2);
  // the array keeps the previous call's contents: the flag must start at zero
  MCU(cudaMemsetAsync(err, 0, sizeof(int), st));
  mlp_pack_kernel<<<(kHid * kHid + 255) / 256, 256, 0, st>>>(params, w1b, w2b);
  MCU(cudaGetLastError());
  MlpDev d;
  d.w1 = w1b; d.w2 = w2b;
  d.b1 = params + kOffB1; d.b2 = params + kOffB2; d.w3 = params + kOffW3; d.b3 = params + kOffB3;
  const long long tiles = (rows + kTile - 1) / kTile;
  const int grid = (int)std::min<long long>(tiles, 2LL * sms);
  mlp_infer_kernel<<<grid, kInferThreads, sizeof(InferSmem), st>>>((const __nv_bfloat16*)feat, rows, d, out, err, 0);
  MCU(cudaGetLastError());
  int e = 0;
  MCU(cudaMemcpyAsync(&e, err, sizeof(int), cudaMemcpyDeviceToHost, st));
  MCU(cudaStreamSynchronize(st));
  if (e) return mfail(SIM_ECUDA, "tensor-core wait timed out");
  return SIM_OK;
}
