// The warm-start network (64 -> 256 -> 256 -> 256 -> 64, ReLU on the hidden
// layers; BF16 operands, FP32 accumulation) on chip, a CTA per SM taking
// 128-row tiles of the input in turn: k_mlp_infer, two tiles in flight;
// k_mlp_fused, the forward pass of training with the loss and the whole
// backward chain behind it; and the weight gradients of all layers in
// k_mlp_wgrad.
//
//   * operands in shared memory in the tensor core's K-major layout with the
//     128-byte swizzle (8-row groups of 1024 bytes), written by TMA tiled
//     loads (cp.async.bulk.tensor, tensor maps with SWIZZLE_128B) for the
//     input and the weights, and by the epilogue's swizzled stores for the
//     activations (or gradients), which stay in one 64 KB buffer per tile;
//   * the weight blocks ([256 x 64] each) stream through a ring from L2 (in
//     training the output layer's 64 x 256 stay resident);
//   * warp 17 issues the TMA loads, warp 16 the MMAs (M = 128, K = 16 per
//     instruction) and the TMA stores, warps 0-15 read the accumulators back
//     (tcgen05.ld; warp w the lanes 32 (w % 4).. and half (w / 4) % 2 of 64
//     columns), add the bias, apply ReLU (or the saved mask), round to BF16
//     and store the next layer's operand: two groups of eight warps, in
//     training a group the even, the other the odd 64-column blocks of a
//     layer, in inference a group per tile in flight;
//   * training: a layer's epilogue hands its operand over in four K-blocks, and
//     two accumulators (256 fp32 columns of tensor memory each) alternate, so
//     the next layer's MMAs start when the first 64 columns are ready instead
//     of after the last.
// Measured: inference of 444544 rows 233 -> 164 us (0.9 PFLOP/s; a tile 13.6 k
// cycles, 5.1 k of them tensor work, 2.6 k waits for weights with two 32 KB
// blocks in flight, 3.1 k for epilogues where the short first and last layers
// meet); a training step of 16384 rows 548 -> 80 us.
// Training keeps the ReLU masks in registers, forms the loss and its gradient
// in the output epilogue, and stores the hidden activations and the gradients
// of every layer row-major by TMA (k_mlp_wgrad reads them as they are, with
// MN-major descriptors: no transposed copies).
// Every mbarrier wait is bounded: on timeout the kernel records an error,
// waits (bounded) for its copies in flight, frees its tensor memory and
// returns.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <algorithm>
#include <string>

#include "dm_internal.h"
#include "dm_mlp.cuh"
#include "dm_tc.cuh"

namespace dm {

namespace {

constexpr int kTM = 128;         // rows per tile
constexpr int kGroup = 256;      // threads of an epilogue group (8 warps)
constexpr int kEpi = 2 * kGroup;
constexpr int kThreadsF = kEpi + 64;  // and the MMA and the TMA warp
constexpr int kStages = 3;
// shared memory map (bytes from a 1024-aligned base)
constexpr int kOffW4 = 0;                       // 4 K-blocks of [64][64] bf16: 32 KB
constexpr int kOffH = kOffW4 + 4 * 64 * 128;    // 4 K-blocks of [128][64]: 64 KB
constexpr int kOffX = kOffH + 4 * kTM * 128;    // [128][64]: 16 KB (input; output gradient)
constexpr int kOffRing = kOffX + kTM * 128;     // 3 x [256][64]: 96 KB
constexpr int kStageBytes = 256 * 128;
constexpr int kOffBias = kOffRing + kStages * kStageBytes;  // fp32 biases: 3 x 256 + 64
constexpr int kOffBar = kOffBias + (3 * 256 + 64) * 4;
constexpr int kNumBars = 2 * kStages + 12;
constexpr int kSmemFused = kOffBar + 8 * kNumBars + 16 + 1024;  // barriers, TMEM slot, alignment slack
static_assert(kSmemFused <= 227 * 1024, "shared memory of the fused kernel");
constexpr uint32_t kTmemCols = 512;  // two accumulators of 256 columns

constexpr unsigned kFullMask = 0xffffffffu;

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t *>(&h);
}

// bf16 pair of (x + b, y + c), and the larger of it and 0 (NaN: 0)
__device__ __forceinline__ uint32_t bias_pair(uint32_t x, uint32_t y, float b, float c) {
  uint64_t v, w;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "r"(x), "r"(y));
  asm("mov.b64 %0, {%1, %2};" : "=l"(w) : "f"(b), "f"(c));
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(v), "l"(w));
  float lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
  return pack_bf16(lo, hi);
}
__device__ __forceinline__ uint32_t relu_bf16(uint32_t x) {
  const __nv_bfloat162 z = __hmax2(*reinterpret_cast<const __nv_bfloat162 *>(&x), __nv_bfloat162(0.0f, 0.0f));
  return *reinterpret_cast<const uint32_t *>(&z);
}

// Bounded wait that also gives up when another role of the CTA has failed.
__device__ __forceinline__ bool wait_on(uint64_t *bar, uint32_t parity, volatile int *fail) {
  const uint32_t a = tc::smem_u32(bar);
  for (uint32_t it = 0; it < tc::kWaitLimit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
    if ((it & 255u) == 255u && *fail) return false;
  }
  *fail = 1;
  return false;
}
// The same by a whole warp, with one answer for all its lanes: what follows
// takes every lane (tcgen05.ld), also where only some of them gave up.
__device__ __forceinline__ bool wait_warp(uint64_t *bar, uint32_t parity, volatile int *fail) {
  return __all_sync(kFullMask, wait_on(bar, parity, fail));
}
__device__ __forceinline__ void arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(bar)) : "memory");
}
// One arrival for the warp, after every lane's fences (256 arrivals of single
// threads serialise on the barrier's word).
__device__ __forceinline__ void warp_arrive(uint64_t *bar) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0) arrive(bar);
}
__device__ __forceinline__ void tma_store_2d(const void *tmap, int x, int y, const void *src) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                   reinterpret_cast<uint64_t>(tmap)),
               "r"(x), "r"(y), "r"(tc::smem_u32(src))
               : "memory");
}
__device__ __forceinline__ void store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void store_read_wait() {  // the sources have been read
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void store_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

struct FusedMaps {
  CUtensorMap x, w1, w2, w3, w4;  // loads
  CUtensorMap t4, t3, t2;         // training: transposed weights
  CUtensorMap a[3], d[3], dy;     // training: stores of activations and gradients
};

struct TrainArgs {
  const float *target;  // [M][n_valid]
  int n_valid;
  float scale_den;      // M n_valid
  double loss_den;
  double *loss;
  float *gb4;           // [CTAs][4][64] partial sums of the output gradient
};

}  // namespace

__global__ void __launch_bounds__(kThreadsF, 1)
    k_mlp_fused(const __grid_constant__ FusedMaps maps, const float *__restrict__ b1,
                const float *__restrict__ b2, const float *__restrict__ b3,
                const float *__restrict__ b4, int ntiles, int *err, TrainArgs ta) {
  using namespace tc;
  constexpr int kBlocks = 18;  // streamed weight blocks per tile
  extern __shared__ char smem_raw[];
  char *smem = reinterpret_cast<char *>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  char *W4s = smem + kOffW4, *Hs = smem + kOffH, *Xs = smem + kOffX, *Ring = smem + kOffRing;
  float *sbias = reinterpret_cast<float *>(smem + kOffBias);
  uint64_t *bar = reinterpret_cast<uint64_t *>(smem + kOffBar);
  uint64_t *bar_full = bar, *bar_free = bar + kStages, *bar_acc = bar + 2 * kStages;
  uint64_t *bar_h = bar_acc + 2, *bar_w4 = bar_h + 4, *bar_x = bar_w4 + 1, *bar_xfree = bar_w4 + 2;
  uint64_t *bar_dy = bar_w4 + 3, *bar_stored = bar_w4 + 4;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bar + kNumBars);
  volatile int *fail = reinterpret_cast<volatile int *>(tmem_slot + 1);

  const int my_tiles = blockIdx.x < ntiles ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;

  if (warp == 16) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int i = 0; i < 2 * kStages + 2; ++i) mbar_init(&bar[i], 1);
    for (int i = 0; i < 4; ++i) mbar_init(&bar_h[i], kGroup / 32);
    mbar_init(bar_w4, 1);
    mbar_init(bar_x, 1);
    mbar_init(bar_xfree, 2);
    mbar_init(bar_dy, kEpi / 32);
    mbar_init(bar_stored, 1);
    *fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  for (int i = tid; i < 3 * 256 + 64; i += kThreadsF)
    sbias[i] = i < 256 ? b1[i] : (i < 512 ? b2[i - 256] : (i < 768 ? b3[i - 512] : b4[i - 768]));
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = *tmem_slot;

  if (warp == 17) {
    // ---- TMA loads: the resident weights, then per tile its input and the
    // weight blocks in the order of use, as far ahead as the ring allows
    if (lane == 0 && my_tiles > 0) {
      mbar_expect_tx(bar_w4, 4 * 64 * 128);
      for (int kb = 0; kb < 4; ++kb) tma_load_2d(W4s + kb * 64 * 128, &maps.w4, 64 * kb, 0, bar_w4);
      int g = 0, loaded = 0;
      bool ok = true;
      for (int i = 0; i < my_tiles && ok; ++i) {
        if (i > 0 && !(ok = wait_on(bar_xfree, (uint32_t)((i - 1) & 1), fail))) break;
        mbar_expect_tx(bar_x, kTM * 128);
        tma_load_2d(Xs, &maps.x, 0, ((int)blockIdx.x + i * (int)gridDim.x) * kTM, bar_x);
        loaded = i + 1;
        for (int b = 0; b < kBlocks; ++b, ++g) {
          const int s = g % kStages;
          if (g >= kStages && !(ok = wait_on(&bar_free[s], (uint32_t)((g / kStages - 1) & 1), fail))) break;
          mbar_expect_tx(&bar_full[s], (uint32_t)kStageBytes);
          const CUtensorMap *map = b == 0   ? &maps.w1
                                   : b <= 4 ? &maps.w2
                                   : b <= 8 ? &maps.w3
                                   : b == 9 ? &maps.t4
                                   : b < 14 ? &maps.t3
                                            : &maps.t2;
          const int kb = b == 0 || b == 9 ? 0 : (b < 9 ? (b - 1) & 3 : (b - 10) & 3);
          tma_load_2d(Ring + s * kStageBytes, map, 64 * kb, 0, &bar_full[s]);
        }
      }
      if (!ok || *fail) {  // what is in flight lands before the CTA leaves (bounded)
        mbar_wait(bar_w4, 0);
        for (int k = g > kStages ? g - kStages : 0; k < g; ++k)
          mbar_wait(&bar_full[k % kStages], (uint32_t)((k / kStages) & 1));
        if (loaded) mbar_wait(bar_x, (uint32_t)((loaded - 1) & 1));
      }
    }
  } else if (warp == 16) {
    // ---- MMAs and stores, by one lane
    if (lane == 0 && my_tiles > 0) {
      int g = 0, ph = 0, hphase = 0;
      bool ok = true;
      // K-block b of a layer: A at `a`, B at `w` (N rows), into accumulator ph
      auto mma_block = [&](const char *a, const char *w, int n, bool first) {
        const uint32_t a0 = smem_u32(a), w0 = smem_u32(w), d = tmem + 256u * (uint32_t)(ph & 1);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          mma_bf16(d, make_desc(a0 + 32 * kk, 16, 1024, kSwizzle128B),
                   make_desc(w0 + 32 * kk, 16, 1024, kSwizzle128B), make_idesc(kTM, n), (first && kk == 0) ? 0u : 1u);
      };
      // a layer whose operand the epilogue leaves in H, K-block by K-block; its
      // copy to global memory (training) goes out as each block is complete
      auto h_layer = [&](bool resident, const CUtensorMap *st, int y) {
        for (int kb = 0; kb < 4 && ok; ++kb) {
          if (!(ok = wait_on(&bar_h[kb], (uint32_t)(hphase & 1), fail))) return;
          asm volatile("tcgen05.fence::after_thread_sync;");
          tma_store_2d(st, 64 * kb, y, Hs + kb * (kTM * 128));
          if (resident) {
            mma_block(Hs + kb * (kTM * 128), W4s + kb * 64 * 128, 64, kb == 0);
          } else {
            const int s = g % kStages;
            if (!(ok = wait_on(&bar_full[s], (uint32_t)((g / kStages) & 1), fail))) return;
            mma_block(Hs + kb * (kTM * 128), Ring + s * kStageBytes, 256, kb == 0);
            mma_commit(&bar_free[s]);
            ++g;
          }
        }
        mma_commit(&bar_acc[ph & 1]);
        ++ph;
        ++hphase;
        store_commit();
        store_read_wait();
        arrive(bar_stored);
      };
      // a layer whose operand is the input tile (or the output gradient in its place)
      auto x_layer = [&]() {
        const int s = g % kStages;
        if (!(ok = wait_on(&bar_full[s], (uint32_t)((g / kStages) & 1), fail))) return;
        mma_block(Xs, Ring + s * kStageBytes, 256, true);
        mma_commit(&bar_free[s]);
        ++g;
      };
      for (int i = 0; i < my_tiles && ok; ++i) {
        const int y = ((int)blockIdx.x + i * (int)gridDim.x) * kTM;
        if (!(ok = wait_on(bar_x, (uint32_t)(i & 1), fail))) break;
        x_layer();
        if (!ok) break;
        mma_commit(&bar_acc[ph & 1]);
        ++ph;
        h_layer(false, &maps.a[0], y);
        if (ok) h_layer(false, &maps.a[1], y);
        if (ok && i == 0) ok = wait_on(bar_w4, 0, fail);
        if (ok) h_layer(true, &maps.a[2], y);
        if (ok) {
          if (!(ok = wait_on(bar_dy, (uint32_t)(i & 1), fail))) break;
          asm volatile("tcgen05.fence::after_thread_sync;");
          tma_store_2d(&maps.dy, 0, y, Xs);
          store_commit();
          x_layer();
          if (!ok) break;
          mma_commit(bar_xfree);
          mma_commit(&bar_acc[ph & 1]);
          ++ph;
          store_read_wait();
          arrive(bar_xfree);
          h_layer(false, &maps.d[2], y);
          if (ok) h_layer(false, &maps.d[1], y);
          for (int kb = 0; kb < 4 && ok; ++kb) {  // the first layer's gradient is only stored
            if (!(ok = wait_on(&bar_h[kb], (uint32_t)(hphase & 1), fail))) break;
            tma_store_2d(&maps.d[0], 64 * kb, y, Hs + kb * (kTM * 128));
          }
          if (!ok) break;
          ++hphase;
          store_commit();
          store_read_wait();
          arrive(bar_stored);
        }
      }
      store_wait();
      if (!ok || *fail) {
        // every MMA issued so far is done before the tensor memory is freed
        mma_commit(bar_w4);
        mbar_wait(bar_w4, 1);
      }
    }
  } else {
    // ---- epilogues
    const int quarter = warp & 3, part = warp >> 2, half = part & 1, group = warp >> 3;
    const int row = quarter * 32 + lane;  // this thread's accumulator lane / tile row
    const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
    int ph = 0, stores = 0;
    bool ok = true;
    uint32_t mask[3][2];  // ReLU masks of the hidden layers
    float gb = 0.0f;      // output column 16 part + lane's gradient sum
    auto acc_ready = [&]() -> uint32_t {
      ok = ok && wait_warp(&bar_acc[ph & 1], (uint32_t)((ph >> 1) & 1), fail);
      asm volatile("tcgen05.fence::after_thread_sync;");
      const uint32_t t = tmem + 256u * (uint32_t)(ph & 1) + lane_off;
      ++ph;
      return t;
    };
    // eight columns (chunk ch of the row's eight, swizzled) of the thread's row
    // of a K-block in H (or Xs)
    auto put = [&](char *blk, int ch, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
      *reinterpret_cast<uint4 *>(blk + row * 128 + ((ch ^ (row & 7)) << 4)) = make_uint4(a, b, c, d);
    };
    // the generic-proxy stores become visible to the tensor core's (and TMA's) reads
    auto publish = [] { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); };
    // hidden layer l, forward (bias, ReLU) or backward (mask), into H
    auto hidden = [&](int l, bool back) {
      const uint32_t t = acc_ready();
      if (!ok) return;
      if (stores > 0 && !(ok = wait_warp(bar_stored, (uint32_t)((stores - 1) & 1), fail))) return;
      ++stores;
      uint32_t r[2][32];  // the group's K-blocks: group, group + 2
      const uint32_t tc0 = t + (uint32_t)(64 * group + 32 * half);
      tmem_ld16_nowait(tc0, r[0]);
      tmem_ld16_nowait(tc0 + 16u, r[0] + 16);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int kb = group + 2 * u;
        tmem_wait32(r[u]);
        if (u == 0) {  // the next block's columns come in behind this one's arithmetic
          tmem_ld16_nowait(tc0 + 128u, r[1]);
          tmem_ld16_nowait(tc0 + 144u, r[1] + 16);
        }
        char *blk = Hs + kb * (kTM * 128);
        const float *bias = sbias + 256 * l + 64 * kb + 32 * half;
        uint32_t mk = 0;
        if (back) {
#pragma unroll
          for (int k = 0; k < 3; ++k)
            if (k == l) mk = mask[k][u];
        }
#pragma unroll
        for (int ch = 0; ch < 4; ++ch) {
          uint32_t w[4];
#pragma unroll
          for (int e = 0; e < 8; e += 4) {
            const int j = 8 * ch + e;
            float v[4];
            if (!back) {
              const float4 bb = *reinterpret_cast<const float4 *>(bias + j);
              const float b4[4] = {bb.x, bb.y, bb.z, bb.w};
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                v[k] = fmaxf(__uint_as_float(r[u][j + k]) + b4[k], 0.0f);
                mk |= v[k] > 0.0f ? 1u << (j + k) : 0u;
              }
            } else {
#pragma unroll
              for (int k = 0; k < 4; ++k) v[k] = (mk >> (j + k)) & 1u ? __uint_as_float(r[u][j + k]) : 0.0f;
            }
            w[e / 2] = pack_bf16(v[0], v[1]);
            w[e / 2 + 1] = pack_bf16(v[2], v[3]);
          }
          put(blk, 4 * half + ch, w[0], w[1], w[2], w[3]);
        }
        if (!back) {
#pragma unroll
          for (int k = 0; k < 3; ++k)
            if (k == l) mask[k][u] = mk;
        }
        publish();
        asm volatile("tcgen05.fence::before_thread_sync;");
        warp_arrive(&bar_h[kb]);
      }
    };
    for (int i = 0; i < my_tiles && ok; ++i) {
      const int tile = (int)blockIdx.x + i * (int)gridDim.x;
#pragma unroll
      for (int l = 0; l < 3; ++l)
        if (ok) hidden(l, false);
      if (!ok) break;
      const uint32_t t = acc_ready();
      if (!ok) break;
      // the output layer: 16 columns a warp
      uint32_t r[16];
      tmem_ld16(t + (uint32_t)(16 * part), r);
      const float *bo = sbias + 768 + 16 * part;
      // loss (summed in FP64) and its gradient on the first n_valid columns
      const float *yt = ta.target + ((size_t)tile * kTM + row) * ta.n_valid;
      double ls = 0.0;
      float v[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const int c = 16 * part + j;
        v[j] = 0.0f;
        if (c < ta.n_valid) {  // uniform over the warp
          const float d = __uint_as_float(r[j]) + bo[j] - yt[c];
          ls += (double)d * d;
          v[j] = 2.0f * d / ta.scale_den;
          float sum = v[j];
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(kFullMask, sum, o);
          if (lane == j) gb += sum;
        }
      }
#pragma unroll
      for (int ch = 0; ch < 2; ++ch) {
        const float *a = v + 8 * ch;
        put(Xs, 2 * part + ch, pack_bf16(a[0], a[1]), pack_bf16(a[2], a[3]), pack_bf16(a[4], a[5]),
            pack_bf16(a[6], a[7]));
      }
      publish();
      asm volatile("tcgen05.fence::before_thread_sync;");
      warp_arrive(bar_dy);
      if (16 * part < ta.n_valid) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ls += __shfl_xor_sync(kFullMask, ls, o);
        if (lane == 0) atomicAdd(ta.loss, ls / ta.loss_den);
      }
#pragma unroll
      for (int l = 2; l >= 0; --l)
        if (ok) hidden(l, true);
    }
    if (lane < 16) ta.gb4[((size_t)blockIdx.x * 4 + quarter) * 64 + 16 * part + lane] = gb;
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (tid == 0 && *fail) atomicExch(err, 1);
  if (warp == 16)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
}

namespace {

// ---- inference.  One tile's layers are a chain -- accumulator ready, read
// back, rounded, stored, fenced, handed over, multiplied -- whose waits one tile
// at a time exposes (16.5 k cycles a tile, 5 k of them tensor work).  So a CTA
// has two tiles in flight, each with its operand buffer, its 256 accumulator
// columns and eight epilogue warps: one's epilogue runs beside the other's
// MMAs.  The weight blocks, the output layer's too, stream through the ring
// once per tile.  (Halves of 128 output columns of one tile with two operand
// buffers took 22 k cycles: MMAs of N = 128 read shared memory at its limit.)
constexpr int kIStages = 2;
constexpr int kIOffX = 2 * 4 * kTM * 128;               // after two operand buffers of 64 KB
constexpr int kIOffRing = kIOffX + 2 * kTM * 128;
constexpr int kIOffBar = kIOffRing + kIStages * kStageBytes;
constexpr int kINumBars = 2 * kIStages + 8 + 1;
constexpr int kSmemInfer = kIOffBar + 8 * kINumBars + 16 + 1024;
static_assert(kSmemInfer <= 227 * 1024, "shared memory of the inference kernel");

struct InferMaps {
  CUtensorMap x, w1, w2, w3, w4;
};

}  // namespace

__global__ void __launch_bounds__(kThreadsF, 1)
    k_mlp_infer(const __grid_constant__ InferMaps maps, const float *__restrict__ b1, const float *__restrict__ b2,
                const float *__restrict__ b3, const float *__restrict__ b4, float *__restrict__ Y, int ntiles,
                int *err) {
  using namespace tc;
  extern __shared__ char smem_raw[];
  char *smem = reinterpret_cast<char *>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  char *Ring = smem + kIOffRing;
  uint64_t *bar = reinterpret_cast<uint64_t *>(smem + kIOffBar);
  uint64_t *bar_full = bar, *bar_free = bar + kIStages;
  // per tile in flight: accumulator complete, accumulator read and operand
  // stored, input in, input read
  uint64_t *bar_acc = bar + 2 * kIStages, *bar_h = bar_acc + 2, *bar_x = bar_acc + 4, *bar_xfree = bar_acc + 6;
  uint64_t *bar_end = bar_acc + 8;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bar + kINumBars);
  volatile int *fail = reinterpret_cast<volatile int *>(tmem_slot + 1);

  const int my_tiles = blockIdx.x < ntiles ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  const auto tile_of = [&](int i) { return (int)blockIdx.x + i * (int)gridDim.x; };
  // order of the layers: in slot v, layer v % 4 of an even tile, then of the odd
  // one after it (one or two layers apart 176 us instead of 164, three the same)
  const int slots = 4 * ((my_tiles + 1) / 2);

  if (warp == 16) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int i = 0; i < kINumBars; ++i) mbar_init(&bar[i], 1);
    for (int i = 0; i < 2; ++i) mbar_init(&bar_h[i], kGroup / 32);
    *fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = *tmem_slot;

  if (warp == 17) {
    // ---- TMA loads: the two tiles' inputs, then per layer and tile the weight
    // blocks, as far ahead as the ring allows
    if (lane == 0 && my_tiles > 0) {
      int g = 0, loaded[2] = {0, 0};
      bool ok = true;
      auto weights = [&](int l, int kb) {
        const int s = g % kIStages;
        if (g >= kIStages && !(ok = ok && wait_on(&bar_free[s], (uint32_t)((g / kIStages - 1) & 1), fail))) return;
        char *dst = Ring + s * kStageBytes;
        mbar_expect_tx(&bar_full[s], (uint32_t)kStageBytes);
        if (l < 3) {
          tma_load_2d(dst, l == 0 ? &maps.w1 : l == 1 ? &maps.w2 : &maps.w3, 64 * kb, 0, &bar_full[s]);
        } else {
          for (int u = 0; u < 4; ++u) tma_load_2d(dst + u * 64 * 128, &maps.w4, 64 * u, 0, &bar_full[s]);
        }
        ++g;
      };
      auto input = [&](int i) {
        const int t = i & 1;
        mbar_expect_tx(&bar_x[t], kTM * 128);
        tma_load_2d(smem + kIOffX + t * (kTM * 128), &maps.x, 0, tile_of(i) * kTM, &bar_x[t]);
        ++loaded[t];
      };
      input(0);
      if (my_tiles > 1) input(1);
      for (int v = 0; v < slots && ok; ++v)
        for (int t = 0; t < 2 && ok; ++t) {
          const int l = v & 3, i = 2 * (v >> 2) + t;
          if (i >= my_tiles) continue;
          for (int kb = 0; kb < (l == 1 || l == 2 ? 4 : 1) && ok; ++kb) weights(l, kb);
          if (l == 1 && i + 2 < my_tiles && ok) {  // the first layer has read the input
            ok = wait_on(&bar_xfree[t], (uint32_t)((i >> 1) & 1), fail);
            if (ok) input(i + 2);
          }
        }
      if (!ok || *fail) {  // what is in flight lands before the CTA leaves (bounded)
        for (int k = g > kIStages ? g - kIStages : 0; k < g; ++k)
          mbar_wait(&bar_full[k % kIStages], (uint32_t)((k / kIStages) & 1));
        for (int t = 0; t < 2; ++t)
          if (loaded[t]) mbar_wait(&bar_x[t], (uint32_t)((loaded[t] - 1) & 1));
      }
    }
  } else if (warp == 16) {
    // ---- MMAs, by one lane
    if (lane == 0 && my_tiles > 0) {
      int g = 0, hphase[2] = {0, 0};
      bool ok = true;
      // K = 64 at `a` against n weight rows at `w`, into accumulator columns d
      auto mma_block = [&](const char *a, const char *w, int n, uint32_t d, bool first) {
        const uint32_t a0 = smem_u32(a), w0 = smem_u32(w);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          mma_bf16(tmem + d, make_desc(a0 + 32 * kk, 16, 1024, kSwizzle128B),
                   make_desc(w0 + 32 * kk, 16, 1024, kSwizzle128B), make_idesc(kTM, n), (first && kk == 0) ? 0u : 1u);
      };
      for (int v = 0; v < slots && ok; ++v)
        for (int t = 0; t < 2 && ok; ++t) {
          const int l = v & 3, i = 2 * (v >> 2) + t;
          if (i >= my_tiles) continue;
          const uint32_t d = 256u * (uint32_t)t;
          char *H = smem + t * (4 * kTM * 128);
          if (l == 0) ok = wait_on(&bar_x[t], (uint32_t)((i >> 1) & 1), fail);
          // the accumulator has been read, the operand (layers 1 on) stored
          if (ok && v > 0) {
            ok = wait_on(&bar_h[t], (uint32_t)(hphase[t] & 1), fail);
            ++hphase[t];
          }
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;");
          for (int kb = 0; kb < (l == 1 || l == 2 ? 4 : 1) && ok; ++kb) {
            const int s = g % kIStages;
            if (!(ok = wait_on(&bar_full[s], (uint32_t)((g / kIStages) & 1), fail))) break;
            const char *w = Ring + s * kStageBytes;
            if (l == 3) {
              for (int q = 0; q < 4; ++q) mma_block(H + q * (kTM * 128), w + q * 64 * 128, 64, d, q == 0);
            } else {
              mma_block(l == 0 ? smem + kIOffX + t * (kTM * 128) : H + kb * (kTM * 128), w, 256, d, kb == 0);
            }
            mma_commit(&bar_free[s]);
            ++g;
          }
          if (!ok) break;
          if (l == 0) mma_commit(&bar_xfree[t]);
          mma_commit(&bar_acc[t]);
        }
      if (!ok || *fail) {
        // every MMA issued so far is done before the tensor memory is freed
        mma_commit(bar_end);
        mbar_wait(bar_end, 0);
      }
    }
  } else {
    // ---- epilogues: warps 0-7 of the even tiles, 8-15 of the odd ones
    const int quarter = warp & 3, half = (warp >> 2) & 1, t = warp >> 3;
    const int row = quarter * 32 + lane;  // this thread's accumulator lane / tile row
    const uint32_t acc = tmem + ((uint32_t)(quarter * 32) << 16) + 256u * (uint32_t)t + 32u * (uint32_t)half;
    char *H = smem + t * (4 * kTM * 128);
    uint32_t phase = 0;
    bool ok = true;
    auto acc_ready = [&]() {
      ok = ok && wait_warp(&bar_acc[t], phase & 1u, fail);
      ++phase;
      asm volatile("tcgen05.fence::after_thread_sync;");
    };
    for (int i = t; i < my_tiles && ok; i += 2) {
#pragma unroll 1
      for (int l = 0; l < 3; ++l) {
        acc_ready();
        if (!ok) break;
        const float *bl = l == 0 ? b1 : l == 1 ? b2 : b3;
        uint32_t r[2][32];
        tmem_ld16_nowait(acc, r[0]);
        tmem_ld16_nowait(acc + 16u, r[0] + 16);
#pragma unroll
        for (int kb = 0; kb < 4; ++kb) {
          tmem_wait32(r[kb & 1]);
          if (kb < 3) {  // the next block's columns come in behind this one's arithmetic
            tmem_ld16_nowait(acc + (uint32_t)(64 * (kb + 1)), r[(kb + 1) & 1]);
            tmem_ld16_nowait(acc + (uint32_t)(64 * (kb + 1) + 16), r[(kb + 1) & 1] + 16);
          }
          const float4 *bias = reinterpret_cast<const float4 *>(bl + 64 * kb + 32 * half);
          char *rowp = H + kb * (kTM * 128) + row * 128;
#pragma unroll
          for (int ch = 0; ch < 4; ++ch) {
            uint32_t w[4];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const float4 bb = __ldg(bias + 2 * ch + e);
              const uint32_t *x = r[kb & 1] + 8 * ch + 4 * e;
              w[2 * e] = relu_bf16(bias_pair(x[0], x[1], bb.x, bb.y));
              w[2 * e + 1] = relu_bf16(bias_pair(x[2], x[3], bb.z, bb.w));
            }
            *reinterpret_cast<uint4 *>(rowp + (((4 * half + ch) ^ (row & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
          }
        }
        // the generic-proxy stores become visible to the tensor core's reads
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;");
        warp_arrive(&bar_h[t]);
      }
      if (!ok) break;
      acc_ready();
      if (!ok) break;
      // the output layer: 32 rows of 128 bytes per warp, through its 4 KB of the
      // operand buffer so that eight lanes store a row's 128 bytes
      uint32_t r[32];
      tmem_ld16_nowait(acc, r);
      tmem_ld16_nowait(acc + 16u, r + 16);
      tmem_wait32(r);
      const float4 *bo = reinterpret_cast<const float4 *>(b4 + 32 * half);
      char *buf = H + (warp & 7) * 4096;
#pragma unroll
      for (int ch = 0; ch < 8; ++ch) {
        const float4 bb = __ldg(bo + ch);
        *reinterpret_cast<float4 *>(buf + lane * 128 + ((ch ^ (lane & 7)) << 4)) =
            make_float4(__uint_as_float(r[4 * ch]) + bb.x, __uint_as_float(r[4 * ch + 1]) + bb.y,
                        __uint_as_float(r[4 * ch + 2]) + bb.z, __uint_as_float(r[4 * ch + 3]) + bb.w);
      }
      __syncwarp();
      float4 *o = reinterpret_cast<float4 *>(Y + ((size_t)tile_of(i) * kTM + quarter * 32) * 64 + 32 * half);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int rr = 4 * k + (lane >> 3), ch = lane & 7;
        o[rr * 16 + ch] = *reinterpret_cast<const float4 *>(buf + rr * 128 + ((ch ^ (rr & 7)) << 4));
      }
      // the accumulator and this warp's part of the buffer, which the other
      // warps' next layer overwrites, have been read
      asm volatile("tcgen05.fence::before_thread_sync;");
      warp_arrive(&bar_h[t]);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (tid == 0 && *fail) atomicExch(err, 1);
  if (warp == 16)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
}

namespace {

// ---- weight gradients: dW_l = dZ_l^T A_(l-1) over the batch, all layers in
// one launch.  A CTA takes 128 rows of one layer's dW (for the output layer,
// whose 64 rows are too few, of its transpose) and a share of the batch, 64
// batch rows per stage: both operands are [batch][width] arrays whose width is
// the MMA's M or N, so the descriptors are MN-major (64-wide boxes with the
// 128-byte swizzle: 8 batch rows of 128 bytes per swizzle group, the boxes
// 8 KB apart).  The tensor core truncates as it accumulates: sums of one sign
// over 2700 rows in one chain were off by 4e-7 of their size, over 11000 by
// 5e-6.  So a chain ends after kGSeg stages (512 rows), and eight epilogue warps add it to
// the sums in their registers (FP32, rounded to nearest) while the next one
// fills the other half of the tensor memory; they also sum the hidden biases'
// gradients, the columns of dZ, from the stages (errors now 1e-7 whatever the
// batch).  Bound by the loads and the chain of a share (ten stages at 16384 rows,
// 19 us against 17 in one chain: the bias sums read the stages beside the MMAs;
// chains of 12 stages take the same time, and draining a chain in quarters
// between the stages spilled registers and took 21).  Partials per share, summed
// in a fixed order by k_mlp_update.
constexpr int kGStages = 4;
constexpr int kGSeg = 8;                        // stages of a chain
constexpr int kGWarps = 8;                      // epilogue warps; then the MMA and the TMA warp
constexpr int kGThreads = 32 * (kGWarps + 2);
constexpr int kGBox = 64 * 128;                 // bytes of a 64 x 64 box
constexpr int kGStageBytes = 6 * kGBox;         // 2 boxes of M, up to 4 of N
constexpr int kGOffBar = kGStages * kGStageBytes;
constexpr int kGBars = 2 * kGStages + 5;
constexpr int kSmemGrad = kGOffBar + 8 * kGBars + 16 + 1024;
static_assert(kSmemGrad <= 224 * 1024, "shared memory of the weight-gradient kernel");

struct GradMaps {
  CUtensorMap m[4], n[4];  // per layer: the operand along M, along N
};

__host__ __device__ constexpr uint32_t make_idesc_mn(int M, int N) {  // both operands MN-major
  return tc::make_idesc(M, N) | (1u << 15) | (1u << 16);
}

__global__ void __launch_bounds__(kGThreads, 1)
    k_mlp_wgrad(const __grid_constant__ GradMaps maps, int nkb, int s_small, int s_big, float *part, int *err) {
  using namespace tc;
  extern __shared__ char smem_raw[];
  char *smem = reinterpret_cast<char *>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ float bsum[4][128];  // the bias sums of each quarter of the stages' rows
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint64_t *bar = reinterpret_cast<uint64_t *>(smem + kGOffBar);
  // stages full and free; per half of the tensor memory: chain complete, read
  uint64_t *bar_full = bar, *bar_free = bar + kGStages, *bar_acc = bar + 2 * kGStages, *bar_read = bar_acc + 2;
  uint64_t *bar_end = bar_acc + 4;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bar + kGBars);
  volatile int *fail = reinterpret_cast<volatile int *>(tmem_slot + 1);
  // block -> layer, row tile, share z of S
  int u = blockIdx.x, l = 0;
  int S = s_small;
  while (u >= 2 * S) {
    u -= 2 * S;
    ++l;
    S = l == 0 || l == 3 ? s_small : s_big;
  }
  const int mt = u & 1, z = u >> 1;
  const int N = l == 0 || l == 3 ? 64 : 256;
  const int k0 = (int)((int64_t)nkb * z / S), k1 = (int)((int64_t)nkb * (z + 1) / S);
  const bool bias = l < 3;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(512u));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int i = 0; i < kGStages; ++i) {
      mbar_init(&bar_full[i], 1);
      mbar_init(&bar_free[i], bias ? 1 + kGWarps : 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bar_acc[i], 1);
      mbar_init(&bar_read[i], kGWarps);
    }
    mbar_init(bar_end, 1);
    *fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = *tmem_slot;
  float *out = part + mlp_part_offset(l, s_small, s_big) + (size_t)z * mlp_part_size(l);
  if (warp == kGWarps + 1) {
    // ---- TMA loads
    if (lane == 0) {
      bool ok = true;
      int g = 0;
      for (int k = k0; k < k1; ++k, ++g) {
        const int s = g % kGStages;
        if (g >= kGStages && !(ok = wait_on(&bar_free[s], (uint32_t)((g / kGStages - 1) & 1), fail))) break;
        char *st = smem + s * kGStageBytes;
        mbar_expect_tx(&bar_full[s], (uint32_t)((2 + N / 64) * kGBox));
        for (int b = 0; b < 2; ++b) tma_load_2d(st + b * kGBox, &maps.m[l], 128 * mt + 64 * b, 64 * k, &bar_full[s]);
        for (int b = 0; b < N / 64; ++b) tma_load_2d(st + (2 + b) * kGBox, &maps.n[l], 64 * b, 64 * k, &bar_full[s]);
      }
      if (!ok || *fail)
        for (int k = g > kGStages ? g - kGStages : 0; k < g; ++k)
          mbar_wait(&bar_full[k % kGStages], (uint32_t)((k / kGStages) & 1));
    }
  } else if (warp == kGWarps) {
    // ---- MMAs, by one lane
    if (lane == 0) {
      bool ok = true;
      for (int g = 0; g < k1 - k0 && ok; ++g) {
        const int s = g % kGStages, seg = g / kGSeg, first = g % kGSeg == 0;
        if (first && seg > 1 && !(ok = wait_on(&bar_read[seg & 1], (uint32_t)((seg / 2 - 1) & 1), fail))) break;
        if (!(ok = wait_on(&bar_full[s], (uint32_t)((g / kGStages) & 1), fail))) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
        const uint32_t a0 = smem_u32(smem + s * kGStageBytes), b0 = a0 + 2 * kGBox;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)  // 16 batch rows: two swizzle groups of 1024 bytes
          mma_bf16(tmem + 256u * (uint32_t)(seg & 1), make_desc(a0 + 2048 * kk, kGBox, 1024, kSwizzle128B),
                   make_desc(b0 + 2048 * kk, kGBox, 1024, kSwizzle128B), make_idesc_mn(128, N),
                   first && kk == 0 ? 0u : 1u);
        mma_commit(&bar_free[s]);
        if (g % kGSeg == kGSeg - 1 || g + 1 == k1 - k0) mma_commit(&bar_acc[seg & 1]);
      }
      if (!ok || *fail) {  // every MMA issued is done before the tensor memory is freed
        mma_commit(bar_end);
        mbar_wait(bar_end, 0);
      }
    }
  } else {
    // ---- epilogues: warp w has accumulator lanes 32 (w % 4).. and half w / 4 of the columns
    const int quarter = warp & 3, half = warp >> 2;
    const uint32_t t = tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)(half * (N / 2));
    float acc[4][32];
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int j = 0; j < 32; ++j) acc[c][j] = 0.0f;
    // bias columns 2 pair, 2 pair + 1 of rows 16 rg .. 16 rg + 15 of a stage
    // (a warp reads a row's 128 bytes: no bank conflicts)
    const int pair = tid & 63, rg = tid >> 6;
    const char *bcol = smem + (pair >> 5) * kGBox + 16 * rg * 128 + 4 * (pair & 3);
    const int chunk = (pair & 31) >> 2;
    float b0 = 0.0f, b1 = 0.0f;
    bool ok = true;
    for (int g0 = 0, seg = 0; g0 < k1 - k0; g0 += kGSeg, ++seg) {
      if (bias)
        for (int g = g0; g < min(g0 + kGSeg, k1 - k0) && ok; ++g) {
          const int s = g % kGStages;
          ok = wait_warp(&bar_full[s], (uint32_t)((g / kGStages) & 1), fail);
          if (!ok) break;
          float s0 = 0.0f, s1 = 0.0f;
#pragma unroll
          for (int i0 = 0; i0 < 16; i0 += 8) {  // (eight words in registers beside the sums)
            uint32_t x[8];
#pragma unroll
            for (int i = 0; i < 8; ++i)
              x[i] = *reinterpret_cast<const uint32_t *>(bcol + s * kGStageBytes + (i0 + i) * 128 + ((chunk ^ i) << 4));
            if (i0 == 8) warp_arrive(&bar_free[s]);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              s0 += __uint_as_float(x[i] << 16);
              s1 += __uint_as_float(x[i] & 0xFFFF0000u);
            }
          }
          b0 += s0;
          b1 += s1;
        }
      ok = ok && wait_warp(&bar_acc[seg & 1], (uint32_t)((seg / 2) & 1), fail);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if (32 * c >= N / 2) break;  // uniform
        uint32_t r[32];
        const uint32_t tc0 = t + 256u * (uint32_t)(seg & 1) + 32u * (uint32_t)c;
        tmem_ld16_nowait(tc0, r);
        tmem_ld16_nowait(tc0 + 16u, r + 16);
        tmem_wait32(r);
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[c][j] += __uint_as_float(r[j]);
      }
      asm volatile("tcgen05.fence::before_thread_sync;");
      warp_arrive(&bar_read[seg & 1]);
    }
    // partial: [256 or 64 rows][N] of the layer, then its 256 bias sums
    if (ok) {
      float4 *o = reinterpret_cast<float4 *>(out + (size_t)(128 * mt + 32 * quarter + lane) * N + half * (N / 2));
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if (32 * c >= N / 2) break;
#pragma unroll
        for (int j = 0; j < 8; ++j)
          o[8 * c + j] = make_float4(acc[c][4 * j], acc[c][4 * j + 1], acc[c][4 * j + 2], acc[c][4 * j + 3]);
      }
    }
    bsum[rg][2 * pair] = b0;
    bsum[rg][2 * pair + 1] = b1;
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (bias && tid < 128) out[(size_t)256 * N + 128 * mt + tid] = (bsum[0][tid] + bsum[1][tid]) + (bsum[2][tid] + bsum[3][tid]);
  if (tid == 0 && *fail) atomicExch(err, 1);
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u));
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

// Row-major [rows][cols] bf16 matrix, boxes of 64 columns x box_rows rows,
// 128-byte swizzle.
bool encode(CUtensorMap *m, const void *base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  auto fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {cols, rows};
  const cuuint64_t strides[1] = {cols * 2};
  const cuuint32_t box[2] = {64, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box,
            estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int device_sms() {
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

bool encode_forward(FusedMaps &t, int M, const void *X, const void *const W[4]) {
  return encode(&t.x, X, (uint64_t)M, 64, kTM) && encode(&t.w1, W[0], 256, 64, 256) &&
         encode(&t.w2, W[1], 256, 256, 256) && encode(&t.w3, W[2], 256, 256, 256) &&
         encode(&t.w4, W[3], 64, 256, 64);
}

}  // namespace

// Y [M][64] fp32 = the network on X [M][64] bf16; W[l] the bf16 weights
// [out][in] (256 x 64, 256 x 256, 256 x 256, 64 x 256), b[l] the fp32
// biases.  M % 128 == 0, every pointer 16-byte aligned.  err: device int set
// to 1 on a barrier timeout.
cudaError_t launch_mlp_fused(int M, const void *X, const void *const W[4], const float *const b[4],
                             float *Y, int *err, cudaStream_t st) {
  InferMaps t{};
  if (!(encode(&t.x, X, (uint64_t)M, 64, kTM) && encode(&t.w1, W[0], 256, 64, 256) &&
        encode(&t.w2, W[1], 256, 256, 256) && encode(&t.w3, W[2], 256, 256, 256) && encode(&t.w4, W[3], 64, 256, 64)))
    return cudaErrorInvalidValue;
  const int ntiles = M / kTM, grid = std::min(ntiles, device_sms());
  if (grid == 0) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(k_mlp_infer, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemInfer);
  if (e != cudaSuccess) return e;
  k_mlp_infer<<<grid, kThreadsF, kSmemInfer, st>>>(t, b[0], b[1], b[2], b[3], Y, ntiles, err);
  return cudaGetLastError();
}

MlpTrainShape mlp_train_shape(int M) {
  MlpTrainShape s;
  const int sms = device_sms(), nkb = M / 64;
  s.ctas = std::min(M / kTM, sms);
  // shares of the batch: the hidden layers' products load three times the
  // bytes of the first and last layer's, all CTAs together one per SM
  s.s_small = std::max(1, std::min(nkb, sms / 12));
  s.s_big = std::max(1, std::min(nkb, sms / 6));
  return s;
}

// One pass of the training kernels: activations and gradients into `act`
// [3][M][256], `dz` [3][M][256] and `dy` [M][64] (bf16), the loss added to
// *loss, partial weight gradients into `part` and the output bias's into
// `gb4`.
cudaError_t launch_mlp_train(int M, const void *X, const float *target, int n_valid, const void *const W[4],
                             const void *const Wt[4], const float *const b[4], void *const act[3],
                             void *const dz[3], void *dy, double *loss, float *part, float *gb4, int *err,
                             cudaStream_t st) {
  FusedMaps t{};
  GradMaps g{};
  bool ok = encode_forward(t, M, X, W) && encode(&t.t4, Wt[3], 256, 64, 256) &&
            encode(&t.t3, Wt[2], 256, 256, 256) && encode(&t.t2, Wt[1], 256, 256, 256) &&
            encode(&t.dy, dy, (uint64_t)M, 64, kTM);
  for (int l = 0; l < 3 && ok; ++l)
    ok = encode(&t.a[l], act[l], (uint64_t)M, 256, kTM) && encode(&t.d[l], dz[l], (uint64_t)M, 256, kTM) &&
         encode(&g.m[l], dz[l], (uint64_t)M, 256, 64) &&
         (l == 0 ? encode(&g.n[0], X, (uint64_t)M, 64, 64) : encode(&g.n[l], act[l - 1], (uint64_t)M, 256, 64));
  ok = ok && encode(&g.m[3], act[2], (uint64_t)M, 256, 64) && encode(&g.n[3], dy, (uint64_t)M, 64, 64);
  if (!ok) return cudaErrorInvalidValue;
  const MlpTrainShape s = mlp_train_shape(M);
  cudaError_t e =
      cudaFuncSetAttribute(k_mlp_fused, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemFused);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_mlp_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemGrad);
  if (e != cudaSuccess) return e;
  const TrainArgs ta{target, n_valid, (float)(M * n_valid), (double)(M * n_valid), loss, gb4};
  k_mlp_fused<<<s.ctas, kThreadsF, kSmemFused, st>>>(t, b[0], b[1], b[2], b[3], M / kTM, err, ta);
  k_mlp_wgrad<<<4 * (s.s_small + s.s_big), kGThreads, kSmemGrad, st>>>(g, M / 64, s.s_small, s.s_big, part, err);
  return cudaGetLastError();
}

}  // namespace dm
