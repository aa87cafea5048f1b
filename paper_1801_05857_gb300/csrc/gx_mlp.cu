// The scoring network of the guided deadlock search (no counterpart in the
// paper): a small MLP that predicts a state's distance to the nearest deadlock
// from the histogram of its processes' local states.
//
//   x  = bf16(hist / n)                 (hist[i] = processes in local state i, i < 16;
//                                        n = sum of hist = the network's processes)
//   h1 = bf16(relu(W1 x + b1))          W1: 128 x 16
//   h2 = relu(W2 h1 + b2)               W2: 128 x 128
//   y  = w3 . h2 + b3
//
// The one-hot local state of each process, averaged over processes, is the
// input: the first layer's weights are shared by all processes, and the
// input has the same scale at every network size, which is what lets a
// network trained on small instances score states of larger ones.
// Weights are used in BF16 (rounded to nearest even from FP32 master copies
// that the optimiser updates), and so is each layer's input (x and h1 are
// rounded from FP32), so that both layers are BF16 x BF16 products with
// FP32 accumulation -- the operand types of the tensor cores.  Inference
// (gx_mlp_forward, and the guided search's scoring) and the gradient
// (gx_mlp_grad, gx_mlp_train: grad_tc_kernel below) run on the tensor cores
// (gx_tc.cuh).
//
// Parameter vector (FP32, GX_MLP_PARAMS floats): W1 | b1 | W2 | b2 | w3 | b3.
// Loss: mean over the batch of (y - label)^2.

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include <cuda_bf16.h>

#include "gx_kernels.h"
#include "gx_tc.cuh"

namespace gxm {

constexpr int IN = GX_MLP_IN;
constexpr int H = GX_MLP_HIDDEN;
constexpr int OFF_W1 = 0;
constexpr int OFF_B1 = OFF_W1 + H * IN;
constexpr int OFF_W2 = OFF_B1 + H;
constexpr int OFF_B2 = OFF_W2 + H * H;
constexpr int OFF_W3 = OFF_B2 + H;
constexpr int OFF_B3 = OFF_W3 + H;
constexpr int NPARAM = OFF_B3 + 1;
static_assert(NPARAM == GX_MLP_PARAMS, "parameter count");
constexpr int kGradCtas = GX_MLP_GRAD_CTAS;  // at most this many CTAs, one partial gradient each

// A partial gradient holds W1 and W2 transposed (a column of 128 hidden units
// after the other), as a gradient CTA's threads, one hidden unit each, write them
// in whole lines.
constexpr int kPartial = NPARAM;

// The parameter that element q of a partial gradient belongs to.
__device__ __forceinline__ int partial_param(int q) {
  if (q < OFF_B1) return OFF_W1 + (q % H) * IN + q / H;
  if (q >= OFF_W2 && q < OFF_B2) return OFF_W2 + ((q - OFF_W2) % H) * H + (q - OFF_W2) / H;
  return q;
}

// Element q of the gradient: the sum over the CTAs c, in order, of partial[c][q].
__device__ __forceinline__ float partial_sum(const float* __restrict__ partial, int ctas, int q) {
  float acc = 0.f;
#pragma unroll 8
  for (int c = 0; c < ctas; ++c) acc += partial[(uint64_t)c * kPartial + q];
  return acc;
}

__global__ void reduce_kernel(const float* __restrict__ partial, const float* __restrict__ partial_loss, int ctas,
                              float* __restrict__ g, float* __restrict__ loss) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < NPARAM) g[partial_param(q)] = partial_sum(partial, ctas, q);
  if (q == 0) {
    float l = 0.f;
    for (int c = 0; c < ctas; ++c) l += partial_loss[c];
    *loss = l;
  }
}

// Inference on the tensor cores (gxt::score_tiles).
__device__ unsigned int g_tc_error;
// The weights gx_mlp_forward scores with, packed for the tensor cores (one
// copy per device; calls hold g_forward_mutex from packing to completion), and
// the biases and output weights in constant memory, where they are operands of the
// arithmetic.
__device__ gxt::ScoreWeights g_tc_packed;
struct __align__(16) FwdConst {
  float b1[H], b2[H], w3[H], b3, pad[3];
};
__constant__ FwdConst c_fwd;
static_assert(sizeof(FwdConst) == sizeof(gxt::TcWeights) - offsetof(gxt::TcWeights, b1), "the packed weights' tail");
struct ConstPar {
  __device__ __forceinline__ unsigned long long b1(int k) const {
    return *reinterpret_cast<const unsigned long long*>(&c_fwd.b1[k]);
  }
  __device__ __forceinline__ unsigned long long w3(int k) const {
    return *reinterpret_cast<const unsigned long long*>(&c_fwd.w3[k]);
  }
  __device__ __forceinline__ float b3() const { return c_fwd.b3; }
};

// The first kernel of a call: packs the parameters and clears the error flag.
__global__ void score_pack_kernel(const float* __restrict__ p) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) g_tc_error = 0;
  if (i < gxt::kScorePackItems) gxt::score_pack_item(p, &g_tc_packed, i);
}

// 4,000,037 examples: 182 us (bytes alone 12 us, products alone 78 us at the
// measured BF16 rate), where one CTA per tile and 16-byte reads of the biases from
// shared memory took 350 us.
__global__ void __launch_bounds__(gxt::kScoreThreads, 1)
    mlp_tc_forward_kernel(const gxt::ScoreWeights* __restrict__ packed, const uint8_t* __restrict__ hist, uint64_t n,
                          float* __restrict__ out) {
  extern __shared__ __align__(16) uint8_t tsm[];
  const bool aligned = (reinterpret_cast<uintptr_t>(hist) & 15) == 0;
  const bool ok = gxt::score_tiles(
      tsm, packed, n,
      [&](uint64_t row, uint32_t (&hw)[4]) {
        const uint8_t* src = hist + row * IN;
        if (aligned) {
          const uint4 q = __ldcs(reinterpret_cast<const uint4*>(src));
          hw[0] = q.x;
          hw[1] = q.y;
          hw[2] = q.z;
          hw[3] = q.w;
        } else {
#pragma unroll
          for (int i = 0; i < IN; ++i) hw[i >> 2] |= (uint32_t)src[i] << ((i & 3) * 8);
        }
      },
      [&](uint64_t row, float y) { out[row] = y; },
      [](const gxt::TcWeights&) { return ConstPar{}; });
  if (!ok) atomicOr(&g_tc_error, 1u);
}

// ---- Gradient on the tensor cores.  One CTA of 512 threads per tile of 128
// examples, all of TMEM (512 columns) per CTA.  Every product is a tcgen05
// BF16 x BF16 -> FP32 MMA on operands in shared memory:
//   A1  = X W1^T,  H = bf16(relu(A1 + b1))              (forward, as the scorer)
//   A2  = H W2^T,  y = b3 + w3 . relu(A2 + b2)
//   dy  = 2 (y - label) / n,  D2 = dy w3^T o (A2 + b2 > 0)
//   DH  = D2 W2                                          [128 x 128]
//   [gW2 | gb2] += D2^T [H | 1]                          N = 128 + 16 (ones columns)
//   DA1 = DH o (A1 + b1 > 0)
//   [gW1 | gb1] += DA1^T [X | 1]                         N = 16 + 16
// X, H, D2 and DA1 are written once, an example's row as 16-byte pieces of 8
// elements; the products that take them transposed read the same memory as
// MN-major operands (a core matrix of 8 examples x 8 elements is either a K-major
// piece of the matrix or an MN-major piece of its transpose).
//
// A step's time is a chain of latencies -- loads, five products, the epilogues
// between them -- so the epilogues are spread over 16 warps: warp w owns rows 32 (w
// & 3).. (its TMEM lanes) and columns 32 (w >> 2)... The dot product y keeps its
// order of additions: the four column groups add to it one after the other.
// Step of 1024 examples (8 tiles): 12.4 us a step; with 4 warps, transposed copies of
// the operands and sampling, packing, reduction and Adam in launches of their
// own 42 us.
//
// The gradients accumulate in TMEM over the CTA's tiles, in tile order; gw3 and
// gb3 are summed on the CUDA cores (a fixed butterfly over each warp's lanes,
// then the warps in order), so a CTA's partial gradient does not depend on
// scheduling.  D2 and DA1 enter their products rounded to BF16.
constexpr int kGradThreads = 512;
constexpr uint32_t kTrainCols = 512;
constexpr uint32_t kColAcc = 0, kColDH = 128, kColGW2 = 256, kColGW1 = 400;
// K groups (8 elements) of an example's row: X and 16 ones; H and 16 ones; D2, DA1
constexpr uint32_t kGroupsX = 4, kGroupsH = 18, kGroupsD = 16;
// instruction descriptors: M = 128 with N = 128 (K-major operands), 144 ([H | 1]) and 32 ([X | 1], both MN-major)
constexpr uint32_t kI128 = gxt::idesc_bf16_f32(128, 128), kI144t = gxt::idesc_bf16_f32(128, 144, 1, 1),
                   kI32t = gxt::idesc_bf16_f32(128, 32, 1, 1);

// The parameters as a training CTA holds them: the scorer's image plus W2
// transposed (the B operand of DH = D2 W2: rows j, K = k).
struct __align__(16) TcTrainWeights {
  gxt::TcWeights fw;
  uint8_t w2t[H * H * 2];
};
static_assert(sizeof(TcTrainWeights) % 16 == 0, "bulk copies move multiples of 16 bytes");

struct __align__(1024) TrainSmem {
  uint8_t x[gxt::kRows * kGroupsX * 16];   // [X | 1]
  uint8_t h[gxt::kRows * kGroupsH * 16];   // [H | 1]
  uint8_t d[gxt::kRows * kGroupsD * 16];   // D2
  uint8_t da[gxt::kRows * kGroupsD * 16];  // DA1
  TcTrainWeights wt;
  float y[gxt::kRows];
  float lab[gxt::kRows];
  float red[4][H];                     // per row group: sums of the gw3 terms
  float redl[4][2];                    // per row group: loss and gb3
  uint32_t tmem_slot;
  unsigned long long mbar, mbar_load[3];  // products; W1 and biases, W2, W2^T
};
constexpr size_t kTrainSmemBytes = sizeof(TrainSmem) + 1024;  // + alignment slack
static_assert(kTrainSmemBytes <= 232448, "a training CTA must fit the SM's shared memory");

__device__ unsigned int g_train_error;  // a bounded wait gave up (GX_ERR_SPIN_LIMIT)

// The first kernel of a call: clears the error flag (under the call's lock, like all that
// reads or sets it) and packs the parameters.  W2^T in the core-matrix layout: item (row j,
// K group g) packs W2[8g .. 8g+7][j].
constexpr int kTrainPackItems = gxt::kTcPackItems + H * 16;
__global__ void train_pack_kernel(const float* __restrict__ p, TcTrainWeights* __restrict__ out) {
  if (blockIdx.x == 0 && threadIdx.x == 0) g_train_error = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < kTrainPackItems; i += gridDim.x * blockDim.x) {
    if (i < gxt::kTcPackItems) {
      gxt::tc_pack_item(p, &out->fw, i);
      continue;
    }
    const int item = i - gxt::kTcPackItems, j = item >> 4, g = item & 15;
    const float* c = p + OFF_W2 + (g * 8) * H + j;  // W2[8g][j], stride H down the column
    uint4 q;
    q.x = gxt::pack_bf16x2(c[0 * H], c[1 * H]);
    q.y = gxt::pack_bf16x2(c[2 * H], c[3 * H]);
    q.z = gxt::pack_bf16x2(c[4 * H], c[5 * H]);
    q.w = gxt::pack_bf16x2(c[6 * H], c[7 * H]);
    *reinterpret_cast<uint4*>(out->w2t + gxt::core_offset(j, g * 8, 16)) = q;
  }
}
constexpr int kTrainPackBlocks = (kTrainPackItems + 255) / 256;

__device__ __forceinline__ void st_bf16(uint8_t* base, uint32_t off, float v) {
  *reinterpret_cast<__nv_bfloat16*>(base + off) = __float2bfloat16_rn(v);
}

// Programmatic dependent launch: wait for the kernel in front (and its writes) to
// complete; let the next kernel start.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dependency_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Two warps meet at named barrier `id`.
__device__ __forceinline__ void pair_sync(int id) { asm volatile("barrier.sync %0, 64;" ::"r"(id) : "memory"); }

// Sum of v over the warp's 32 lanes for 32 columns at once, in a fixed order
// (recursive halving: at step h the lanes with bit h set keep the upper half of
// their columns), so lane l ends with the sum of column l.
__device__ __forceinline__ float warp_column_sums(float (&v)[32]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int half = 16; half >= 1; half >>= 1) {
    const bool up = (lane & half) != 0;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const float send = up ? v[i] : v[i + half];
      const float keep = up ? v[i + half] : v[i];
      v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, half);
    }
  }
  return v[0];
}

// The weights a gradient is taken at, packed for the tensor cores (one copy per
// device; calls hold g_train_mutex from packing to completion).
__device__ TcTrainWeights g_train_packed;

// Mini-batch drawn by a counter-based stream: element j is example
// mix64(start + j) mod n of the training set.
struct Draw {
  uint64_t n, start;
  int on;
};

// CTA c takes tiles c, c + gridDim.x, ... of the n examples and writes its partial
// gradient of the mean loss (inv_n = 1 / n) to partial[c], its loss to
// partial_loss[c].
__global__ void __launch_bounds__(kGradThreads, 1)
    grad_tc_kernel(const TcTrainWeights* __restrict__ packed, const uint8_t* __restrict__ hist,
                   const float* __restrict__ label, uint64_t n, const Draw draw, float inv_n,
                   float* __restrict__ partial, float* __restrict__ partial_loss) {
  extern __shared__ __align__(16) uint8_t gsm[];
  TrainSmem* s = reinterpret_cast<TrainSmem*>((reinterpret_cast<uintptr_t>(gsm) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int rg = wid & 3, c = wid >> 2;  // row group (TMEM lanes), column group
  const int t = 32 * rg + lane;          // example of the tile
  const uint64_t tiles = (n + gxt::kRows - 1) / gxt::kRows;
  if (blockIdx.x >= tiles) return;
  using namespace gxt;
  if (tid == 0) {
    mbar_init(saddr(&s->mbar), 1);
    for (int i = 0; i < 3; ++i) mbar_init(saddr(&s->mbar_load[i]), 1);
  }
  if (wid == 0) {
    __syncwarp();
    tmem_alloc(saddr(&s->tmem_slot), kTrainCols);
    tmem_relinquish();
  }
  // the ones columns of [X | 1] and [H | 1] (their products give the bias gradients)
  if (c >= 2) {
    constexpr uint32_t kOnes = 0x3F803F80u;  // two BF16 ones
    const uint4 ones = make_uint4(kOnes, kOnes, kOnes, kOnes);
    uint8_t* base = c == 2 ? s->x : s->h;
    const uint32_t k0 = c == 2 ? IN : H, kg = c == 2 ? kGroupsX : kGroupsH;
    *reinterpret_cast<uint4*>(base + core_offset(t, k0, kg)) = ones;
    *reinterpret_cast<uint4*>(base + core_offset(t, k0 + 8, kg)) = ones;
  }
  // X = bf16(hist / processes) and the labels of a tile, by the first column group
  auto fill_x = [&](uint64_t tile) {
    if (c != 0) return;
    const uint64_t row = tile * kRows + t;
    const bool valid = row < n;
    uint64_t ex = row;
    if (draw.on) {
      uint64_t z = draw.start + row + 0x9E3779B97F4A7C15ull;
      z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
      z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
      ex = (z ^ (z >> 31)) % draw.n;
    }
    uint32_t hw[4] = {0, 0, 0, 0};
    if (valid) {
      const uint8_t* src = hist + ex * IN;
      if ((reinterpret_cast<uintptr_t>(src) & 15) == 0) {
        const uint4 q = *reinterpret_cast<const uint4*>(src);
        hw[0] = q.x;
        hw[1] = q.y;
        hw[2] = q.z;
        hw[3] = q.w;
      } else {
#pragma unroll
        for (int i = 0; i < IN; ++i) hw[i >> 2] |= (uint32_t)src[i] << ((i & 3) * 8);
      }
    }
    s->lab[t] = valid ? label[ex] : 0.f;
    const float inv = feature_scale(hw);
    uint32_t q[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t w = hw[i >> 1], sh = (i & 1) * 16;
      q[i] = pack_bf16x2((float)((w >> sh) & 0xFFu) * inv, (float)((w >> (sh + 8)) & 0xFFu) * inv);
    }
    *reinterpret_cast<uint4*>(s->x + core_offset(t, 0, kGroupsX)) = make_uint4(q[0], q[1], q[2], q[3]);
    *reinterpret_cast<uint4*>(s->x + core_offset(t, 8, kGroupsX)) = make_uint4(q[4], q[5], q[6], q[7]);
  };
  fill_x(blockIdx.x);
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // everything so far needs nothing of the kernel in front; the weights do
  grid_dependency_wait();
  grid_dependency_launch();
  if (tid == 0) {
    const TcWeights* fw = &packed->fw;
    constexpr uint32_t kW1 = sizeof(fw->w1), kW2 = sizeof(fw->w2), kRest = sizeof(TcWeights) - kW1 - kW2;
    mbar_expect_tx(saddr(&s->mbar_load[0]), kW1 + kRest);
    bulk_g2s(saddr(&s->wt.fw.w1), fw->w1, kW1, saddr(&s->mbar_load[0]));
    bulk_g2s(saddr(&s->wt.fw.b1), fw->b1, kRest, saddr(&s->mbar_load[0]));
    mbar_expect_tx(saddr(&s->mbar_load[1]), kW2);
    bulk_g2s(saddr(&s->wt.fw.w2), fw->w2, kW2, saddr(&s->mbar_load[1]));
    mbar_expect_tx(saddr(&s->mbar_load[2]), (uint32_t)sizeof(packed->w2t));
    bulk_g2s(saddr(&s->wt.w2t), packed->w2t, (uint32_t)sizeof(packed->w2t), saddr(&s->mbar_load[2]));
  }
  const uint32_t tm = s->tmem_slot, lb = (uint32_t)(32 * rg) << 16;
  uint32_t phase = 0;
  // one commit, then every thread waits; false when any thread gave up
  auto commit_wait = [&]() -> bool {
    if (tid == 0) mma_commit(saddr(&s->mbar));
    const bool w = mbar_wait_bounded(saddr(&s->mbar), phase);
    phase ^= 1u;
    const int bad = __syncthreads_or(!w);
    tc_fence_after();
    return bad == 0;
  };
  // the copies must land before the CTA leaves, so each is waited for, twice if need be
  auto load_wait = [&](int i) -> bool {
    bool w = mbar_wait_bounded(saddr(&s->mbar_load[i]), 0);
    if (!w) w = mbar_wait_bounded(saddr(&s->mbar_load[i]), 0);
    return __syncthreads_or(!w) == 0;
  };
  bool ok = load_wait(0);
  float gw3acc = 0.f, gb3acc = 0.f, lossacc = 0.f;
  uint32_t first = 1;
  int waited = 1;  // weight copies waited for
  const TcWeights& W = s->wt.fw;
  for (uint64_t tile = blockIdx.x; ok && tile < tiles; tile += gridDim.x) {
    if (!first) {
      fill_x(tile);
      fence_async_smem();
      __syncthreads();
    }
    const bool valid = tile * kRows + t < n;
    if (tid == 0) {
      tc_fence_after();
      mma_bf16_i(tm + kColAcc, smem_desc(saddr(s->x), 128, 128 * kGroupsX), smem_desc(saddr(W.w1), 128, 256), kI128, 0u);
    }
    if (!(ok = commit_wait())) break;
    // H = bf16(relu(A1 + b1)); the ReLU's mask of A1 kept for the backward pass
    uint32_t mask1 = 0;
    {
      float a[32];
      tmem_ld32(tm + lb + kColAcc + 32 * c, a);
      uint32_t q[16];
#pragma unroll
      for (int e = 0; e < 32; ++e) {
        a[e] += W.b1[32 * c + e];
        if (a[e] > 0.f) mask1 |= 1u << e;
        a[e] = fmaxf(a[e], 0.f);
      }
#pragma unroll
      for (int e = 0; e < 16; ++e) q[e] = pack_bf16x2(a[2 * e], a[2 * e + 1]);
#pragma unroll
      for (int g = 0; g < 4; ++g)
        *reinterpret_cast<uint4*>(s->h + core_offset(t, 32 * c + 8 * g, kGroupsH)) =
            make_uint4(q[4 * g], q[4 * g + 1], q[4 * g + 2], q[4 * g + 3]);
    }
    tc_fence_before();
    fence_async_smem();
    if (first) {
      ok = load_wait(1);
      waited = 2;
      if (!ok) break;
    } else {
      __syncthreads();
    }
    if (tid == 0) {
      tc_fence_after();
#pragma unroll
      for (uint32_t kk = 0; kk < H / 16; ++kk)
        mma_bf16_i(tm + kColAcc, smem_desc(saddr(s->h) + 256u * kk, 128, 128 * kGroupsH),
                   smem_desc(saddr(W.w2) + 256u * kk, 128, 2048), kI128, kk > 0 ? 1u : 0u);
    }
    if (!(ok = commit_wait())) break;
    // y, then dy, D2 = dy w3 o (A2 + b2 > 0) and the gw3 terms dy relu(A2 + b2)
    float a[32];
    tmem_ld32(tm + lb + kColAcc + 32 * c, a);
#pragma unroll
    for (int e = 0; e < 32; ++e) a[e] += W.b2[32 * c + e];
    {
      float w3[32];
#pragma unroll
      for (int e = 0; e < 32; ++e) w3[e] = W.w3[32 * c + e];
      // the column groups of a row group in order: warp (rg, c) hands y on to (rg, c + 1)
      float y = W.b3;
      if (c > 0) {
        pair_sync(1 + rg * 3 + c - 1);
        y = s->y[t];
      }
#pragma unroll
      for (int e = 0; e < 32; ++e) y += w3[e] * fmaxf(a[e], 0.f);
      s->y[t] = y;
      if (c < 3) pair_sync(1 + rg * 3 + c);
      __syncthreads();
    }
    {
      const float y = s->y[t], lab = s->lab[t];
      const float dy = valid ? 2.f * (y - lab) * inv_n : 0.f;
      if (c == 0) {
        if (valid) lossacc += (y - lab) * (y - lab) * inv_n;
        gb3acc += dy;
      }
      float v[32];
      uint32_t q[16];
#pragma unroll
      for (int e = 0; e < 32; ++e) {
        const float z = a[e];
        v[e] = dy * fmaxf(z, 0.f);
        a[e] = z > 0.f ? dy * W.w3[32 * c + e] : 0.f;
      }
#pragma unroll
      for (int e = 0; e < 16; ++e) q[e] = pack_bf16x2(a[2 * e], a[2 * e + 1]);
#pragma unroll
      for (int g = 0; g < 4; ++g)
        *reinterpret_cast<uint4*>(s->d + core_offset(t, 32 * c + 8 * g, kGroupsD)) =
            make_uint4(q[4 * g], q[4 * g + 1], q[4 * g + 2], q[4 * g + 3]);
      tc_fence_before();
      fence_async_smem();
      if (first) {
        ok = load_wait(2);
        waited = 3;
        if (!ok) break;
      } else {
        __syncthreads();
      }
      if (tid == 0) {
        tc_fence_after();
#pragma unroll
        for (uint32_t kk = 0; kk < H / 16; ++kk)
          mma_bf16_i(tm + kColDH, smem_desc(saddr(s->d) + 256u * kk, 128, 2048),
                     smem_desc(saddr(s->wt.w2t) + 256u * kk, 128, 2048), kI128, kk > 0 ? 1u : 0u);
        mma_commit(saddr(&s->mbar));
        // D2^T [H | 1]: K steps of 16 examples (two rows of core matrices); it runs behind DH's epilogue
#pragma unroll
        for (uint32_t kk = 0; kk < kRows / 16; ++kk)
          mma_bf16_i(tm + kColGW2, smem_desc(saddr(s->d) + 2u * kk * 128 * kGroupsD, 128 * kGroupsD, 128),
                     smem_desc(saddr(s->h) + 2u * kk * 128 * kGroupsH, 128 * kGroupsH, 128), kI144t,
                     (first && kk == 0) ? 0u : 1u);
      }
      gw3acc += warp_column_sums(v);
    }
    {
      const bool w = mbar_wait_bounded(saddr(&s->mbar), phase);
      phase ^= 1u;
      tc_fence_after();
      if (!(ok = __syncthreads_or(!w) == 0)) break;
    }
    // DA1 = DH o (A1 + b1 > 0)
    {
      tmem_ld32(tm + lb + kColDH + 32 * c, a);
      uint32_t q[16];
#pragma unroll
      for (int e = 0; e < 32; ++e) a[e] = ((mask1 >> e) & 1u) ? a[e] : 0.f;
#pragma unroll
      for (int e = 0; e < 16; ++e) q[e] = pack_bf16x2(a[2 * e], a[2 * e + 1]);
#pragma unroll
      for (int g = 0; g < 4; ++g)
        *reinterpret_cast<uint4*>(s->da + core_offset(t, 32 * c + 8 * g, kGroupsD)) =
            make_uint4(q[4 * g], q[4 * g + 1], q[4 * g + 2], q[4 * g + 3]);
    }
    tc_fence_before();
    fence_async_smem();
    __syncthreads();
    if (tid == 0) {
      tc_fence_after();
#pragma unroll
      for (uint32_t kk = 0; kk < kRows / 16; ++kk)
        mma_bf16_i(tm + kColGW1, smem_desc(saddr(s->da) + 2u * kk * 128 * kGroupsD, 128 * kGroupsD, 128),
                   smem_desc(saddr(s->x) + 2u * kk * 128 * kGroupsX, 128 * kGroupsX, 128), kI32t,
                   (first && kk == 0) ? 0u : 1u);
    }
    if (!(ok = commit_wait())) break;
    first = 0;
  }
  while (waited < 3) load_wait(waited++);  // after a wait that gave up
  if (ok) {
    // row t of gW2 and gW1 (hidden unit t), gb2[t], gb1[t]
    float* g = partial + (uint64_t)blockIdx.x * kPartial;
    float a[32];
    tmem_ld32(tm + lb + kColGW2 + 32 * c, a);
#pragma unroll
    for (int e = 0; e < 32; ++e) g[OFF_W2 + (32 * c + e) * H + t] = a[e];
    if (c == 0) {
      tmem_ld32(tm + lb + kColGW1, a);  // columns 400-431: gW1, then gb1 (ones columns)
#pragma unroll
      for (int i = 0; i < IN; ++i) g[OFF_W1 + i * H + t] = a[i];
      g[OFF_B1 + t] = a[IN];
    } else if (c == 1) {
      tmem_ld32(tm + lb + kColGW2 + H, a);  // columns 384-415: gb2 (ones columns), then gW1
      g[OFF_B2 + t] = a[0];
    }
    // gw3 and gb3, loss: the row groups' sums in order
    s->red[rg][32 * c + lane] = gw3acc;
    if (c == 0) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        lossacc += __shfl_xor_sync(0xFFFFFFFFu, lossacc, o);
        gb3acc += __shfl_xor_sync(0xFFFFFFFFu, gb3acc, o);
      }
      if (lane == 0) {
        s->redl[rg][0] = lossacc;
        s->redl[rg][1] = gb3acc;
      }
    }
    __syncthreads();
    if (c == 0) g[OFF_W3 + t] = ((s->red[0][t] + s->red[1][t]) + s->red[2][t]) + s->red[3][t];
    if (tid == 0) {
      g[OFF_B3] = ((s->redl[0][1] + s->redl[1][1]) + s->redl[2][1]) + s->redl[3][1];
      partial_loss[blockIdx.x] = ((s->redl[0][0] + s->redl[1][0]) + s->redl[2][0]) + s->redl[3][0];
    }
  } else if (tid == 0) {
    atomicOr(&g_train_error, 1u);
  }
  tc_fence_before();
  __syncthreads();
  if (wid == 0) {
    tc_fence_after();
    tmem_dealloc(tm, kTrainCols);
  }
}

// Self-test of the bounded wait every tensor-core product is awaited with: one
// warp waits on an mbarrier that nothing arrives on, for `limit` polls, and
// records that it gave up.
__device__ unsigned int g_wait_gave_up;

__global__ void wait_selftest_kernel(uint32_t limit) {
  __shared__ unsigned long long bar;
  if (threadIdx.x == 0) gxt::mbar_init(gxt::saddr(&bar), 1);
  __syncthreads();
  const bool done = gxt::mbar_wait_bounded(gxt::saddr(&bar), 0, limit);
  if (threadIdx.x == 0) g_wait_gave_up = done ? 0u : 1u;
}

// One Adam step (Kingma & Ba 2015) on the FP32 master parameters: a thread per
// parameter sums its partial gradients, updates it and writes it into the packed
// weights that the next step's gradient is taken at.
__global__ void __launch_bounds__(256) update_kernel(const float* __restrict__ partial,
                                                     const float* __restrict__ partial_loss, int ctas,
                                                     float* p, float* m, float* v, float lr, float b1t, float b2t,
                                                     TcTrainWeights* __restrict__ packed, float* __restrict__ loss) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // moments lie as the partial gradients do
  const int i = partial_param(q < NPARAM ? q : 0);
  // (m, v and p too, which the step before wrote: only the wait makes another grid's
  // writes visible, although the gradient in front has waited for that step)
  grid_dependency_wait();
  grid_dependency_launch();
  if (q == 0) {
    float l = 0.f;
    for (int c = 0; c < ctas; ++c) l += partial_loss[c];
    *loss = l;
  }
  if (q >= NPARAM) return;
  const float m0 = m[q], v0 = v[q], p0 = p[i];
  const float gi = partial_sum(partial, ctas, q);
  // (which product is fused with the sum is written out: left to the compiler it has
  // changed with the order of the loads, and the trained bits with it)
  const float mi = __fmaf_rn(0.1f, gi, __fmul_rn(0.9f, m0));
  const float vi = __fmaf_rn(__fmul_rn(0.001f, gi), gi, __fmul_rn(0.999f, v0));
  m[q] = mi;
  v[q] = vi;
  const float x = p0 - lr * (mi / (1.f - b1t)) / (sqrtf(vi / (1.f - b2t)) + 1e-8f);
  p[i] = x;
  gxt::TcWeights& w = packed->fw;
  if (i < OFF_B1) {
    st_bf16(w.w1, gxt::core_offset(i / IN, i % IN, 2), x);
  } else if (i < OFF_W2) {
    w.b1[i - OFF_B1] = x;
  } else if (i < OFF_B2) {
    const int k = (i - OFF_W2) / H, j = (i - OFF_W2) % H;
    st_bf16(w.w2, gxt::core_offset(k, j, 16), x);
    st_bf16(packed->w2t, gxt::core_offset(j, k, 16), x);
  } else if (i < OFF_W3) {
    w.b2[i - OFF_B2] = x;
  } else if (i < OFF_B3) {
    w.w3[i - OFF_W3] = __bfloat162float(__float2bfloat16_rn(x));
  } else {
    w.b3 = x;
  }
}

}  // namespace gxm

namespace {
#define GM_CUDA(call)                                                                       \
  do {                                                                                      \
    cudaError_t e_ = (call);                                                                \
    if (e_ != cudaSuccess)                                                                  \
      return gx::fail(GX_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_));     \
  } while (0)

// Kernel attributes belong to the current device, so they are set on every
// call (a few microseconds) rather than once per process.
gx_status set_forward_smem() {
  GM_CUDA(cudaFuncSetAttribute(gxm::mlp_tc_forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)gxt::kScoreSmemBytes));
  return GX_OK;
}

gx_status set_train_smem() {
  GM_CUDA(cudaFuncSetAttribute(gxm::grad_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)gxm::kTrainSmemBytes));
  return GX_OK;
}
}  // namespace

extern "C" {

gx_status gx_mlp_init(float* params, uint64_t seed, void* stream) {
  gx::clear_error();
  if (!params) return gx::fail(GX_ERR_INVALID, "params is NULL");
  // uniform(-1/sqrt(fan_in), 1/sqrt(fan_in)) from a splitmix64 stream, biases 0
  std::vector<float> h(gxm::NPARAM, 0.f);
  uint64_t s = seed;
  auto next = [&]() {
    s += 0x9E3779B97F4A7C15ull;
    uint64_t z = s;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return (double)(z >> 11) * (1.0 / 9007199254740992.0);  // [0, 1)
  };
  auto fill = [&](int off, int count, int fan_in) {
    const double r = 1.0 / std::sqrt((double)fan_in);
    for (int i = 0; i < count; ++i) h[off + i] = (float)((2.0 * next() - 1.0) * r);
  };
  fill(gxm::OFF_W1, gxm::H * gxm::IN, gxm::IN);
  fill(gxm::OFF_W2, gxm::H * gxm::H, gxm::H);
  fill(gxm::OFF_W3, gxm::H, gxm::H);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  GM_CUDA(cudaMemcpyAsync(params, h.data(), sizeof(float) * h.size(), cudaMemcpyHostToDevice, st));
  GM_CUDA(cudaStreamSynchronize(st));
  return GX_OK;
}

static std::mutex g_forward_mutex;
static std::mutex g_train_mutex;

// The gradient over n examples (drawn from a training set when `draw` is given) at
// the packed weights: one CTA per tile of 128 examples, at most GX_MLP_GRAD_CTAS
// CTAs, each writing its partial gradient.
cudaError_t launch_grad_tc(const uint8_t* hist, const float* label, uint64_t n, gxm::Draw draw, float* partial,
                           float* partial_loss, const gxm::TcTrainWeights* packed, bool overlap, cudaStream_t st) {
  const uint64_t tiles = (n + gxt::kRows - 1) / gxt::kRows;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)std::min<uint64_t>(tiles, gxm::kGradCtas));
  cfg.blockDim = dim3(gxm::kGradThreads);
  cfg.dynamicSmemBytes = gxm::kTrainSmemBytes;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = overlap ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, gxm::grad_tc_kernel, packed, hist, label, n, draw, 1.0f / (float)n, partial,
                            partial_loss);
}

gx_status gx_mlp_forward(const float* params, const uint8_t* hist, uint64_t n, float* out, void* stream) {
  gx::clear_error();
  if (!params || (n && (!hist || !out))) return gx::fail(GX_ERR_INVALID, "NULL device pointer");
  if (n == 0) return GX_OK;
  gx_status s = set_forward_smem();
  if (s != GX_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int dev = 0, sms = 0;
  GM_CUDA(cudaGetDevice(&dev));
  GM_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const uint64_t tiles = (n + gxt::kRows - 1) / gxt::kRows;
  const uint64_t grid = std::min<uint64_t>(tiles, (uint64_t)sms);
  std::lock_guard<std::mutex> lock(g_forward_mutex);
  gxt::ScoreWeights* packed = nullptr;
  GM_CUDA(cudaGetSymbolAddress(reinterpret_cast<void**>(&packed), gxm::g_tc_packed));
  gxm::score_pack_kernel<<<gxt::kScorePackBlocks, 256, 0, st>>>(params);
  GM_CUDA(cudaMemcpyToSymbolAsync(gxm::c_fwd, packed->w.b1, sizeof(gxm::FwdConst), 0, cudaMemcpyDeviceToDevice, st));
  gxm::mlp_tc_forward_kernel<<<(unsigned)grid, gxt::kScoreThreads, gxt::kScoreSmemBytes, st>>>(packed, hist, n, out);
  GM_CUDA(cudaGetLastError());
  unsigned int err = 0;
  GM_CUDA(cudaMemcpyFromSymbolAsync(&err, gxm::g_tc_error, sizeof(err), 0, cudaMemcpyDeviceToHost, st));
  GM_CUDA(cudaStreamSynchronize(st));
  if (err) return gx::fail(GX_ERR_SPIN_LIMIT, "tensor-core scoring timed out waiting for an MMA");
  return GX_OK;
}

gx_status gx_wait_selftest(uint32_t spin_limit, void* stream) {
  gx::clear_error();
  if (spin_limit == 0 || spin_limit > gxt::kSpinLimit)
    return gx::fail(GX_ERR_INVALID, "spin_limit must be 1.." + std::to_string(gxt::kSpinLimit));
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const unsigned int unset = 2u;
  GM_CUDA(cudaMemcpyToSymbolAsync(gxm::g_wait_gave_up, &unset, sizeof(unset), 0, cudaMemcpyHostToDevice, st));
  gxm::wait_selftest_kernel<<<1, 32, 0, st>>>(spin_limit);
  GM_CUDA(cudaGetLastError());
  unsigned int gave_up = 2u;
  GM_CUDA(cudaMemcpyFromSymbolAsync(&gave_up, gxm::g_wait_gave_up, sizeof(gave_up), 0, cudaMemcpyDeviceToHost, st));
  GM_CUDA(cudaStreamSynchronize(st));
  if (gave_up == 1u)
    return gx::fail(GX_ERR_SPIN_LIMIT, "the wait gave up after " + std::to_string(spin_limit) + " polls");
  if (gave_up != 0u) return gx::fail(GX_ERR_CUDA, "the self-test kernel did not report");
  return GX_OK;
}

gx_status gx_mlp_grad(const float* params, const uint8_t* hist, const float* label, uint64_t n,
                      float* grad, float* loss, void* stream) {
  gx::clear_error();
  if (!params || !grad || !loss || (n && (!hist || !label))) return gx::fail(GX_ERR_INVALID, "NULL device pointer");
  if (n == 0) return GX_OK;
  gx_status s = set_train_smem();
  if (s != GX_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int grid = (int)std::min<uint64_t>((n + gxt::kRows - 1) / gxt::kRows, gxm::kGradCtas);
  float* scratch = nullptr;  // one partial gradient and loss per CTA
  GM_CUDA(cudaMallocAsync(reinterpret_cast<void**>(&scratch), sizeof(float) * (uint64_t)grid * (gxm::kPartial + 1), st));
  std::lock_guard<std::mutex> lock(g_train_mutex);
  gxm::TcTrainWeights* packed = nullptr;
  GM_CUDA(cudaGetSymbolAddress(reinterpret_cast<void**>(&packed), gxm::g_train_packed));
  gxm::train_pack_kernel<<<gxm::kTrainPackBlocks, 256, 0, st>>>(params, packed);
  float* scratch_loss = scratch + (uint64_t)grid * gxm::kPartial;
  cudaError_t e = launch_grad_tc(hist, label, n, gxm::Draw{}, scratch, scratch_loss, packed, false, st);
  if (e == cudaSuccess) {
    gxm::reduce_kernel<<<(gxm::NPARAM + 255) / 256, 256, 0, st>>>(scratch, scratch_loss, grid, grad, loss);
    e = cudaGetLastError();
  }
  cudaFreeAsync(scratch, st);
  if (e != cudaSuccess) return gx::fail(GX_ERR_CUDA, std::string("gradient kernels: ") + cudaGetErrorString(e));
  unsigned int err = 0;
  GM_CUDA(cudaMemcpyFromSymbolAsync(&err, gxm::g_train_error, sizeof(err), 0, cudaMemcpyDeviceToHost, st));
  GM_CUDA(cudaStreamSynchronize(st));
  if (err) return gx::fail(GX_ERR_SPIN_LIMIT, "tensor-core gradient timed out waiting for an MMA");
  return GX_OK;
}

gx_status gx_mlp_train(float* params, float* state, const uint8_t* hist, const float* label, uint64_t n,
                       uint32_t batch, uint32_t steps, float lr, uint64_t seed, float* loss, void* stream) {
  gx::clear_error();
  if (!params || !state || !hist || !label || !loss) return gx::fail(GX_ERR_INVALID, "NULL device pointer");
  if (n == 0 || batch == 0) return gx::fail(GX_ERR_INVALID, "empty training set or batch");
  gx_status s = set_train_smem();
  if (s != GX_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // state: m | v | partial losses | partial gradients (up to GX_MLP_GRAD_CTAS of both)
  float* m = state;
  float* v = state + gxm::NPARAM;
  float* partial_loss = state + 2 * gxm::NPARAM;
  float* partial = partial_loss + gxm::kGradCtas;
  GM_CUDA(cudaMemsetAsync(state, 0, sizeof(float) * 2 * gxm::NPARAM, st));
  GM_CUDA(cudaMemsetAsync(loss, 0, sizeof(float) * steps, st));
  std::lock_guard<std::mutex> lock(g_train_mutex);
  gxm::TcTrainWeights* packed = nullptr;
  GM_CUDA(cudaGetSymbolAddress(reinterpret_cast<void**>(&packed), gxm::g_train_packed));
  gxm::train_pack_kernel<<<gxm::kTrainPackBlocks, 256, 0, st>>>(params, packed);
  const int ctas = (int)std::min<uint64_t>(((uint64_t)batch + gxt::kRows - 1) / gxt::kRows, gxm::kGradCtas);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((gxm::NPARAM + 255) / 256);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  double b1t = 1.0, b2t = 1.0;
  for (uint32_t t = 0; t < steps; ++t) {
    b1t *= 0.9;
    b2t *= 0.999;
    // both launches of a step start before the kernel in front of them has ended and wait for it
    // where they need its results (the first step's gradient follows the packing in full order)
    GM_CUDA(launch_grad_tc(hist, label, batch, gxm::Draw{n, seed + (uint64_t)t * batch, 1}, partial, partial_loss,
                           packed, t > 0, st));
    GM_CUDA(cudaLaunchKernelEx(&cfg, gxm::update_kernel, (const float*)partial, (const float*)partial_loss, ctas, params,
                               m, v, lr, (float)b1t, (float)b2t, packed, loss + t));
  }
  GM_CUDA(cudaGetLastError());
  unsigned int err = 0;
  GM_CUDA(cudaMemcpyFromSymbolAsync(&err, gxm::g_train_error, sizeof(err), 0, cudaMemcpyDeviceToHost, st));
  GM_CUDA(cudaStreamSynchronize(st));
  if (err) return gx::fail(GX_ERR_SPIN_LIMIT, "tensor-core gradient timed out waiting for an MMA");
  return GX_OK;
}

}  // extern "C"
