// sg_qnet.cu -- the learned part: dueling Q-network (Sec. 2 "Dueling DQN",
// Sec. 4.3.1 discrete actions), the VEM eps-greedy rollout with the network
// fused into the simulator loop (Sec. 3.1.1, Alg. 1), the device replay ring
// (Alg. 1 step 5, Alg. 2 step 1) and the double-DQN learner with Adam
// (Alg. 2 step 2; appendix hyperparameter table).
//
// Networks (SG_QNET_DUELING): in -> 256 -> 256 -> 6 (value + 5 advantages),
// ReLU, Q = V + A - mean(A); (SG_QNET_PAPER) the paper's in -> 256 -> 128 ->
// 5 with Q the outputs (Sec. 4.3.2).  The kernels run both at the dueling
// shapes: the paper network's 128 second-layer units and 5 outputs sit in
// the first rows of the 256-unit / 6-output storage and every other weight
// and bias stays exactly zero (its pre-activation is 0, so the ReLU mask
// zeroes its gradient and Adam never moves it, and adding its zero products
// leaves the other sums unchanged); only the head differs.  Weights are BF16
// on the tensor cores with FP32 accumulation; FP32 master weights, Adam
// moments and a target copy live on the device.  Flat parameter order inside
// (padded): W1[256][in] b1[256] W2[256][256] b2[256] W3[6][256] b3[6]; the
// C ABI shows each network's own (compact) order.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "sg_device.cuh"
#include "sg_host.h"
#include "sg_mma.cuh"
#include "sg_tc.cuh"
#include "sparrow_gb.h"

using namespace sg;

namespace {

constexpr int kHid = 256;
constexpr int kLdh = kHid + 8;  // padded row of a 256-wide BF16 matrix
constexpr int kOut = 6;
constexpr int kOutPad = 8;
constexpr int kTile = 16;       // envs / samples per CTA = warps per CTA
constexpr int kThreads = kTile * 32;
constexpr uint32_t kStreamSample = 4;
constexpr uint32_t kStreamInit = 5;

// Byte layout of the BF16 weight image (identical in global and shared memory).
struct ImgLayout {
  int n_in, k1, ld1;   // input width, padded to 16, row stride
  int w1, w2, w3, b1, b2, b3, bytes;
  int plain;           // 1: the outputs are the Q-values (the paper's network)
};

ImgLayout img_layout(int n_in, int plain = 0) {
  ImgLayout L;
  L.n_in = n_in;
  L.plain = plain;
  L.k1 = (n_in + 15) / 16 * 16;
  L.ld1 = L.k1 + 8;
  L.w1 = 0;
  L.w2 = L.w1 + kHid * L.ld1 * 2;
  L.w3 = L.w2 + kHid * kLdh * 2;
  L.b1 = L.w3 + kOutPad * kLdh * 2;
  L.b2 = L.b1 + kHid * 4;
  L.b3 = L.b2 + kHid * 4;
  L.bytes = (L.b3 + kOutPad * 4 + 15) / 16 * 16;
  return L;
}

// Offsets of the flat FP32 parameter vector.
struct ParamLayout {
  int w1, b1, w2, b2, w3, b3, total;
};
// Floats per CTA row of the gradient partials: every parameter, the Huber
// sum, padded to a multiple of 4 so that rows start 16-byte aligned.
__host__ __device__ constexpr long long partial_stride(int total) { return (total + 1 + 3) / 4 * 4; }

ParamLayout param_layout(int n_in) {
  ParamLayout P;
  P.w1 = 0;
  P.b1 = P.w1 + kHid * n_in;
  P.w2 = P.b1 + kHid;
  P.b2 = P.w2 + kHid * kHid;
  P.w3 = P.b2 + kHid;
  P.b3 = P.w3 + kOut * kHid;
  P.total = P.b3 + kOut;
  return P;
}

// The paper network's compact parameter index of padded index i, or -1 for a
// padding entry (always zero): W1[256][in] b1[256] W2[128][256] b2[128]
// W3[5][128] b3[5].
constexpr int kPaperH2 = 128;
__host__ __device__ inline int paper_index(int i, const ParamLayout& P, int n_in) {
  if (i < P.w2) return i;  // W1, b1 unchanged
  const int c_w2 = P.w2, c_b2 = c_w2 + kPaperH2 * kHid, c_w3 = c_b2 + kPaperH2, c_b3 = c_w3 + 5 * kPaperH2;
  if (i < P.b2) {
    const int j = i - P.w2, r = j / kHid, k = j % kHid;
    return r < kPaperH2 ? c_w2 + r * kHid + k : -1;
  }
  if (i < P.w3) {
    const int r = i - P.b2;
    return r < kPaperH2 ? c_b2 + r : -1;
  }
  if (i < P.b3) {
    const int j = i - P.w3, o = j / kHid, k = j % kHid;
    return o < 5 && k < kPaperH2 ? c_w3 + o * kPaperH2 + k : -1;
  }
  const int o = i - P.b3;
  return o < 5 ? c_b3 + o : -1;
}
inline int paper_params(int n_in) { return kHid * n_in + kHid + kPaperH2 * kHid + kPaperH2 + 5 * kPaperH2 + 5; }

}  // namespace

// Device view of a replay ring: slot-major SoA, entry e = slot * n_envs + env.
struct ReplayDev {
  float* s;              // [cap][obs_dim]
  float* s2;             // [cap][obs_dim]
  uint8_t* a;            // [cap]
  float* r;              // [cap]
  uint8_t* term;         // [cap] collided or arrived
  unsigned long long* steps;  // vectorized steps recorded so far; behind it the CTA count of replay_advance
  int slots, n_envs, obs_dim;
  unsigned long long inv_full, inv_slots;  // floor((2^64 - 1) / (sampled entries of a full ring, slots))
  int reserve;           // newest slots the learner never samples (an actor may be writing them)
};

struct sg_replay {
  ReplayDev d;
  long long cap = 0;
  int device = 0;
};

struct sg_qnet {
  int n_in = 0;
  int arch = SG_QNET_DUELING;
  int device = 0;
  ImgLayout IL;
  ParamLayout PL;
  float* master = nullptr;  // [P]
  float* target = nullptr;  // [P]
  float* adam_m = nullptr;
  float* adam_v = nullptr;
  uint8_t* img = nullptr;    // online BF16 image
  uint8_t* img_t = nullptr;  // target BF16 image
  unsigned long long* step = nullptr;  // optimiser steps taken (device)
  unsigned* td_fail = nullptr;         // [2] kTdFail* bits of the current TD step, CTAs of its update that are done
  // learner scratch, sized for max_batch
  int max_batch = 0;
  void* frag = nullptr;      // TdFrag of the 16-sample tiles (mma.sync learner)
  int td_clusters = 1;       // clusters of k_td_tile / k_td_tc that fit the device
  int rollout_mt = 0;        // m-tiles per CTA of the fused rollout (0 = choose by waves)
  int lim_rollout = 0;       // CTA caps of the tcgen05 rollout / learner grids (0 = every SM)
  int lim_learner = 0;
  uint8_t* img_tc = nullptr; // the online weights in the tensor cores' shared-memory layout (batched forward)
  uint8_t* img_tc_t = nullptr; // the target weights in the same layout (tcgen05 learner)
  int sms = 0;               // multiprocessors of the device (persistent grids)
};

// --------------------------------------------------------------- kernels

// Image entries from the FP32 parameters: W1/W2/W3 rounded to BF16 into the
// padded layout (pad entries zero), biases copied.
__global__ void k_build_image(const float* __restrict__ th, uint8_t* __restrict__ img, ImgLayout L, ParamLayout P) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  bf16* W1 = reinterpret_cast<bf16*>(img + L.w1);
  bf16* W2 = reinterpret_cast<bf16*>(img + L.w2);
  bf16* W3 = reinterpret_cast<bf16*>(img + L.w3);
  float* b1 = reinterpret_cast<float*>(img + L.b1);
  float* b2 = reinterpret_cast<float*>(img + L.b2);
  float* b3 = reinterpret_cast<float*>(img + L.b3);
  const int n1 = kHid * L.ld1, n2 = kHid * kLdh, n3 = kOutPad * kLdh;
  if (i < n1) {
    const int r = i / L.ld1, k = i % L.ld1;
    W1[i] = __float2bfloat16_rn(k < L.n_in ? th[P.w1 + r * L.n_in + k] : 0.0f);
  } else if (i < n1 + n2) {
    const int j = i - n1, r = j / kLdh, k = j % kLdh;
    W2[j] = __float2bfloat16_rn(k < kHid ? th[P.w2 + r * kHid + k] : 0.0f);
  } else if (i < n1 + n2 + n3) {
    const int j = i - n1 - n2, r = j / kLdh, k = j % kLdh;
    W3[j] = __float2bfloat16_rn(r < kOut && k < kHid ? th[P.w3 + r * kHid + k] : 0.0f);
  } else if (i < n1 + n2 + n3 + kHid) {
    const int j = i - n1 - n2 - n3;
    b1[j] = th[P.b1 + j];
  } else if (i < n1 + n2 + n3 + 2 * kHid) {
    const int j = i - n1 - n2 - n3 - kHid;
    b2[j] = th[P.b2 + j];
  } else if (i < n1 + n2 + n3 + 2 * kHid + kOutPad) {
    const int j = i - n1 - n2 - n3 - 2 * kHid;
    b3[j] = j < kOut ? th[P.b3 + j] : 0.0f;
  }
}

static int image_elems(const ImgLayout& L) { return kHid * L.ld1 + kHid * kLdh + kOutPad * kLdh + 2 * kHid + kOutPad; }

// Seeded uniform(-1/sqrt(fan_in), 1/sqrt(fan_in)) initialisation; parameter
// j of the network's own (compact) order draws counter j, padding stays 0.
__global__ void k_init_params(float* __restrict__ th, ParamLayout P, int n_in, int plain, unsigned long long seed) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P.total) return;
  const int j = plain ? paper_index(i, P, n_in) : i;
  if (j < 0) {
    th[i] = 0.0f;
    return;
  }
  const float fan = i < P.w2 ? (float)n_in : (i < P.w3 || !plain ? (float)kHid : (float)kPaperH2);
  const float bound = 1.0f / sqrtf(fan);
  const float u = u24_hi(sm_at(sm_at(sm_at(seed, kStreamInit), 0ull), (uint64_t)j));
  th[i] = -bound + u * (bound + bound);
}

// Copy the image into shared memory (16-byte vectors).
__device__ __forceinline__ void stage_image(uint8_t* dst, const uint8_t* __restrict__ src, int bytes) {
  const int4* s = reinterpret_cast<const int4*>(src);
  int4* d = reinterpret_cast<int4*>(dst);
  for (int i = threadIdx.x; i < bytes / 16; i += blockDim.x) d[i] = __ldg(s + i);
}

// The same through the bulk-copy engine: thread 0 issues the copies (image
// bytes are a multiple of 16, both ends 16-byte aligned) on the mbarrier
// `bar` (initialised by the caller with one arrival), every thread waits
// for its phase `parity` (bounded).  CTA-wide; false when the copy did not
// complete within the bound.
constexpr int kStageChunk = 32 * 1024;
__device__ __forceinline__ void stage_image_issue(uint8_t* dst, const uint8_t* __restrict__ src, int bytes,
                                                  uint64_t* bar) {
  mbar_expect_tx(bar, (uint32_t)bytes);
  for (int off = 0; off < bytes; off += kStageChunk)
    bulk_g2s(dst + off, src + off, (uint32_t)min(kStageChunk, bytes - off), bar);
}
__device__ __forceinline__ bool stage_image_bulk(uint8_t* dst, const uint8_t* __restrict__ src, int bytes,
                                                 uint64_t* bar, uint32_t parity, uint32_t tries) {
  if (threadIdx.x == 0) stage_image_issue(dst, src, bytes, bar);
  return __syncthreads_and(mbar_wait(bar, parity, tries));
}

// Pointers into a shared-memory copy of the image.
struct QW {
  const bf16* W1;
  const bf16* W2;
  const bf16* W3;
  const float* b1;
  const float* b2;
  const float* b3;
  int k1, ld1;
};
__device__ __forceinline__ QW qw_at(const uint8_t* base, const ImgLayout& L) {
  QW w;
  w.W1 = reinterpret_cast<const bf16*>(base + L.w1);
  w.W2 = reinterpret_cast<const bf16*>(base + L.w2);
  w.W3 = reinterpret_cast<const bf16*>(base + L.w3);
  w.b1 = reinterpret_cast<const float*>(base + L.b1);
  w.b2 = reinterpret_cast<const float*>(base + L.b2);
  w.b3 = reinterpret_cast<const float*>(base + L.b3);
  w.k1 = L.k1;
  w.ld1 = L.ld1;
  return w;
}

__device__ __forceinline__ void group_barrier(int id, int nthreads) {
  asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(nthreads) : "memory");
}

// B fragments of k-step k0 of 16 samples X[16][ldx] (two n-tiles of 8).
__device__ __forceinline__ void load_x16(uint32_t (&x)[4], const bf16* X, int ldx, int k0, int lane) {
  ldsm_x4(x, X + ((lane & 7) + (lane >> 4) * 8) * ldx + k0 + ((lane >> 3) & 1) * 8);
}
// One hidden layer of 16 rows by 16 warps of 16 units: H[16][256] = bf16(ReLU(X
// W^T + b)).  Bound by shared-memory reads: with the weights as the A operand
// each is read once and the 16 rows once per warp (256 KB a layer of 256
// inputs); with the rows as A and 8 units per warp and pass it was 384 KB.
// kRows = 8: rows 0..7 only (the others keep what H holds): half of the MMAs.
// With bar >= 0 H may be X: the 16 warps meet on that named barrier between
// their last read and their stores.
template <int kRows = 16>
__device__ __forceinline__ void hidden_layer(const bf16* X, int ldx, int nks, const bf16* W, int ldw, const float* b,
                                             bf16* H, int warp, int lane, int bar = -1) {
  constexpr int kNt = kRows / 8;
  const int g = lane >> 2, q = lane & 3, u0 = 16 * warp;
  float c[kNt][4] = {};
#pragma unroll 4
  for (int ks = 0; ks < nks; ++ks) {
    uint32_t a[4], x[4];
    load_a_row(a, W, ldw, u0, 16 * ks, lane);
    if (kNt == 2)
      load_x16(x, X, ldx, 16 * ks, lane);
    else
      load_b_col(x[0], x[1], X, ldx, 16 * ks, 0, lane);
    mma_bf16(c[0], a, x[0], x[1]);
    if (kNt == 2) mma_bf16(c[kNt - 1], a, x[2], x[3]);
  }
  const float bl = b[u0 + g], bh = b[u0 + g + 8];
  if (bar >= 0) group_barrier(bar, 512);
#pragma unroll
  for (int t = 0; t < kNt; ++t)
#pragma unroll
    for (int j = 0; j < 4; ++j)
      H[(8 * t + 2 * q + (j & 1)) * kLdh + u0 + g + (j >> 1) * 8] =
          __float2bfloat16_rn(fmaxf(c[t][j] + (j >> 1 ? bh : bl), 0.f));
}

// Head of 16 rows (one warp): O[16][8] = H2 * W3^T + b3 (FP32), two
// accumulator chains (even / odd k-steps) summed in a fixed order.
__device__ __forceinline__ void head_layer(const bf16* H2, const QW& w, float* O, int lane) {
  const int g = lane >> 2, q = lane & 3;
  float acc0[4] = {0.f, 0.f, 0.f, 0.f}, acc1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
  for (int k0 = 0; k0 < kHid; k0 += 32) {
    uint32_t a[4], b[4];
    // W3 rows 0..7, columns k0 .. k0 + 31: the B fragments of both k-steps
    ldsm_x4(b, w.W3 + (lane & 7) * kLdh + k0 + (lane >> 3) * 8);
    load_a_row(a, H2, kLdh, 0, k0, lane);
    mma_bf16(acc0, a, b[0], b[1]);
    load_a_row(a, H2, kLdh, 0, k0 + 16, lane);
    mma_bf16(acc1, a, b[2], b[3]);
  }
  const int n = 2 * q;
  O[g * kOutPad + n] = (acc0[0] + acc1[0]) + w.b3[n];
  O[g * kOutPad + n + 1] = (acc0[1] + acc1[1]) + w.b3[n + 1];
  O[(g + 8) * kOutPad + n] = (acc0[2] + acc1[2]) + w.b3[n];
  O[(g + 8) * kOutPad + n + 1] = (acc0[3] + acc1[3]) + w.b3[n + 1];
}

// The forward of one 16-row tile by a group of 16 warps that synchronise
// among themselves on named barrier `bar` (0: the whole CTA is the group;
// otherwise the other warps of the CTA run on); wg = the warp's index in its
// group.  kRows = 8: the rows from 8 on hold no sample.  H2 may be H1.
template <int kRows = 16>
__device__ __forceinline__ void mlp_tile(const QW& w, const bf16* X, bf16* H1, bf16* H2, float* O, int wg, int lane,
                                         int bar = 0) {
  hidden_layer<kRows>(X, w.ld1, w.k1 / 16, w.W1, w.ld1, w.b1, H1, wg, lane);
  group_barrier(bar, 512);
  hidden_layer<kRows>(H1, kLdh, kHid / 16, w.W2, kLdh, w.b2, H2, wg, lane, H2 == H1 ? bar : -1);
  group_barrier(bar, 512);
  if (wg == 0) head_layer(H2, w, O, lane);
  group_barrier(bar, 512);
}

// Dueling combine and greedy action of one row of head outputs:
// Q_a = (V + A_a) - mean(A), argmax with the lowest index on ties.
__device__ __forceinline__ uint32_t greedy_action(const float* o, float* qv = nullptr, int plain = 0) {
  if (plain) {
    // the paper's network: the outputs are the Q-values
    uint32_t best = 0;
    float bq = o[0];
    if (qv) qv[0] = bq;
#pragma unroll
    for (int a = 1; a < kOut - 1; ++a) {
      if (qv) qv[a] = o[a];
      if (o[a] > bq) {
        bq = o[a];
        best = (uint32_t)a;
      }
    }
    return best;
  }
  const float V = o[0];
  const float meanA = ((((o[1] + o[2]) + o[3]) + o[4]) + o[5]) / 5.0f;
  uint32_t best = 0;
  float bq = (V + o[1]) - meanA;
  if (qv) qv[0] = bq;
#pragma unroll
  for (int a = 1; a < kOut - 1; ++a) {
    const float qa = (V + o[1 + a]) - meanA;
    if (qv) qv[a] = qa;
    if (qa > bq) {
      bq = qa;
      best = (uint32_t)a;
    }
  }
  return best;
}

// This warp's observation row (lane share `o`) into a BF16 tile row.
__device__ __forceinline__ void obs_to_tile(bf16* row, const ObsRegs& o, int B, int lane) {
  if (lane < B) row[lane] = __float2bfloat16_rn(o.b0);
  if (lane + 32 < B) row[lane + 32] = __float2bfloat16_rn(o.b1);
  if (lane < 5) row[B + lane] = __float2bfloat16_rn(o.ex);
}

// ------------------------------------------------ tcgen05 batched forward
// Q[M][5] of obs[M][n_in] on the fifth-generation tensor cores, 128 rows per
// tile.  A persistent CTA (one per SM) holds W1 and W2 in shared memory (one
// set of bulk asynchronous copies (TMA) from a copy of the online network in
// the tensor cores' layout, k_tc_image) and the whole 512-column tensor
// memory.  Per tile: the threads convert the 128 input rows to BF16 (X, shared
// memory); one thread issues the MMAs of a hidden layer (tcgen05.mma, FP32
// accumulators in tensor memory) and commits them to an mbarrier; 16 warps
// read the accumulators back (warps w, w + 4, .. take the rows of lane quarter
// w % 4 and 64 columns each) and add the bias, apply ReLU and round to BF16.
// H1 goes back into the first half of the columns it was read from
// (tcgen05.st) and is the A operand of layer 2's MMAs.  H2 is read in the
// fragment shape of mma.sync and never leaves the registers: the head (6
// outputs) is eight m16n8k16 a warp on its 64 columns, the four column groups'
// sums meet in shared memory and three more warps write the Q-values.
// Tensor-memory columns:
//   [0, 256)   layer 1 accumulators; H1 in the first half of each 64
//   [256, 512) layer 2 accumulators
// Bound by the tensor cores' layer 2 (2,048 cycles a tile) with the two
// epilogues behind it; the next tile's layer 1 runs beside the layer-2
// epilogue.  As a tcgen05 layer of its own the head (16 MMAs at their
// 88-cycle floor for any N up to 128, and H2's store) sat in that chain, and
// row-wise input loads took 24 lines a warp instruction: 2^20 rows of 37
// inputs 185 -> 154 us.
// Shared memory: X 128 x k1 | W1 256 x k1 | W2 256 x 256 (the canonical K-major
// layout of sg_tc.cuh) | head sums.  Same BF16 recipe as the mma.sync kernels
// (BF16 inputs, weights and hidden activations, FP32 sums); only the
// summation order differs.
constexpr int kTcRows = 128;
constexpr uint32_t kTcTries = 1u << 24;  // bound of every mbarrier wait (polls)
// The launch takes the whole shared memory of an SM (one CTA per SM either
// way), so that every descriptor-addressed byte lies inside the allocation.
constexpr uint32_t kTcSmemLaunch = 227u * 1024u - 4096u;

struct TcSmem {
  uint32_t x, w1, w2, part, bytes;
};
__host__ __device__ inline uint32_t tc_up(uint32_t v) { return (v + 1023u) & ~1023u; }
__host__ __device__ inline TcSmem tc_smem(int k1) {
  TcSmem t;
  t.x = 0;
  t.w1 = tc_up(t.x + (uint32_t)(kTcRows * k1 * 2));
  t.w2 = tc_up(t.w1 + (uint32_t)(kHid * k1 * 2));
  t.part = tc_up(t.w2 + (uint32_t)(kHid * kHid * 2));  // head sums [2][4][128][8] float
  t.bytes = tc_up(t.part + (uint32_t)(2 * 4 * kTcRows * kOutPad * 4));
  return t;
}
// k1 <= 80 (n_in <= 69): 220 KB, inside the launch's shared memory
static_assert(kTcRows * 80 * 2 + 1024 + kHid * 80 * 2 + kHid * kHid * 2 + 32 * 1024 + 1024 <= kTcSmemLaunch,
              "tcgen05 forward: operands exceed the shared memory");
// The weight copy in global memory: blocks identical to their shared-memory
// images, so that each is one bulk copy.
// For the fused rollout W1 and W2 in two 128-row halves each, for the batched
// forward and the learner as one 256-row operand each (all canonical operands).
struct TcImg {
  uint32_t w1, w2a, w2b, w3, w1h, w2f, bytes;
};
__host__ __device__ inline TcImg tc_img(int k1) {
  TcImg t;
  t.w1 = 0;
  t.w2a = (uint32_t)(kHid * k1 * 2);
  t.w2b = t.w2a + 128u * kHid * 2u;
  t.w3 = t.w2b + 128u * kHid * 2u;
  t.w1h = t.w3 + 16u * kHid * 2u;
  t.w2f = t.w1h + (uint32_t)(kHid * k1 * 2);
  t.bytes = t.w2f + (uint32_t)(kHid * kHid * 2);
  return t;
}

// The online weights from the BF16 image (rows of ld1 / kLdh elements) into
// the canonical layout: W1 (256 rows), W2 rows 0..127 and 128..255 (two
// 128-row operands), W3 (16 rows, 6 used).
__global__ void k_tc_image(const uint8_t* __restrict__ img, ImgLayout L, uint8_t* __restrict__ out) {
  const TcImg T = tc_img(L.k1);
  const int n1 = kHid * (L.k1 / 8), n2 = kHid * (kHid / 8), n3 = 16 * (kHid / 8);
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n1 + n2 + n3; c += gridDim.x * blockDim.x) {
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    uint32_t dst;
    if (c < n1) {
      const int n = c % kHid, kg = c / kHid;
      v = __ldg(reinterpret_cast<const uint4*>(img + L.w1 + ((size_t)n * L.ld1 + kg * 8) * 2));
      dst = T.w1 + kmajor_offset(n, kg * 8, kHid);
      // the same chunk in its 128-row half
      *reinterpret_cast<uint4*>(out + T.w1h + (uint32_t)((n >> 7) * 128 * L.k1 * 2) +
                                kmajor_offset(n & 127, kg * 8, 128)) = v;
    } else if (c < n1 + n2) {
      const int j = c - n1, n = j % kHid, kg = j / kHid;
      v = __ldg(reinterpret_cast<const uint4*>(img + L.w2 + ((size_t)n * kLdh + kg * 8) * 2));
      dst = n < 128 ? T.w2a + kmajor_offset(n, kg * 8, 128) : T.w2b + kmajor_offset(n - 128, kg * 8, 128);
      // in the 256-row operand
      *reinterpret_cast<uint4*>(out + T.w2f + kmajor_offset(n, kg * 8, kHid)) = v;
    } else {
      const int j = c - n1 - n2, n = j % 16, kg = j / 16;
      if (n < kOutPad) v = __ldg(reinterpret_cast<const uint4*>(img + L.w3 + ((size_t)n * kLdh + kg * 8) * 2));
      dst = T.w3 + kmajor_offset(n, kg * 8, 16);
    }
    *reinterpret_cast<uint4*>(out + dst) = v;
  }
}

// Epilogue warps of the batched forward: four per lane quarter (warp w
// takes lanes 32 (w % 4) .. and the kTfCols accumulator columns of group
// w / 4).
constexpr int kTfEpiWarps = 16;
constexpr int kTfEpiThreads = kTfEpiWarps * 32;
constexpr int kTfWriters = 96;                               // Q-value writers
constexpr int kTfThreads = kTfEpiThreads + 32 + kTfWriters;  // + the MMA-issue warp
constexpr int kTfCols = kHid / (kTfEpiWarps / 4);
static_assert(kTfCols % 32 == 0, "each epilogue warp's columns hold whole 16-column chunks and head accumulators");

// Hidden-layer epilogue in tensor memory: this thread's lane (row
// 32 (warp % 4) + lane), accumulator columns [tacc + kTfCols g, + kTfCols) for
// g = warp / 4, plus the bias, ReLU, rounded to BF16 pairs and stored over the
// first half of those columns (units kTfCols g + 2 c, + 1 in column
// tacc + kTfCols g + c).  The load of the next 16 columns is in flight while
// a chunk is converted; a chunk's 8 output columns lie below every column
// still to be read, and each load completes before the columns it frees are
// written.  Returns once the stores have completed.
__device__ __forceinline__ void tc_epilogue_tmem(uint32_t tacc, const float* bias, int warp) {
  constexpr int kChunks = kTfCols / 16;
  const uint32_t t = tacc + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * kTfCols);
  const float4* b4 = reinterpret_cast<const float4*>(bias + (warp >> 2) * kTfCols);
  uint32_t r[2][16];
  tmem_ld16_nowait(t, r[0]);
  tmem_ld_wait();
#pragma unroll
  for (int ch = 0; ch < kChunks; ++ch) {
    if (ch + 1 < kChunks) tmem_ld16_nowait(t + (uint32_t)(16 * (ch + 1)), r[(ch + 1) & 1]);
    const uint32_t(&v)[16] = r[ch & 1];
    uint32_t w[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float4 bb = b4[4 * ch + j];
      w[2 * j] = pack_bf16x2_relu(__uint_as_float(v[4 * j]) + bb.x, __uint_as_float(v[4 * j + 1]) + bb.y);
      w[2 * j + 1] = pack_bf16x2_relu(__uint_as_float(v[4 * j + 2]) + bb.z, __uint_as_float(v[4 * j + 3]) + bb.w);
    }
    tmem_st8(t + (uint32_t)(8 * ch), w);
    if (ch + 1 < kChunks) tmem_ld_wait();
  }
  tmem_st_wait();
}
// Tensor-memory column (relative to the layer's accumulators) of K step ks
// of the packed activations.
__host__ __device__ constexpr uint32_t tf_a_col(int ks) {
  return (uint32_t)((ks / (kTfCols / 16)) * kTfCols + (ks % (kTfCols / 16)) * 8);
}

// One layer from a tensor-memory A operand (the packed activations of
// tc_epilogue_tmem with accumulators at column a, K = 256):
// D[d] = A x B^T for B in shared memory of Rb rows (K-major, canonical);
// one thread.
__device__ __forceinline__ void tc_layer_ta(uint32_t d, uint32_t a, uint32_t b_smem, int Rb) {
  const uint32_t idesc = idesc_bf16_f32(kTcRows, Rb);
  const uint32_t lb = (uint32_t)Rb * 16;
#pragma unroll 1
  for (int ks = 0; ks < kHid / 16; ++ks)
    tc_mma_bf16_ta(d, a + tf_a_col(ks), smem_desc(b_smem + (uint32_t)ks * 2 * lb, lb, 128), idesc, ks > 0 ? 1u : 0u);
}

// Layer-2 epilogue and head of a warp's 64 columns [tacc + 64 (warp / 4), + 64):
// its 32 rows in two halves of 16, bias and ReLU into A fragments, times the
// columns' W3 fragments w3 (b0, b1 of each 16-column step); the sums of row r to
// out[8 r ..].
__device__ __forceinline__ void tf_epilogue_head(uint32_t tacc, const float* bias, const uint32_t (&w3)[8], float* out,
                                                 int warp, int lane) {
  static_assert(kTfCols == 64, "one fragment load per half");
  const int g = lane >> 2, q = lane & 3;
  const uint32_t t = tacc + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * kTfCols);
  const float2* b2 = reinterpret_cast<const float2*>(bias + (warp >> 2) * kTfCols) + q;
  uint32_t r[2][32];
  tmem_ld_frag64_nowait(t, r[0]);
  tmem_ld_frag64_nowait(t + (16u << 16), r[1]);
  tmem_ld_wait();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      uint32_t a[4];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float2 bb = b2[4 * (2 * i + j)];
        const uint32_t* v = r[h] + 4 * (2 * i + j);
        a[2 * j] = pack_bf16x2_relu(__uint_as_float(v[0]) + bb.x, __uint_as_float(v[1]) + bb.y);
        a[2 * j + 1] = pack_bf16x2_relu(__uint_as_float(v[2]) + bb.x, __uint_as_float(v[3]) + bb.y);
      }
      mma_bf16(acc, a, w3[2 * i], w3[2 * i + 1]);
    }
    float* o = out + ((warp & 3) * 32 + 16 * h + g) * kOutPad + 2 * q;
    *reinterpret_cast<float2*>(o) = make_float2(acc[0], acc[1]);
    *reinterpret_cast<float2*>(o + 8 * kOutPad) = make_float2(acc[2], acc[3]);
  }
}

// Input rows of a tile into the X operand (BF16; its padding columns are zero
// from the start) in two steps: tc_fetch_x loads the tile's floats, which are
// contiguous, in order over the threads (a line a warp instruction),
// tc_store_x converts and stores them.  div: ceil(2^20 / n_in), exact for the
// index / n_in of at most 128 x 69 floats.
constexpr int kTcXFloats = (kTcRows * 69 + kTfEpiThreads - 1) / kTfEpiThreads;
__device__ __forceinline__ void tc_fetch_x(float (&x)[kTcXFloats], const float* __restrict__ obs, int n_in, int M,
                                           long long tile, int tid) {
  const long long first = tile * kTcRows;
  const int total = (int)min((long long)kTcRows, M - first) * n_in;
  const float* src = obs + first * n_in;
#pragma unroll
  for (int i = 0; i < kTcXFloats; ++i) {
    const int e = tid + i * kTfEpiThreads;
    x[i] = e < total ? __ldg(src + e) : 0.0f;
  }
}
__device__ __forceinline__ void tc_store_x(uint8_t* xs, const float (&x)[kTcXFloats], int n_in, uint32_t div, int tid) {
#pragma unroll
  for (int i = 0; i < kTcXFloats; ++i) {
    const int e = tid + i * kTfEpiThreads;
    if (e < kTcRows * n_in) {
      const int row = (int)(((uint32_t)e * div) >> 20), k = e - row * n_in;
      *reinterpret_cast<bf16*>(xs + kmajor_offset(row, k, kTcRows)) = __float2bfloat16_rn(x[i]);
    }
  }
  fence_async_smem();
}

// Warps 0..15 run the epilogues and convert the inputs, warp 16 (one lane)
// copies the weights and issues every MMA, so that the issue, which waits
// while the tensor cores' queue is full, never holds up an epilogue, and warps
// 17..19 write Q.  The input loads (2,000 cycles) follow the layer-1 epilogue,
// beside layer 2: issued before it they hold its tensor-memory waits (188 us a
// call of 2^20 rows), and on warps 17..19 alone they are too slow (217 us).
// They meet on mbarriers, one phase per tile each: bar_x (X
// stored), bar_h1 (H1 stored and the previous tile's layer 2 read), and the
// MMA commits bar_l1, bar_l2 (layer complete); the head sums of tile t pass
// through named barriers 1 + t % 2 (written) and 3 + t % 2 (read).  Order on
// the tensor cores: layer 2 (t) once H1 (t) is stored; layer 1 (t + 1) once
// layer 2 (t) is complete and X (t + 1) is stored.
__global__ void __launch_bounds__(kTfThreads, 1) k_qnet_forward_tc(const uint8_t* __restrict__ img,
                                                                const uint8_t* __restrict__ timg, ImgLayout L,
                                                                const float* __restrict__ obs, int M,
                                                                float* __restrict__ qout) {
  extern __shared__ __align__(1024) uint8_t tsm[];
  __shared__ uint64_t bar_w, bar_l1, bar_l2, bar_x, bar_h1, bar_drain;
  __shared__ uint32_t tslot;
  __shared__ int s_fail;
  __shared__ __align__(16) float sb1[kHid];
  __shared__ __align__(16) float sb2[kHid];
  const TcSmem T = tc_smem(L.k1);
  const TcImg G = tc_img(L.k1);
  uint8_t* xs = tsm + T.x;
  float* part = reinterpret_cast<float*>(tsm + T.part);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ntiles = (M + kTcRows - 1) / kTcRows;
  // this CTA's tiles: blockIdx.x + i gridDim.x, i < my_tiles
  const int my_tiles = (int)blockIdx.x < ntiles ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  for (int i = tid; i < kHid; i += kTfThreads) {
    sb1[i] = __ldg(reinterpret_cast<const float*>(img + L.b1) + i);
    sb2[i] = __ldg(reinterpret_cast<const float*>(img + L.b2) + i);
  }
  for (int i = tid; i < kTcRows * L.k1 / 8; i += kTfThreads)
    reinterpret_cast<uint4*>(xs)[i] = make_uint4(0u, 0u, 0u, 0u);
  fence_async_smem();
  if (warp == 0) tmem_alloc(&tslot, 512);
  if (tid == 0) {
    mbar_init(&bar_w, 1);
    mbar_init(&bar_l1, 1);
    mbar_init(&bar_l2, 1);
    mbar_init(&bar_drain, 1);
    mbar_init(&bar_x, kTfEpiThreads);
    mbar_init(&bar_h1, kTfEpiThreads);
    s_fail = 0;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tacc = tslot, tacc2 = tacc + 256u;
  volatile int* fail = &s_fail;
  constexpr int kHandover = kTfEpiThreads + kTfWriters;
  if (warp == kTfEpiWarps) {
    if (lane == 0 && my_tiles > 0) {
      // ---- MMA issue
      const uint32_t sx = smem_u32(xs), sw1 = smem_u32(tsm + T.w1), sw2 = smem_u32(tsm + T.w2);
      auto issue_l1 = [&]() {
        const uint32_t idesc = idesc_bf16_f32(kTcRows, kHid);
        const uint32_t la = kTcRows * 16, lb = kHid * 16;
        for (int ks = 0; ks < L.k1 / 16; ++ks)
          tc_mma_bf16(tacc, smem_desc(sx + (uint32_t)ks * 2 * la, la, 128),
                      smem_desc(sw1 + (uint32_t)ks * 2 * lb, lb, 128), idesc, ks > 0 ? 1u : 0u);
        tc_commit(&bar_l1);
      };
      // the resident weights: W1, W2 (one 256-row operand)
      mbar_expect_tx(&bar_w, G.w2a + kHid * kHid * 2u);
      bulk_g2s(tsm + T.w1, timg + G.w1, G.w2a, &bar_w);
      bulk_g2s(tsm + T.w2, timg + G.w2f, kHid * kHid * 2u, &bar_w);
      bool ok = mbar_wait_or_fail(&bar_w, 0, kTcTries, fail) && mbar_wait_or_fail(&bar_x, 0, kTcTries, fail);
      if (ok) {
        tc_fence_after();
        issue_l1();
      }
      for (int it = 0; ok && it < my_tiles; ++it) {
        const uint32_t par = (uint32_t)it & 1u;
        // layer 2 (t): D[256, 512) = H1 W2^T, N = 256
        ok = mbar_wait_or_fail(&bar_h1, par, kTcTries, fail);
        if (!ok) break;
        tc_fence_after();
        tc_layer_ta(tacc2, tacc, sw2, kHid);
        tc_commit(&bar_l2);
        // layer 1 (t + 1) over H1 (t), once layer 2 (t) has read it
        if (it + 1 < my_tiles) {
          ok = mbar_wait_or_fail(&bar_x, par ^ 1u, kTcTries, fail) && mbar_wait_or_fail(&bar_l2, par, kTcTries, fail);
          if (!ok) break;
          tc_fence_after();
          issue_l1();
        }
      }
      // every MMA of this thread, and the weight copies, complete before the
      // tensor memory is freed (bounded waits)
      tc_commit(&bar_drain);
      mbar_wait(&bar_drain, 0, kTcTries);
      mbar_wait(&bar_w, 0, kTcTries);
    }
  } else if (warp > kTfEpiWarps) {
    // ---- read-out: rows of tile i from the four column groups' head sums
    // (NaN where a wait ran out)
    const int w = tid - kTfEpiThreads - 32;
    auto tile_of = [&](int i) { return (long long)blockIdx.x + (long long)i * gridDim.x; };
    float b3[kOut];
#pragma unroll
    for (int j = 0; j < kOut; ++j) b3[j] = __ldg(reinterpret_cast<const float*>(img + L.b3) + j);
    for (int i = 0; i < my_tiles; ++i) {
      group_barrier(1 + (i & 1), kHandover);
      const bool good = *fail == 0;
      const long long first = tile_of(i) * kTcRows;
      for (int r = w; r < kTcRows; r += kTfWriters) {
        const float* p = part + (i & 1) * 4 * kTcRows * kOutPad + r * kOutPad;
        float o[kOutPad];
#pragma unroll
        for (int j = 0; j < kOutPad; j += 2) {
          float2 v[4];
#pragma unroll
          for (int gq = 0; gq < 4; ++gq) v[gq] = *reinterpret_cast<const float2*>(p + gq * kTcRows * kOutPad + j);
          o[j] = (v[0].x + v[1].x) + (v[2].x + v[3].x);
          o[j + 1] = (v[0].y + v[1].y) + (v[2].y + v[3].y);
        }
        if (first + r < M) {
          float qv[5];
#pragma unroll
          for (int j = 0; j < kOut; ++j) o[j] += b3[j];
          greedy_action(o, qv, L.plain);
#pragma unroll
          for (int a = 0; a < 5; ++a) qout[(first + r) * 5 + a] = good ? qv[a] : __int_as_float(0x7fc00000);
        }
      }
      __threadfence_block();
      asm volatile("bar.arrive %0, %1;\n" ::"r"(3 + (i & 1)), "n"(kHandover) : "memory");
    }
  } else {
    // ---- epilogues, inputs (warps 0..15)
    const uint32_t div = ((1u << 20) + (uint32_t)L.n_in - 1u) / (uint32_t)L.n_in;
    bool ok = true;
    auto wait = [&](uint64_t* bar, uint32_t par) {
      ok = __all_sync(0xffffffffu, ok && mbar_wait_or_fail(bar, par, kTcTries, fail));
      if (ok) tc_fence_after();
    };
    // this lane's W3 fragments: outputs g, columns 64 (warp / 4) + 16 i + 2 q ..
    uint32_t w3[8];
    {
      const bf16* w = reinterpret_cast<const bf16*>(img + L.w3) + (lane >> 2) * kLdh + (warp >> 2) * kTfCols + 2 * (lane & 3);
#pragma unroll
      for (int i = 0; i < 8; ++i) w3[i] = __ldg(reinterpret_cast<const uint32_t*>(w + 8 * i));
    }
    float xr[kTcXFloats];
    if (my_tiles > 0) {
      tc_fetch_x(xr, obs, L.n_in, M, blockIdx.x, tid);
      tc_store_x(xs, xr, L.n_in, div, tid);
      mbar_arrive(&bar_x);
    }
    for (int it = 0; it < my_tiles; ++it) {
      const uint32_t par = (uint32_t)it & 1u;
      wait(&bar_l1, par);
      if (ok) tc_epilogue_tmem(tacc, sb1, warp);  // H1 over the layer-1 accumulators
      tc_fence_before();
      mbar_arrive(&bar_h1);
      // X is free (layer 1 of t is complete): the next tile's inputs while layer 2 runs
      if (ok && it + 1 < my_tiles) {
        tc_fetch_x(xr, obs, L.n_in, M, (long long)blockIdx.x + (long long)(it + 1) * gridDim.x, tid);
        tc_store_x(xs, xr, L.n_in, div, tid);
        mbar_arrive(&bar_x);
      }
      if (it >= 2) group_barrier(3 + (it & 1), kHandover);  // the sums of t - 2 are read
      wait(&bar_l2, par);
      if (ok)
        tf_epilogue_head(tacc2, sb2, w3, part + ((it & 1) * 4 + (warp >> 2)) * kTcRows * kOutPad, warp, lane);
      __threadfence_block();
      asm volatile("bar.arrive %0, %1;\n" ::"r"(1 + (it & 1)), "n"(kHandover) : "memory");
    }
    // the read-out's last arrivals
    for (int it = max(my_tiles, 2); it < my_tiles + 2; ++it) group_barrier(3 + (it & 1), kHandover);
    tc_fence_before();
  }
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tmem_free(tacc, 512);
}

// One thread of every CTA of a rollout, after the CTA's last use of the ring's
// step counter: the last CTA advances it by the K steps recorded and leaves
// the CTA count (behind it) zero for the next launch.  A learner on another
// stream may read the counter at any moment (ring_steps): every CTA's entries
// are ordered before the count, and the counts before the new value.
__device__ __forceinline__ void replay_advance(const ReplayDev& rp, int use_replay, int K) {
  if (!use_replay) return;
  unsigned* done = reinterpret_cast<unsigned*>(rp.steps + 1);
  __threadfence();
  if (atomicAdd(done, 1u) == gridDim.x - 1u) {
    __threadfence();
    *done = 0u;
    *rp.steps += (unsigned long long)K;
  }
}
// The counter as a learner reads it: the entries that it counts are visible
// after this load.
__device__ __forceinline__ unsigned long long ring_steps(const ReplayDev& rp) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];\n" : "=l"(v) : "l"(rp.steps) : "memory");
  return v;
}

// VEM eps-greedy rollout with the network fused in: per step, the 16 envs of
// a group write their observations to a BF16 tile, the tile goes through the
// network on the tensor cores, every env takes argmax Q or (with probability
// eps_i) the random action, then steps; the transition is appended to the
// replay ring.  One warp per env; 16 envs per group, MT groups per CTA
// sharing the weight image.  The groups synchronise only among themselves
// (named barriers), so one group's env step overlaps the other's network.
template <int MT, bool kDyn, bool kFast>
__global__ void __launch_bounds__(512 * MT, 1)
    k_rollout_q(const __grid_constant__ DevCfg c, SimPtrs p, const uint8_t* __restrict__ img, ImgLayout L, int K,
                const float* __restrict__ eps, ReplayDev rp, int use_replay, const int* __restrict__ order, int epc,
                float* __restrict__ obs_out,
                float* __restrict__ obs_seq, uint8_t* __restrict__ act_seq, float* __restrict__ rew_seq,
                uint8_t* __restrict__ done_seq) {
  extern __shared__ __align__(16) uint8_t smem[];
  uint8_t* sw = smem;
  bf16* X = reinterpret_cast<bf16*>(smem + L.bytes);
  constexpr int kRows = 16 * MT;
  bf16* H1 = X + kRows * L.ld1;
  // layer 2 over layer 1: at most 48 (padded) inputs then fit 196 KB of shared
  // memory with 32 envs, which leaves the scans 60 KB of L1 instead of 28
  float* O = reinterpret_cast<float*>(H1 + kRows * kLdh);
  __shared__ uint64_t bar_img;
  if (threadIdx.x == 0) {
    // the weights on their way while the envs take their first observation
    mbar_init(&bar_img, 1);
    stage_image_issue(sw, img, L.bytes, &bar_img);
  }
  for (int i = threadIdx.x; i < kRows * L.ld1; i += blockDim.x) X[i] = __float2bfloat16_rn(0.0f);
  const QW w = qw_at(sw, L);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int grp = warp >> 4, wg = warp & 15, bar = 1 + grp;
  bf16* Xg = X + grp * 16 * L.ld1;
  bf16* H1g = H1 + grp * 16 * kLdh;
  float* Og = O + grp * 16 * kOutPad;
  // CTAs take envs grouped by map, so that one CTA's scans share cache lines;
  // epc <= kRows envs per CTA (fewer than the tile when that spreads the
  // envs over more SMs; the tile's other rows stay zero)
  const int slot = blockIdx.x * epc + warp;
  const bool live = warp < epc && slot < c.n_envs;
  const int env = live ? order[slot] : 0;
  const long long n = c.n_envs;
  EnvConst k;
  Env s;
  ObsRegs o;
  o.b0 = o.b1 = o.ex = 0.0f;
  float eps_i = 0.0f;
  uint64_t akey = 0;
  // dynamic obstacles: lane o holds disc o, every lane the centres
  Obst b = {0.0f, 0.0f, 0.0f, 0.0f};
  Discs dsc;
  if (live) {
    k = env_const(c, p, env, lane);
    s = load_env(p, env);
    if (kDyn) {
      if (lane < c.n_dyn) b = load_obst(p, lane, env);
      gather_discs(c, b, dsc);
    }
    const Noise z = noise_for(k, s.sigma, s.ep_id, s.ep_step, lane);
    Aux aux;
    observe<kDyn, kFast>(c, k, s, z, lane, o, aux, &dsc);  // the current observation, from the state
    eps_i = eps[env];
    akey = sm_at(sm_at(c.seed, kStreamAction), (uint64_t)env);
  }
  const unsigned long long rbase = use_replay ? *rp.steps : 0ull;
  uint32_t slot_t = use_replay ? (uint32_t)(rbase % (unsigned long long)rp.slots) : 0u;  // ring slot of step i
  uint32_t ra_batch = 0, ex_batch = 0;
  __syncthreads();  // the barrier is initialised
  if (!__syncthreads_and(mbar_wait(&bar_img, 0u, kTcTries))) {
    // no weights: the launch's outputs are incomplete; one more bounded wait
    // for the copy before the CTA exits
    if (threadIdx.x == 0) {
      atomicOr(p.status, SG_DEV_TIMEOUT);
      mbar_wait(&bar_img, 0u, kTcTries);
      replay_advance(rp, use_replay, K);
    }
    return;
  }
  for (int i = 0; i < K; ++i) {
    if (live) obs_to_tile(Xg + wg * L.ld1, o, c.B, lane);
    group_barrier(bar, 512);
    if (MT == 1 && epc <= 8)
      mlp_tile<8>(w, Xg, H1g, H1g, Og, wg, lane, bar);
    else
      mlp_tile(w, Xg, H1g, H1g, Og, wg, lane, bar);
    if (!live) continue;
    if ((i & 31) == 0) {
      // lane l draws the random action and the exploration uniform of step t + l
      const uint64_t h = sm_at(akey, (uint64_t)(s.t + (uint32_t)lane));
      ra_batch = (uint32_t)(sm_at(h, 0ull) >> 32) % (uint32_t)c.n_actions;
      ex_batch = __ballot_sync(kFull, u24_hi(sm_at(h, 1ull)) < eps_i);
    }
    const uint32_t ra = __shfl_sync(kFull, ra_batch, i & 31);
    const bool explore = (ex_batch >> (i & 31)) & 1u;
    const uint32_t greedy = greedy_action(Og + wg * kOutPad, nullptr, L.plain);
    const uint32_t a = explore ? ra : greedy;
    long long e = 0;
    float* srow = nullptr;
    float* s2row = nullptr;
    if (use_replay) {
      e = (long long)slot_t * rp.n_envs + env;
      slot_t = slot_t + 1u == (uint32_t)rp.slots ? 0u : slot_t + 1u;
      srow = rp.s + e * rp.obs_dim;
      s2row = rp.s2 + e * rp.obs_dim;
      write_obs(srow, o, c.B, lane);
    }
    const StepOut r = env_step<kDyn, kFast>(c, p, k, s, a, lane, o, s2row, &b, &dsc);
    if (use_replay) {
      if (!r.done) write_obs(s2row, o, c.B, lane);
      if (lane == 0) {
        rp.a[e] = (uint8_t)a;
        rp.r[e] = r.rew;
        rp.term[e] = (r.done & 3u) ? 1 : 0;
      }
    }
    if (obs_seq) write_obs(obs_seq + ((long long)i * n + env) * c.obs_dim, o, c.B, lane);
    if (lane == 0) {
      if (act_seq) act_seq[i * n + env] = (uint8_t)a;
      if (rew_seq) rew_seq[i * n + env] = r.rew;
      if (done_seq) done_seq[i * n + env] = (uint8_t)r.done;
    }
  }
  if (live) {
    if (obs_out) write_obs(obs_out + (long long)env * c.obs_dim, o, c.B, lane);
    if (lane == 0) store_env(p, env, s);
    if (kDyn && lane < c.n_dyn) store_obst(p, lane, env, b);
  }
  __syncthreads();  // this CTA's reads of the step counter are done
  if (threadIdx.x == 0) replay_advance(rp, use_replay, K);
}

// ---------------------------------------- tcgen05 fused eps-greedy rollout
// For large env counts: 128 envs per CTA form one 128-row tile of the
// network.  Per step the network runs on the tile on the tensor cores
// (tcgen05 MMAs into 256 tensor-memory columns, epilogues split over the 8
// warps of each lane quarter), warps 0-3 take the greedy actions from the
// head, the first four warps run what every env of the tile takes, one env per
// lane (lane_motion, as in sg_sim_step), and then every warp takes the rest row
// by row from a shared counter (bit-row collision test, scan, AutoReset),
// writing the next observation as the tile's BF16 row and the FP32 outputs
// and ring entries.  Same VEM draws, same simulator values as k_rollout_q; the Q
// values differ from it only in the summation order.
//
// Shared memory is kept small (102 KB) so that L1 keeps room for the maps the
// scans read: the hidden activations stay in tensor memory (an epilogue packs
// its BF16 pairs into the first half of the columns it read, the next layer's A
// operand; layer 1 in columns [0, 256), layer 2 in [256, 512), the head in
// [16, 32); in shared memory, 136 KB, 65,536 envs x 32 steps took 3,566 us against
// 3,518), and all of W1 (two 128-row halves) and W2 (four 32 KB pieces: the K
// halves of its two 128-row halves) stream through two 32 KB buffers by bulk
// copies every step, each copy issued as soon as its buffer's previous MMAs are
// done (both W1 halves during the env steps, the first two W2 pieces during
// the layer-1 epilogue); W3 stays.
constexpr int kQtEnvs = 128;
constexpr int kQtWarps = 32;
constexpr int kQtThreads = kQtWarps * 32;
constexpr uint32_t kQtBuf = 32u * 1024u;
constexpr uint32_t kQtRecOff = (uint32_t)(kQtEnvs * 80 * 2);  // step records behind the input tile (k1 <= 80)
// The env steps of a tile: what every env takes, one env per lane of the first
// four warps (lane_motion); the bit-row collision test and AutoReset, which
// few take, go with the scans, a warp per row.  With 16 warps of 8 lanes doing
// the whole scalar step, 65,536 envs x 32 steps took 4,112 us (3,664 now).
struct QtSmem {
  uint32_t hx, b0, b1, w3, bytes;
};
__host__ __device__ inline QtSmem qt_smem() {
  QtSmem t;
  t.hx = 0;
  t.b0 = kQtRecOff + kQtEnvs * (uint32_t)sizeof(MotionRec);
  t.b1 = t.b0 + kQtBuf;
  t.w3 = t.b1 + kQtBuf;
  t.bytes = t.w3 + 16u * kHid * 2u;
  return t;
}

// Epilogue of a hidden layer by 32 warps: warp w takes the rows of lane
// quarter w % 4 and columns [32 (w / 4), + 32) of the accumulators at tacc and
// packs them into the first 16 of these columns.
__device__ __forceinline__ void qt_epilogue(uint32_t tacc, const float* bias, int warp) {
  const int c = (warp >> 2) * 32;
  const uint32_t t = tacc + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c;
  float v[32];
  tmem_ld32(t, v);
  uint32_t w[16];
#pragma unroll
  for (int j = 0; j < 16; ++j)
    w[j] = pack_bf16x2(fmaxf(v[2 * j] + bias[c + 2 * j], 0.f), fmaxf(v[2 * j + 1] + bias[c + 2 * j + 1], 0.f));
  tmem_st16(t, w);
  tmem_st_wait();
}
// Column (relative to the layer's accumulators) of K step ks of the packed
// activations.
__device__ __forceinline__ uint32_t qt_a_col(int ks) { return (uint32_t)((ks >> 1) * 32 + (ks & 1) * 8); }

// This lane's share of an observation row into row r of the BF16 input tile.
__device__ __forceinline__ void qt_obs_to_tile(uint8_t* xs, int r, float b0, float b1, float ex, int B, int lane) {
  if (lane < B) *reinterpret_cast<bf16*>(xs + kmajor_offset(r, lane, kQtEnvs)) = __float2bfloat16_rn(b0);
  if (lane + 32 < B) *reinterpret_cast<bf16*>(xs + kmajor_offset(r, lane + 32, kQtEnvs)) = __float2bfloat16_rn(b1);
  if (lane < 5) *reinterpret_cast<bf16*>(xs + kmajor_offset(r, B + lane, kQtEnvs)) = __float2bfloat16_rn(ex);
}

// The weight stream of the fused rollout, run by the CTA's thread 0: chunk
// copies into two buffers (one mbarrier each for the copy, one for the MMAs
// that read the buffer) with every copy and every MMA group waited exactly
// once, in order.
struct QtStream {
  uint64_t* ld;    // [2] copy complete
  uint64_t* mm;    // [2] MMAs reading the buffer complete
  uint8_t* buf[2];
  uint32_t pl[2], pm[2];
  bool ld_out[2], mm_out[2];
  bool ok;
  // copy `bytes` from src into buffer b once its previous MMAs are done
  __device__ __forceinline__ void load(int b, const void* src, uint32_t bytes) {
    if (!ok) return;
    if (mm_out[b]) {
      ok = mbar_wait(&mm[b], pm[b], kTcTries);
      pm[b] ^= 1u;
      mm_out[b] = false;
      if (!ok) return;
    }
    mbar_expect_tx(&ld[b], bytes);
    bulk_g2s(buf[b], src, bytes, &ld[b]);
    ld_out[b] = true;
  }
  // MMAs D[tacc] (+)= A x buffer b^T (Rb rows, K; A in shared memory, or packed
  // in tensor memory at ta from its K step ks0; onto D when acc), then commits:
  // the buffer's barrier, and the layer barrier when `last`
  __device__ __forceinline__ void mma(int b, uint32_t tacc, const uint8_t* a, uint32_t ta, int Rb, int K,
                                      uint64_t* layer, bool last, int ks0 = 0, bool acc = false) {
    if (!ok) return;
    if (ld_out[b]) {
      ok = mbar_wait(&ld[b], pl[b], kTcTries);
      pl[b] ^= 1u;
      ld_out[b] = false;
      if (!ok) return;
    }
    tc_fence_after();
    const uint32_t idesc = idesc_bf16_f32(kQtEnvs, Rb);
    const uint32_t sb = smem_u32(buf[b]);
    const uint32_t la = kQtEnvs * 16, lb = (uint32_t)Rb * 16;
    for (int ks = 0; ks < K / 16; ++ks) {
      const uint64_t db = smem_desc(sb + (uint32_t)ks * 2 * lb, lb, 128);
      if (a)
        tc_mma_bf16(tacc, smem_desc(smem_u32(a) + (uint32_t)ks * 2 * la, la, 128), db, idesc, ks > 0 ? 1u : 0u);
      else
        tc_mma_bf16_ta(tacc, ta + qt_a_col(ks0 + ks), db, idesc, (acc || ks > 0) ? 1u : 0u);
    }
    tc_commit(&mm[b]);
    mm_out[b] = true;
    if (last) tc_commit(layer);
  }
  // bounded waits for whatever is still in flight
  __device__ __forceinline__ void drain() {
    for (int b = 0; b < 2; ++b) {
      if (mm_out[b]) mbar_wait(&mm[b], pm[b], kTcTries);
      if (ld_out[b]) mbar_wait(&ld[b], pl[b], kTcTries);
    }
  }
};

// State of env i through L2: with time slicing another SM may have written
// it during this launch.
__device__ __forceinline__ Env load_env_l2(const SimPtrs& p, int i) {
  Env s;
  const int n = p.n;
  s.x = __ldcg(p.f + 0 * n + i);
  s.y = __ldcg(p.f + 1 * n + i);
  s.phi = __ldcg(p.f + 2 * n + i);
  s.vl = __ldcg(p.f + 3 * n + i);
  s.va = __ldcg(p.f + 4 * n + i);
  s.dt = __ldcg(p.f + 5 * n + i);
  s.K = __ldcg(p.f + 6 * n + i);
  s.cap = __ldcg(p.f + 7 * n + i);
  s.sigma = __ldcg(p.f + 8 * n + i);
  s.ep_step = __ldcg(p.u + 0 * n + i);
  s.ep_id = __ldcg(p.u + 1 * n + i);
  s.t = __ldcg(p.u + 2 * n + i);
  s.fifo = __ldcg(p.u + 3 * n + i);
  f_sincos(s.phi, s.sphi, s.cphi);
  return s;
}

__device__ __forceinline__ unsigned qt_ld_acquire(const unsigned* a) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(a) : "memory");
  return v;
}
__device__ __forceinline__ void qt_st_release(unsigned* a, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;\n" ::"l"(a), "r"(v) : "memory");
}
constexpr unsigned kQtWaitIters = 1u << 22;  // x ~256 ns sleeps: about a second

// Time slicing (sync != null): a resident grid takes (segment of seg steps,
// 128-env block) items in segment-major order from a device counter; an item
// waits (bounded) until the previous segment of its block is published, and
// takes its first observation from the replay ring (the entry the previous
// segment wrote), or scans it when there is no ring.  sync: [nblk] segments
// done per block, item counter, abort word; zero at launch.
template <bool kFast>
__global__ void __launch_bounds__(kQtThreads, 1)
    k_rollout_q_tc(const __grid_constant__ DevCfg c, SimPtrs p, const uint8_t* __restrict__ img,
                   const uint8_t* __restrict__ timg, ImgLayout L, int K, const float* __restrict__ eps, ReplayDev rp,
                   int use_replay, const int* __restrict__ order, int seg, unsigned* __restrict__ sync,
                   float* __restrict__ obs_out, float* __restrict__ obs_seq, uint8_t* __restrict__ act_seq,
                   float* __restrict__ rew_seq, uint8_t* __restrict__ done_seq) {
  extern __shared__ __align__(1024) uint8_t tsm[];
  __shared__ uint64_t bar_ld[2], bar_mm[2], bar_layer;
  __shared__ uint32_t tslot;
  __shared__ int item_sh;
  __shared__ int ok_sh;
  __shared__ int greedy[kQtEnvs];
  __shared__ uint8_t act_sh[kQtEnvs];
  __shared__ int scan_next, row_heavy, row_light;
  __shared__ uint8_t row_list[kQtEnvs];
  __shared__ Env env_sh[kQtEnvs];                 // the tile's env states within a segment
  __shared__ unsigned long long akey_sh[kQtEnvs];  // their action-stream keys
  __shared__ float sb1[kHid], sb2[kHid], sb3[kOutPad];
  const QtSmem T = qt_smem();
  const TcImg G = tc_img(L.k1);
  uint8_t* hx = tsm + T.hx;  // the input tile
  uint8_t* w3s = tsm + T.w3;
  MotionRec* rec = reinterpret_cast<MotionRec*>(tsm + T.hx + kQtRecOff);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long n = c.n_envs;
  const int nblk = (int)((n + kQtEnvs - 1) / kQtEnvs);
  const int seglen = seg > 0 ? seg : K;
  const int nseg = (K + seglen - 1) / seglen;
  const long long nitems = (long long)nblk * nseg;
  const uint32_t w1h_bytes = 128u * (uint32_t)L.k1 * 2u, w2q_bytes = 64u * kHid * 2u;
  for (int i = tid; i < kHid; i += kQtThreads) {
    sb1[i] = __ldg(reinterpret_cast<const float*>(img + L.b1) + i);
    sb2[i] = __ldg(reinterpret_cast<const float*>(img + L.b2) + i);
  }
  if (tid < kOutPad) sb3[tid] = __ldg(reinterpret_cast<const float*>(img + L.b3) + tid);
  for (int i = tid; i < (int)(16u * kHid * 2u / 16u); i += kQtThreads)
    reinterpret_cast<uint4*>(w3s)[i] = __ldg(reinterpret_cast<const uint4*>(timg + G.w3) + i);
  if (warp == 0) tmem_alloc(&tslot, 512);
  if (tid == 0) {
    for (int b = 0; b < 2; ++b) {
      mbar_init(&bar_ld[b], 1);
      mbar_init(&bar_mm[b], 1);
    }
    mbar_init(&bar_layer, 1);
    ok_sh = 1;
  }
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tacc = tslot, tacc2 = tacc + 256u;
  QtStream S;  // meaningful in thread 0
  S.ld = bar_ld;
  S.mm = bar_mm;
  S.buf[0] = tsm + T.b0;
  S.buf[1] = tsm + T.b1;
  S.pl[0] = S.pl[1] = S.pm[0] = S.pm[1] = 0u;
  S.ld_out[0] = S.ld_out[1] = S.mm_out[0] = S.mm_out[1] = false;
  S.ok = true;
  uint32_t player = 0;  // phase of the layer barrier
  bool layer_out = false, ok = true;
  const unsigned long long rbase = use_replay ? *rp.steps : 0ull;
  const int B = c.B;
  const int row0 = warp * 4;
  for (int iter = 0;; ++iter) {
    // ---- the next item: a segment of one 128-env block ----
    if (tid == 0) {
      long long it;
      if (!sync)
        it = iter == 0 ? (long long)blockIdx.x : nitems;
      else
        it = (!ok || __ldcg(&sync[nblk + 1])) ? nitems : (long long)atomicAdd(&sync[nblk], 1u);
      if (sync && it < nitems && it >= nblk) {
        const unsigned need = (unsigned)(it / nblk);
        unsigned w = 0;
        while (qt_ld_acquire(&sync[it % nblk]) < need) {
          if (++w > kQtWaitIters || qt_ld_acquire(&sync[nblk + 1])) {
            atomicOr(p.status, SG_DEV_TIMEOUT);
            atomicExch(&sync[nblk + 1], 1u);
            it = nitems;
            break;
          }
          __nanosleep(256);
        }
      }
      item_sh = (ok && it < nitems) ? (int)it : -1;
    }
    __syncthreads();
    const int item = item_sh;
    __syncthreads();  // item_sh is rewritten by the next iteration
    if (item < 0) break;
    const int blk = item % nblk, s0 = (item / nblk) * seglen, s1 = min(K, s0 + seglen);
    // the segment's first observation: four rows per warp (row0 .. row0 + 3)
    const int slot0 = blk * kQtEnvs + row0;
    const int nv = max(0, min(4, (int)n - slot0));
    const bool live = lane < nv;
    const int env = live ? order[slot0 + lane] : 0;
    // the env-step lanes: row tid of the tile
    const bool slive = tid < kQtEnvs && (long long)blk * kQtEnvs + tid < n;
    const int senv = slive ? order[blk * kQtEnvs + tid] : 0;
    // the tile: zero (padding columns, rows without an env), then the first
    // observation of the segment
    for (int i = tid; i < kQtEnvs * L.k1 / 8; i += kQtThreads)
      reinterpret_cast<uint4*>(hx)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    if (s0 > 0 && use_replay) {
      const long long sl = (long long)((rbase + (unsigned long long)s0) % (unsigned long long)rp.slots);
      for (int e = 0; e < nv; ++e) {
        const int ie = __shfl_sync(kFull, env, e);
        const float* src = rp.s + (sl * rp.n_envs + ie) * rp.obs_dim;
        for (int k = lane; k < c.obs_dim; k += 32)
          *reinterpret_cast<bf16*>(hx + kmajor_offset(row0 + e, k, kQtEnvs)) = __float2bfloat16_rn(__ldcg(src + k));
      }
    } else {
      if (live) lane_observe(c, p, env, load_env_l2(p, env), rec + row0 + lane);
      __syncwarp();
      for (int e = 0; e < nv; ++e) {
        const MotionRec* r = rec + row0 + e;
        const uint4 w0 = rec_word<false>(r, 0), w1 = rec_word<false>(r, 1);
        const RecScan q = rec_scan(c, rec_word<false>(r, 3), rec_word<false>(r, 4), lane);
        ObsRegs o;
        scan_pose<false, kFast>(c, q.sm, q.nb, q.off0, q.off1, __uint_as_float(w0.x), __uint_as_float(w0.y),
                                __uint_as_float(w0.z), __uint_as_float(w0.w), ((uint64_t)w1.y << 32) | w1.x, q.k0, lane,
                                o.b0, o.b1);
        o.ex = lane < 5 ? r->ex[lane] : 0.0f;
        qt_obs_to_tile(hx, row0 + e, o.b0, o.b1, o.ex, B, lane);
        if (use_replay) {
          const long long sl = (long long)((rbase + (unsigned long long)s0) % (unsigned long long)rp.slots);
          write_obs(rp.s + (sl * rp.n_envs + r->env) * rp.obs_dim, o, B, lane);
        }
      }
    }
    fence_async_smem();
    // ring slot of step t
    int slot = use_replay ? (int)((rbase + (unsigned long long)s0) % (unsigned long long)rp.slots) : 0;
    for (int t = s0; t < s1; ++t) {
      // ---- the network on the tile of observations t ----
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
      // layer 1: two 128-unit halves of W1 through the buffers (normally
      // loaded during the previous env steps), then the two K-half pieces of
      // W2's first 128 rows into them as soon as each half's MMAs are done
      if (tid == 0) {
        if (!S.ld_out[0]) S.load(0, timg + G.w1h, w1h_bytes);
        if (!S.ld_out[1]) S.load(1, timg + G.w1h + w1h_bytes, w1h_bytes);
        S.mma(0, tacc, hx, 0u, 128, L.k1, &bar_layer, false);
        S.mma(1, tacc + 128u, hx, 0u, 128, L.k1, &bar_layer, true);
        S.load(0, timg + G.w2a, w2q_bytes);
        S.load(1, timg + G.w2a + w2q_bytes, w2q_bytes);
        if (!S.ok) ok_sh = 0;
      }
      layer_out = true;
      __syncthreads();  // ok_sh as thread 0 left it
      ok = __syncthreads_and(ok_sh && mbar_wait(&bar_layer, player, kTcTries));
      if (!ok) break;
      player ^= 1u;
      layer_out = false;
      tc_fence_after();
      qt_epilogue(tacc, sb1, warp);
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
      // layer 2: two 128-unit halves (N = 128: an MMA of M = 128 costs about
      // as much at N = 64 as at 128), each from the two 32 KB K-half pieces
      // of its rows through the buffers (piece c: K steps 8 c .. 8 c + 7);
      // the second half's pieces are both in flight before either is needed
      if (tid == 0) {
        S.mma(0, tacc2, nullptr, tacc, 128, kHid / 2, &bar_layer, false, 0, false);
        S.mma(1, tacc2, nullptr, tacc, 128, kHid / 2, &bar_layer, false, 8, true);
        S.load(0, timg + G.w2b, w2q_bytes);
        S.load(1, timg + G.w2b + w2q_bytes, w2q_bytes);
        S.mma(0, tacc2 + 128u, nullptr, tacc, 128, kHid / 2, &bar_layer, false, 0, false);
        S.mma(1, tacc2 + 128u, nullptr, tacc, 128, kHid / 2, &bar_layer, true, 8, true);
        if (!S.ok) ok_sh = 0;
      }
      layer_out = true;
      __syncthreads();  // ok_sh as thread 0 left it
      ok = __syncthreads_and(ok_sh && mbar_wait(&bar_layer, player, kTcTries));
      if (!ok) break;
      player ^= 1u;
      layer_out = false;
      tc_fence_after();
      qt_epilogue(tacc2, sb2, warp);
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
      // head (W3 resident), and the next step's W1 halves into the buffers
      if (tid == 0) {
        tc_fence_after();
        const uint32_t idesc = idesc_bf16_f32(kQtEnvs, 16);
        const uint32_t sw = smem_u32(w3s);
        for (int ks = 0; ks < kHid / 16; ++ks)
          tc_mma_bf16_ta(tacc + 16u, tacc2 + qt_a_col(ks), smem_desc(sw + (uint32_t)ks * 2 * 256, 256, 128), idesc,
                         ks > 0 ? 1u : 0u);
        tc_commit(&bar_layer);
        if (t + 1 < s1) {
          S.load(0, timg + G.w1h, w1h_bytes);
          S.load(1, timg + G.w1h + w1h_bytes, w1h_bytes);
        }
        if (!S.ok) ok_sh = 0;
      }
      layer_out = true;
      __syncthreads();  // ok_sh as thread 0 left it
      ok = __syncthreads_and(ok_sh && mbar_wait(&bar_layer, player, kTcTries));
      if (!ok) break;
      player ^= 1u;
      layer_out = false;
      if (warp < 4) {
        float v[32];
        tc_fence_after();
        tmem_ld32(tacc + 16u + ((uint32_t)(warp * 32) << 16), v);
        float o[kOut];
#pragma unroll
        for (int j = 0; j < kOut; ++j) o[j] = v[j] + sb3[j];
        greedy[warp * 32 + lane] = (int)greedy_action(o, nullptr, L.plain);
      }
      // the next input tile starts from zero
      for (int i = tid; i < kQtEnvs * L.k1 / 8; i += kQtThreads)
        reinterpret_cast<uint4*>(hx)[i] = make_uint4(0u, 0u, 0u, 0u);
      if (tid == 0) scan_next = row_heavy = row_light = 0;
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
      // ---- the env steps of the tile: one env per lane of the first warps ----
      if (slive) {
        // the state stays in shared memory between the steps of a segment
        // (stored to global memory at its end)
        Env s = t == s0 ? load_env_l2(p, senv) : env_sh[tid];
        if (t == s0) akey_sh[tid] = sm_at(sm_at(c.seed, kStreamAction), (uint64_t)senv);
        // VEM (Sec. 3.1.1): with probability eps_i the random action of step t
        const uint64_t h = sm_at(akey_sh[tid], (uint64_t)s.t);
        const uint32_t ra = (uint32_t)(sm_at(h, 0ull) >> 32) % (uint32_t)c.n_actions;
        const bool explore = u24_hi(sm_at(h, 1ull)) < __ldg(eps + senv);
        const uint32_t a = explore ? ra : (uint32_t)greedy[tid];
        lane_motion<false>(c, p, senv, s, a, rec + tid, nullptr);
        env_sh[tid] = s;
        act_sh[tid] = (uint8_t)a;
        if (act_seq) act_seq[(long long)t * n + senv] = (uint8_t)a;
      }
      const int rows = (int)min((long long)kQtEnvs, n - (long long)blk * kQtEnvs);
      if (tid < kQtEnvs) {
        // the rows in the order they are handed out: two-beam lanes and resets
        // first, so that no long row is the last
        const bool heavy = slive && ((rec[tid].nbk & 0xFFu) > 32u || (rec[tid].done & 7u));
        const unsigned hm = __ballot_sync(kFull, heavy), lm = __ballot_sync(kFull, slive && !heavy);
        const unsigned below = (1u << lane) - 1u;
        int hb = 0, lb = 0;
        if (lane == 0) {
          hb = atomicAdd(&row_heavy, __popc(hm));
          lb = atomicAdd(&row_light, __popc(lm));
        }
        hb = __shfl_sync(kFull, hb, 0) + __popc(hm & below);
        lb = __shfl_sync(kFull, lb, 0) + __popc(lm & below);
        if (slive) row_list[heavy ? hb : rows - 1 - lb] = (uint8_t)tid;
      }
      // every record of the tile is written; the scans (one or two per env,
      // 16 to 64 beams) are handed out row by row through a shared counter,
      // so that no warp waits at the next step's barrier for a slow one
      __syncthreads();
      const long long slot_t = slot, slot_n = slot + 1 == rp.slots ? 0 : slot + 1;
      slot = (int)slot_n;
      for (;;) {
        int e = 0;
        if (lane == 0) e = atomicAdd(&scan_next, 1);
        e = __shfl_sync(kFull, e, 0);
        if (e >= rows) break;
        e = row_list[e];
        const MotionRec* r = rec + e;
        const uint4 w1 = rec_word<false>(r, 1), w3 = rec_word<false>(r, 3);
        const int ie = (int)w3.w;
        const RecScan q = rec_scan(c, w3, rec_word<false>(r, 4), lane);
        uint32_t d = w1.w;
        ObsRegs o;
        float mn;
        {
          const uint4 w0 = rec_word<false>(r, 0);
          const float x = __uint_as_float(w0.x), y = __uint_as_float(w0.y);
          if (d & kRecSlow) {
            const MapDesc m = p.maps[p.env_map[ie]];
            d = (d & 7u) | (collide_rows_warp(c, m, p.atlas + m.word_off, x, y, lane) ? 1u : 0u);
          }
          mn = scan_pose<false, kFast>(c, q.sm, q.nb, q.off0, q.off1, x, y, __uint_as_float(w0.z),
                                       __uint_as_float(w0.w), ((uint64_t)w1.y << 32) | w1.x, q.k0, lane, o.b0, o.b1);
        }
        o.ex = lane < 5 ? r->ex[lane] : 0.0f;
        const float rw = (d & 1u) ? -10.0f : (d & 2u) ? 75.0f : reward_finish(c, __uint_as_float(w1.z), mn);
        if (use_replay) {
          // transition t: s2 is the observation after the step, before a reset
          const long long en = slot_t * rp.n_envs + ie;
          write_obs(rp.s2 + en * rp.obs_dim, o, B, lane);
          if (lane == 0) {
            rp.a[en] = act_sh[e];
            rp.r[en] = rw;
            rp.term[en] = (d & 3u) ? 1 : 0;
          }
        }
        if (lane == 0) {
          if (rew_seq) rew_seq[(long long)t * n + ie] = rw;
          if (done_seq) done_seq[(long long)t * n + ie] = (uint8_t)d;
        }
        if (d) {
          // AutoReset (Sec. 3.2.5): a new episode, observed at its step 0
          const MapDesc m = p.maps[p.env_map[ie]];
          const Layout L2 = layout_of(c, m);
          Env s;
          s.t = env_sh[e].t;
          const uint32_t ep = env_sh[e].ep_id + 1u;
          __syncwarp();
          reset_env(c, m, p.clr + m.clr_off, L2, sm_at(sm_at(c.seed, kStreamReset), (uint64_t)ie), s, ep, lane);
          if (lane == 0) env_sh[e] = s;
          o.ex = obs_extra(c, L2, s, goal_frame(L2, s), lane);
          scan_pose<false, kFast>(c, q.sm, q.nb, q.off0, q.off1, s.x, s.y, s.phi, s.sigma,
                                  sm_at(sm_at(sm_at(c.seed, kStreamNoise), (uint64_t)ie), (uint64_t)s.ep_id << 32),
                                  lane_scan_start(c, p, m, s.x, s.y), lane, o.b0, o.b1);
        }
        // the observation t + 1: the next tile row, the outputs, the next ring entry's s
        qt_obs_to_tile(hx, e, o.b0, o.b1, o.ex, B, lane);
        if (obs_seq) write_obs(obs_seq + ((long long)t * n + ie) * c.obs_dim, o, B, lane);
        if (t == K - 1 && obs_out) write_obs(obs_out + (long long)ie * c.obs_dim, o, B, lane);
        if (use_replay && t + 1 < K) write_obs(rp.s + (slot_n * rp.n_envs + ie) * rp.obs_dim, o, B, lane);
      }
      fence_async_smem();
    }
    if (!ok) {
      if (tid == 0) atomicOr(p.status, SG_DEV_TIMEOUT);
      break;  // CTA-uniform: the launch's outputs from here on are incomplete
    }
    __syncthreads();  // the last step's resets are in env_sh
    if (slive) store_env(p, senv, env_sh[tid]);
    if (!sync) break;
    // publish the block's segment: its env state and ring entries are stored
    __threadfence();
    __syncthreads();
    if (tid == 0) qt_st_release(&sync[blk], (unsigned)(s0 / seglen + 1));
  }
  // free the tensor memory once nothing is in flight (bounded waits)
  if (tid == 0) S.drain();
  if (layer_out && ok_sh) mbar_wait(&bar_layer, player, kTcTries);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tmem_free(tacc, 512);
  if (tid == 0) replay_advance(rp, use_replay, K);
}

// ------------------------------------------------------------ learner
// Why a TD step produced no update (bits of a device word cleared at the
// start of every step): a weight-image copy did not complete within its
// bounded wait, or a sample's action index is outside the action table.
// The update then writes NaN loss and gradient and leaves the parameters, the
// Adam moments and the image untouched; the step count does not advance.
constexpr unsigned kTdFailCopy = 1u;
constexpr unsigned kTdFailAction = 2u;
// x mod d with inv = floor((2^64 - 1) / d): the quotient from the high product
// is at most two too small (x / d - x inv / 2^64 < 2).
__device__ __forceinline__ unsigned long long mod_inv(unsigned long long x, unsigned long long d,
                                                      unsigned long long inv) {
  unsigned long long r = x - __umul64hi(x, inv) * d;
  if (r >= d) r -= d;
  if (r >= d) r -= d;
  return r;
}
// The draw of sample i of optimiser step `tstep`.
__device__ __forceinline__ uint64_t sample_hash(unsigned long long seed, unsigned long long tstep, int i) {
  return sm_at(sm_at(sm_at(sm_at(seed, kStreamSample), tstep), (uint64_t)i), 0ull);
}
// Ring entry of a sample with draw h and st steps recorded: uniform over the
// V = min(steps, slots - reserve) most recently completed slots, so that a
// rollout running concurrently (which writes the next slots) is never read.
// With j = h mod (V n_envs): slot = (steps - 1 - j / n_envs) mod slots,
// env = j mod n_envs.  Whoever reads parts of one sample uses one value of st
// (offer_steps): the counter may change between two loads.
__device__ __forceinline__ long long sample_entry(uint64_t h, unsigned long long st, const ReplayDev& rp) {
  const unsigned long long usable = (unsigned long long)(rp.slots - rp.reserve);
  const unsigned long long V = st < usable ? st : usable;
  if (V == 0) return -1;
  // the ring holds at most 2^31 entries, so j and its quotient fit 32 bits;
  // back < V <= slots, so one correction replaces the modulo of the difference
  const uint32_t n = (uint32_t)rp.n_envs;
  const unsigned long long D = V * (unsigned long long)n;
  const uint32_t j = (uint32_t)(V == usable ? mod_inv(h, D, rp.inv_full) : h % D);
  const uint32_t back = j / n, last = (uint32_t)mod_inv(st - 1ull, (unsigned long long)rp.slots, rp.inv_slots);
  const uint32_t slot = last >= back ? last - back : last + (uint32_t)rp.slots - back;
  const long long e = (long long)slot * n + (j - back * n);
  return SG_IN_BOUNDS(e >= 0 && e < (long long)rp.slots * rp.n_envs) ? e : -1;
}

// Gather 16 rows of a ring array into a BF16 tile (zero padded).
__device__ __forceinline__ void gather_tile(bf16* X, int ld1, const float* __restrict__ src, const int* rows,
                                            int obs_dim, int warp, int lane) {
  const int e = rows[warp];
  for (int k = lane; k < ld1; k += 32) {
    const float v = (e >= 0 && k < obs_dim) ? src[(long long)e * obs_dim + k] : 0.0f;
    X[warp * ld1 + k] = __float2bfloat16_rn(v);
  }
}

// Loss and gradient of 16 samples per CTA.  Forward of Q_online(s) keeping
// the activations, delta = Q(s, a) - y, dL/dQ(s,a) = clip(delta, -1, 1) / B,
// back through the dueling combine, W3, ReLU, W2, ReLU, W1.  The CTA's
// parameter gradient (and Huber sum) goes to its own row of `partial`, so
// that the reduction order is fixed.
__global__ void __launch_bounds__(kThreads, 1)
    k_td_grad(const uint8_t* __restrict__ img, ImgLayout L, ParamLayout P, ReplayDev rp,
              const int* __restrict__ idx, const float* __restrict__ y, int batch, float* __restrict__ partial,
              unsigned* __restrict__ fail) {
  extern __shared__ __align__(16) uint8_t smem[];
  uint8_t* sw = smem;
  bf16* S = reinterpret_cast<bf16*>(smem + L.bytes);
  bf16* H1 = S + kTile * L.ld1;
  bf16* H2 = H1 + kTile * kLdh;  // becomes dZ2 after the head gradient
  bf16* D1 = H2 + kTile * kLdh;  // dZ1
  float* O = reinterpret_cast<float*>(D1 + kTile * kLdh);
  float* DO = O + kTile * kOutPad;  // dL/d(head outputs) [16][8]
  __shared__ int rows[kTile];
  __shared__ float hub[kTile];
  __shared__ uint64_t bar_img;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, q = lane & 3;
  const int i = blockIdx.x * kTile + warp;
  if (lane == 0) rows[warp] = i < batch ? idx[i] : -1;
  if (threadIdx.x == 0) mbar_init(&bar_img, 1);
  __syncthreads();
  if (!stage_image_bulk(sw, img, L.bytes, &bar_img, 0u, kTcTries)) {
    // the image copy did not complete: no gradient (k_grad_sum reads the
    // flag); one more bounded wait for the copy before the CTA exits
    if (threadIdx.x == 0) {
      atomicOr(fail, kTdFailCopy);
      mbar_wait(&bar_img, 0u, kTcTries);
    }
    return;
  }
  gather_tile(S, L.ld1, rp.s, rows, rp.obs_dim, warp, lane);
  __syncthreads();
  const QW w = qw_at(sw, L);
  mlp_tile(w, S, H1, H2, O, warp, lane);
  // dL/dQ and back through Q_a = V + A_a - mean(A)
  if (lane == 0) {
    float qv[5];
    greedy_action(O + warp * kOutPad, qv, L.plain);
    const int e = rows[warp];
    float gq = 0.0f, hl = 0.0f;
    if (e >= 0) {
      int a = rp.a[e];
      float d;
      if (a >= 5) {
        // outside the action table: no loss term, and no update this step
        atomicOr(fail, kTdFailAction);
        a = 0;
        d = __int_as_float(0x7fc00000);
      } else {
        d = qv[a] - y[i];
      }
      const float ad = fabsf(d);
      hl = ad <= 1.0f ? 0.5f * d * d : ad - 0.5f;
      // a NaN target (a failed target copy) stays NaN through the clip
      gq = (isnan(d) ? d : fminf(fmaxf(d, -1.0f), 1.0f)) / (float)batch;
      if (L.plain) {
        for (int k = 0; k < 5; ++k) DO[warp * kOutPad + k] = k == a ? gq : 0.0f;
        DO[warp * kOutPad + 5] = 0.0f;
      } else {
        DO[warp * kOutPad + 0] = gq;
        for (int k = 0; k < 5; ++k) DO[warp * kOutPad + 1 + k] = (k == a ? gq : 0.0f) - gq / 5.0f;
      }
    } else {
      for (int k = 0; k < 6; ++k) DO[warp * kOutPad + k] = 0.0f;
    }
    DO[warp * kOutPad + 6] = 0.0f;
    DO[warp * kOutPad + 7] = 0.0f;
    hub[warp] = hl;
  }
  __syncthreads();
  float* pg = partial + (long long)blockIdx.x * partial_stride(P.total);
  // head gradient on the CUDA cores: dW3[o][j] = sum_s DO[s][o] H2[s][j],
  // db3[o] = sum_s DO[s][o]; dH2 = DO W3 (BF16 W3 as in the forward), masked
  // by the ReLU into dZ2 (written over H2 after a barrier)
  const int tid = threadIdx.x;
  float dz2v[kTile];
  if (tid < kHid) {
    const int j = tid;
    float acc[kOut];
    for (int o = 0; o < kOut; ++o) acc[o] = 0.0f;
    for (int s = 0; s < kTile; ++s) {
      const float h = __bfloat162float(H2[s * kLdh + j]);
      for (int o = 0; o < kOut; ++o) acc[o] += DO[s * kOutPad + o] * h;
    }
    for (int o = 0; o < kOut; ++o) pg[P.w3 + o * kHid + j] = acc[o];
    float db2 = 0.0f;
    for (int s = 0; s < kTile; ++s) {
      float dh = 0.0f;
      for (int o = 0; o < kOut; ++o) dh += DO[s * kOutPad + o] * __bfloat162float(w.W3[o * kLdh + j]);
      const float v = __bfloat162float(H2[s * kLdh + j]) > 0.0f ? dh : 0.0f;
      dz2v[s] = v;
      db2 += v;
    }
    pg[P.b2 + j] = db2;
  }
  if (tid < kOut) {
    float acc = 0.0f;
    for (int s = 0; s < kTile; ++s) acc += DO[s * kOutPad + tid];
    pg[P.b3 + tid] = acc;
  }
  if (tid == 0) {
    float acc = 0.0f;
    for (int s = 0; s < kTile; ++s) acc += hub[s];
    pg[P.total] = acc;
  }
  __syncthreads();
  if (tid < kHid)
    for (int s = 0; s < kTile; ++s) H2[s * kLdh + tid] = __float2bfloat16_rn(dz2v[s]);
  __syncthreads();
  bf16* DZ2 = H2;
  // dW2[m][n] = sum_s dZ2[s][m] H1[s][n]: M = N = 256, K = 16 -> 512 tiles,
  // 32 per warp (A = dZ2^T, B = H1, both stored sample-major)
  for (int t = warp; t < 16 * 32; t += kTile) {
    const int m0 = (t >> 5) * 16, n0 = (t & 31) * 8;
    uint32_t a[4], b0, b1;
    load_a_col(a, DZ2, kLdh, m0, 0, lane);
    load_b_row(b0, b1, H1, kLdh, 0, n0, lane);
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    mma_bf16(acc, a, b0, b1);
    float* dst = pg + P.w2;
    *reinterpret_cast<float2*>(dst + (m0 + g) * kHid + n0 + 2 * q) = make_float2(acc[0], acc[1]);
    *reinterpret_cast<float2*>(dst + (m0 + g + 8) * kHid + n0 + 2 * q) = make_float2(acc[2], acc[3]);
  }
  // dH1 = dZ2 W2 (B = W2 stored [out][in] -> "row" layout), masked -> dZ1
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    const int n0 = 8 * warp + 128 * half;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    for (int k0 = 0; k0 < kHid; k0 += 16) {
      uint32_t a[4], b0, b1;
      load_a_row(a, DZ2, kLdh, 0, k0, lane);
      load_b_row(b0, b1, w.W2, kLdh, k0, n0, lane);
      mma_bf16(acc, a, b0, b1);
    }
    const int n = n0 + 2 * q;
    const bool m00 = __bfloat162float(H1[g * kLdh + n]) > 0.f, m01 = __bfloat162float(H1[g * kLdh + n + 1]) > 0.f;
    const bool m10 = __bfloat162float(H1[(g + 8) * kLdh + n]) > 0.f;
    const bool m11 = __bfloat162float(H1[(g + 8) * kLdh + n + 1]) > 0.f;
    *reinterpret_cast<uint32_t*>(D1 + g * kLdh + n) = pack_bf16x2(m00 ? acc[0] : 0.f, m01 ? acc[1] : 0.f);
    *reinterpret_cast<uint32_t*>(D1 + (g + 8) * kLdh + n) = pack_bf16x2(m10 ? acc[2] : 0.f, m11 ? acc[3] : 0.f);
    // db1 needs the FP32 values: reduce the 16 rows of this fragment column
    float c0 = (m00 ? acc[0] : 0.f) + (m10 ? acc[2] : 0.f);
    float c1 = (m01 ? acc[1] : 0.f) + (m11 ? acc[3] : 0.f);
    for (int off = 4; off < 32; off <<= 1) {
      c0 += __shfl_xor_sync(kFull, c0, off);
      c1 += __shfl_xor_sync(kFull, c1, off);
    }
    if (g == 0) {
      pg[P.b1 + n] = c0;
      pg[P.b1 + n + 1] = c1;
    }
  }
  __syncthreads();
  // dW1[m][k] = sum_s dZ1[s][m] S[s][k]: M = 256, N = k1, K = 16
  const int nt1 = L.k1 / 8;
  for (int t = warp; t < 16 * nt1; t += kTile) {
    const int m0 = (t / nt1) * 16, n0 = (t % nt1) * 8;
    uint32_t a[4], b0, b1;
    load_a_col(a, D1, kLdh, m0, 0, lane);
    load_b_row(b0, b1, S, L.ld1, 0, n0, lane);
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    mma_bf16(acc, a, b0, b1);
    float* dst = pg + P.w1;
    const int c0 = n0 + 2 * q, c1 = c0 + 1;
    if (c0 < L.n_in) {
      dst[(m0 + g) * L.n_in + c0] = acc[0];
      dst[(m0 + g + 8) * L.n_in + c0] = acc[2];
    }
    if (c1 < L.n_in) {
      dst[(m0 + g) * L.n_in + c1] = acc[1];
      dst[(m0 + g + 8) * L.n_in + c1] = acc[3];
    }
  }
}

// ------------------------------------------------------- parameter update
// Everything that follows the gradient of a TD step, per parameter: Adam
// (Kingma & Ba) on the FP32 master, the BF16 entry in the image and in the
// tensor cores' copies, and on a target step the target network's copies.
// The last CTA of the launch advances the step count and clears the step's
// failure word, so that nothing else has to run before the next step.  As
// five launches (reduce + Adam, tensor-core copy, step count, target check, a
// memset) the same work cost a batch-256 step 25 of its 57 us.
struct TdUpdate {
  float* th;
  float* m;
  float* v;
  float* tgt;
  uint8_t* img;
  uint8_t* img_t;
  uint8_t* tc;
  uint8_t* tc_t;
  unsigned long long* step;
  unsigned* fail;
  unsigned* tick;            // CTAs that are done (0 between launches)
  float lr;
  int every;                 // target period (optimiser steps), <= 0: never
  float* loss;
  float* grad;
  int batch;
  ParamLayout P;
  ImgLayout L;
};
// What a launch does: read once per thread.  A failed step changes nothing,
// and its unchanged step count decides about the target.
struct UpdRun {
  bool adam, sync;
  bool sync_failed;  // sync of a failed step
  float d1, d2;      // 1 - beta1^t, 1 - beta2^t
};
constexpr float kBeta1 = 0.9f, kBeta2 = 0.999f, kAdamEps = 1e-8f;

__device__ __forceinline__ UpdRun upd_begin(const TdUpdate& u) {
  UpdRun r = {false, false, false, 1.0f, 1.0f};
  if (u.lr != 0.0f) {
    const unsigned long long st = *u.step;
    const float t = (float)(st + 1ull);
    r.adam = true;
    r.d1 = 1.0f - powf(kBeta1, t);
    r.d2 = 1.0f - powf(kBeta2, t);
    if (u.every > 0) {
      const unsigned long long rem = st % (unsigned long long)u.every;
      r.sync_failed = rem == 0ull;
      r.sync = rem + 1ull == (unsigned long long)u.every;
    }
  }
  return r;
}
__device__ __forceinline__ void upd_fail(bool failed, UpdRun& r) {
  if (!failed) return;
  r.adam = false;
  r.sync = r.sync_failed;
}

// The new value of parameter i from its gradient (th, m, v: its old values).
__device__ __forceinline__ float upd_adam(const TdUpdate& u, const UpdRun& r, int i, float g, float th, float m,
                                          float v) {
  const float mi = kBeta1 * m + (1.0f - kBeta1) * g;
  const float vi = kBeta2 * v + (1.0f - kBeta2) * g * g;
  u.m[i] = mi;
  u.v[i] = vi;
  const float mh = mi / r.d1;
  const float vh = vi / r.d2;
  const float nth = th - u.lr * mh / (sqrtf(vh) + kAdamEps);
  u.th[i] = nth;
  return nth;
}
__device__ __forceinline__ void upd_grad(const TdUpdate& u, int i, float g) {
  if (!u.grad) return;
  const int j = u.L.plain ? paper_index(i, u.P, u.L.n_in) : i;
  if (j >= 0) u.grad[j] = g;
}

// Elements (r, k .. k + kN - 1) of a weight matrix (1, 2 or 3), one 2- or
// 4-byte word, in the image and in every tensor-core copy (k even when kN = 2).
template <int kW, int kN>
__device__ __forceinline__ void upd_image(uint8_t* img, uint8_t* tc, const ImgLayout& L, int r, int k, float a,
                                          float b) {
  const TcImg T = tc_img(L.k1);
  const uint32_t v = pack_bf16x2(a, b);
  auto put = [&](uint8_t* at) {
    if (kN == 2)
      *reinterpret_cast<uint32_t*>(at) = v;
    else
      *reinterpret_cast<uint16_t*>(at) = (uint16_t)v;
  };
  if (kW == 1) {
    put(img + L.w1 + (r * L.ld1 + k) * 2);
    put(tc + T.w1 + kmajor_offset(r, k, kHid));
    put(tc + T.w1h + (uint32_t)((r >> 7) * 128 * L.k1 * 2) + kmajor_offset(r & 127, k, 128));
  } else if (kW == 2) {
    put(img + L.w2 + (r * kLdh + k) * 2);
    put(tc + (r < 128 ? T.w2a : T.w2b) + kmajor_offset(r & 127, k, 128));
    put(tc + T.w2f + kmajor_offset(r, k, kHid));
  } else {
    put(img + L.w3 + (r * kLdh + k) * 2);
    put(tc + T.w3 + kmajor_offset(r, k, 16));
  }
}
template <int kW, int kN>
__device__ __forceinline__ void upd_images(const TdUpdate& u, const UpdRun& r, int row, int k, float a, float b) {
  if (r.adam) upd_image<kW, kN>(u.img, u.tc, u.L, row, k, a, b);
  if (r.sync) upd_image<kW, kN>(u.img_t, u.tc_t, u.L, row, k, a, b);
}
// The image entry of bias i.
__device__ __forceinline__ void upd_bias(const TdUpdate& u, const UpdRun& r, int i, float a) {
  const ParamLayout& P = u.P;
  const int at = i < P.w2 ? u.L.b1 + (i - P.b1) * 4 : i < P.w3 ? u.L.b2 + (i - P.b2) * 4 : u.L.b3 + (i - P.b3) * 4;
  if (r.adam) *reinterpret_cast<float*>(u.img + at) = a;
  if (r.sync) *reinterpret_cast<float*>(u.img_t + at) = a;
}
// Parameter i on its own (gradient g; th, m, v: its old values): everything
// above for one element.
__device__ __forceinline__ void upd_one(const TdUpdate& u, const UpdRun& r, int i, float g, float th, float m,
                                        float v) {
  upd_grad(u, i, g);
  if (!r.adam && !r.sync) return;
  float a = th;
  if (r.adam) a = upd_adam(u, r, i, g, th, m, v);
  if (r.sync) u.tgt[i] = a;
  const ParamLayout& P = u.P;
  if (i < P.b1) {
    upd_images<1, 1>(u, r, i / u.L.n_in, i % u.L.n_in, a, a);
  } else if (i >= P.w2 && i < P.b2) {
    upd_images<2, 1>(u, r, (i - P.w2) / kHid, (i - P.w2) % kHid, a, a);
  } else if (i >= P.w3 && i < P.b3) {
    upd_images<3, 1>(u, r, (i - P.w3) / kHid, (i - P.w3) % kHid, a, a);
  } else {
    upd_bias(u, r, i, a);
  }
}
// Every CTA, at its end: the last one advances the step count (of a step that
// changed the parameters) and clears the failure word.
__device__ __forceinline__ void upd_end(const TdUpdate& u, bool failed) {
  __syncthreads();  // this CTA's reads of *step and *fail are done
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(u.tick, 1u) == gridDim.x - 1u) {
      if (u.lr != 0.0f && !failed) *u.step += 1ull;
      *u.fail = 0u;
      *u.tick = 0u;
    }
  }
}

// Gradient rows (one per CTA of the gradient kernel) summed in row order,
// thread per parameter: the allocation-free gradient.
__global__ void __launch_bounds__(256) k_grad_sum(TdUpdate u, const float* __restrict__ partial, int nblk) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i > u.P.total) return;
  const long long ld = partial_stride(u.P.total);
  float g = 0.0f;
#pragma unroll 8
  for (int b = 0; b < nblk; ++b) g += partial[(long long)b * ld + i];
  if (*u.fail) g = __int_as_float(0x7fc00000);
  if (i < u.P.total)
    upd_grad(u, i, g);
  else if (u.loss)
    *u.loss = g / (float)u.batch;
}

// --------------------------------------------------- mma.sync learner
// Small batches, in 16-sample tiles.  A cluster of three CTAs takes a tile:
// rank 0 the forward on s, ranks 1 and 2 those of the online and the target
// network on s' (each CTA holds its network's image for all its tiles); the
// next-state Q-values go to rank 0 through distributed shared memory, which
// forms the targets and runs the backward pass.  The weight gradients are
// sums over the batch of outer products, so rank 0 stores its operands
// (dZ2, H1, dZ1, X: 8 KB each at most) as the fragments that k_td_update's
// MMAs take, and no CTA writes a 330 KB gradient of its own.  Bound by the
// latency of the chain gather - three layers - backward: at batch 256 the
// two forwards in a row of one kernel, then a forward and the backward of a
// second, took 30 of the step's 57 us.
constexpr int kTpRanks = 3;
constexpr int kLtRows = 128;             // samples of a tile of the tcgen05 learner
constexpr int kLtSub = kLtRows / kTile;  // its 16-sample fragment tiles
constexpr int kVecDb2 = kHid, kVecW3 = 2 * kHid, kVecB3 = kVecW3 + kOut * kHid, kVecHub = kVecB3 + kOut;
constexpr int kVecLd = (kVecHub + 1 + 31) / 32 * 32;  // db1 | db2 | dW3 | db3 | Huber sum
constexpr int kFragTile = 16 * 32;                    // 16-byte words of a 16 x 256 operand
struct TdFrag {
  uint4* z2;   // [tiles][16 unit blocks][32 lanes]: A fragments of dZ2^T
  uint4* h1;   // [tiles][16 unit pairs][32]: B fragments of H1
  uint4* z1;   // [tiles][16][32]: A fragments of dZ1^T
  uint4* x;    // [tiles][k1 / 16][32]: B fragments of X
  uint4* h2;   // [tiles][16][32]: A fragments of H2^T (128-sample learner)
  float* dout; // [tiles][16][8]: dL/d(head outputs), the Huber term in column 7 (128-sample learner)
  float* vec;  // [tiles][kVecLd]; [tiles / 8][kVecLd] of the 128-sample learner
};
inline size_t td_frag_bytes(int tiles, int k1) {
  return (size_t)tiles * ((4 * kFragTile + k1 / 16 * 32) * 16 + (kTile * kOutPad + kVecLd) * 4);
}
inline TdFrag td_frag(void* base, int tiles, int k1) {
  TdFrag f;
  f.z2 = static_cast<uint4*>(base);
  f.h1 = f.z2 + (size_t)tiles * kFragTile;
  f.z1 = f.h1 + (size_t)tiles * kFragTile;
  f.h2 = f.z1 + (size_t)tiles * kFragTile;
  f.x = f.h2 + (size_t)tiles * kFragTile;
  f.dout = reinterpret_cast<float*>(f.x + (size_t)tiles * (k1 / 16 * 32));
  f.vec = f.dout + (size_t)tiles * kTile * kOutPad;
  return f;
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory"); }
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
  return r;
}
// A float into the same variable of another CTA of the cluster.
__device__ __forceinline__ void st_cluster(float* p, uint32_t rank, float v) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  asm volatile("st.shared::cluster.f32 [%0], %1;\n" ::"r"(a), "f"(v) : "memory");
}

// The ring's step counter for a learner's cluster.  Its CTAs gather s and s' of
// the same samples, and a rollout on another stream may advance the counter
// between two loads, so they agree on the first CTA's reading.  A cluster barrier
// before the gather costs 0.6 us of a step (batch 256: 15.8 -> 16.4, its fences);
// instead each CTA goes on with its own reading (own[0], by one thread), one warp of
// the first CTA sends the others its value while they are at the first tile's
// head (to own[1], counted on their barrier bar), and a CTA that has read another
// one repeats that tile: 15.7 us, 19.1 when it has to.
constexpr int kOfferWarp = 8;
__device__ __forceinline__ void offer_steps(unsigned long long* own, uint64_t* bar, int ranks) {
  cluster_wait();  // every CTA of the cluster has started, its barrier is initialised
  const int r = threadIdx.x & 31;
  if (r > 0 && r < ranks) {
    uint32_t a, b;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(a) : "r"(smem_u32(own + 1)), "r"(r));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(b) : "r"(smem_u32(bar)), "r"(r));
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.u64 [%0], %1, [%2];\n" ::"r"(a),
                 "l"(own[0]), "r"(b)
                 : "memory");
  }
  __syncwarp();
}

// dL/d(head outputs) of a sample, every thread the same (two 16-byte reads).
__device__ __forceinline__ void load_do(const float* p, float (&d)[kOutPad]) {
  const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
  d[0] = a.x, d[1] = a.y, d[2] = a.z, d[3] = a.w, d[4] = b.x, d[5] = b.y, d[6] = b.z, d[7] = b.w;
}

// kRanks = 1 (a learner with SMs of its own): one CTA takes the three roles of a
// tile in turn, Q(s') first; the target network's image goes over the online one
// and back (two copies a tile).  The same values.
template <int kRanks>
__global__ void __cluster_dims__(kRanks, 1, 1) __launch_bounds__(kThreads, 1)
    k_td_tile(const uint8_t* img, const uint8_t* img_t, ImgLayout L, ReplayDev rp, unsigned long long seed,
              const unsigned long long* step, int batch, float gamma, TdFrag f, unsigned* fail) {
  extern __shared__ __align__(16) uint8_t smem[];
  uint8_t* sw = smem;
  bf16* X = reinterpret_cast<bf16*>(smem + L.bytes);
  bf16* H1 = X + kTile * L.ld1;
  bf16* H2 = H1 + kTile * kLdh;  // becomes dZ1
  bf16* Z2 = H2 + kTile * kLdh;
  float* O = reinterpret_cast<float*>(Z2 + kTile * kLdh);
  float* DO = O + kTile * kOutPad;  // dL/d(head outputs) [16][8]
  __shared__ uint64_t bar_w1, bar_w2;
  __shared__ float next_q[2][2][kTile * kOutPad];  // rank 0: head outputs of s' by tile parity and network
  __shared__ int rows[kTile];
  __shared__ float hub[kTile];
  __shared__ uint64_t bar_steps;
  __shared__ unsigned long long steps_sh[2];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int q = lane & 3, g = lane >> 2;
  uint32_t rank = kRanks == 1 ? 1u : cluster_rank();
  const int ntiles = (batch + kTile - 1) / kTile, stride = (int)gridDim.x / kRanks;
  if (tid == kThreads - 1) {
    mbar_init(&bar_w1, 1);
    mbar_init(&bar_w2, 1);
    mbar_init(&bar_steps, 1);
    if (kRanks > 1 && rank != 0) mbar_expect_tx(&bar_steps, 8u);
  }
  __syncwarp();
  cluster_arrive();  // every CTA of the cluster has started before the first remote store
  pdl_wait();
  pdl_launch_dependents();
  const unsigned long long tstep = __ldcg(step);
  if (tid == 0) steps_sh[0] = ring_steps(rp);
  auto load_image = [&]() {
    // layer 1 starts when W1 and the vectors behind W2 are here
    const uint8_t* src = rank == 2 ? img_t : img;
    mbar_expect_tx(&bar_w1, (uint32_t)(L.w2 + L.bytes - L.w3));
    bulk_g2s(sw, src, (uint32_t)L.w2, &bar_w1);
    bulk_g2s(sw + L.w3, src + L.w3, (uint32_t)(L.bytes - L.w3), &bar_w1);
    mbar_expect_tx(&bar_w2, (uint32_t)(L.w3 - L.w2));
    for (int off = L.w2; off < L.w3; off += kStageChunk)
      bulk_g2s(sw + off, src + off, (uint32_t)min(kStageChunk, L.w3 - off), &bar_w2);
  };
  if (tid == kThreads - 1) load_image();
  __syncthreads();
  const QW w = qw_at(sw, L);
  bool ok = true, first = true;  // first: the image's copy is still to be waited for, its phase
  uint32_t phase = 0u;
  int tile = (int)blockIdx.x / kRanks;
  uint64_t h = sample_hash(seed, tstep, tile * kTile + warp);
  unsigned long long st = steps_sh[0];
  bool agreed = rank == 0 || kRanks == 1;  // st is the cluster's
  for (int turn = 0; tile < ntiles; ++turn, tile += kRanks == 1 && turn % 3 ? 0 : stride) {
    const int it = kRanks == 1 ? turn / 3 : turn;
    if (kRanks == 1) {
      rank = (uint32_t)((turn + 1) % 3);
      if (rank != 1u && ok) {
        fence_async_smem();  // this thread's reads of the image before the copy overwrites it
        __syncthreads();
        if (tid == kThreads - 1) load_image();
        phase ^= 1u;
        first = true;
      }
    }
    {
      const int i = tile * kTile + warp;
      if (turn > 0) h = sample_hash(seed, tstep, i);
      const int e = i < batch ? (int)sample_entry(h, st, rp) : -1;
      const float* src = (rank == 0 ? rp.s : rp.s2) + (long long)e * rp.obs_dim;
      for (int k = lane; k < L.ld1; k += 32)
        X[warp * L.ld1 + k] = __float2bfloat16_rn(e >= 0 && k < rp.obs_dim ? src[k] : 0.0f);
      if (lane == 0) rows[warp] = e;
    }
    ok = __syncthreads_and(ok && (!first || mbar_wait(&bar_w1, phase, kTcTries)));
    // this sample's reward, flag and action on their way during the forward
    int e = -1, act = 0;
    float rwd = 0.0f, nt = 1.0f;
    if (rank == 0 && tid < kTile) {
      e = rows[tid];
      if (e >= 0) {
        act = rp.a[e];
        rwd = rp.r[e];
        nt = rp.term[e] ? 0.0f : 1.0f;
      }
    }
    if (ok) hidden_layer(X, L.ld1, L.k1 / 16, w.W1, L.ld1, w.b1, H1, warp, lane);
    ok = __syncthreads_and(ok && (!first || mbar_wait(&bar_w2, phase, kTcTries)));
    first = false;
    if (ok) hidden_layer(H1, kLdh, kHid / 16, w.W2, kLdh, w.b2, H2, warp, lane);
    __syncthreads();
    if (ok && warp == 0) head_layer(H2, w, O, lane);
    if (kRanks > 1 && turn == 0 && rank == 0 && warp == kOfferWarp) offer_steps(steps_sh, &bar_steps, kRanks);
    __syncthreads();
    if (!agreed) {
      ok = __syncthreads_and(ok && mbar_wait(&bar_steps, 0u, kTcTries));
      agreed = true;
      if (ok && st != steps_sh[1]) {
        // the first CTA read another value: the tile again
        st = steps_sh[1];
        if (tid == 0) ring_steps(rp);  // acquire: what the gather above left in L1 may be older than st
        __syncthreads();
        turn = -1, tile -= stride;
        continue;
      }
    }
    if (kRanks > 1 && turn == 0 && !(rank == 0 && warp == kOfferWarp)) cluster_wait();  // the start's arrival
    if (rank != 0 && tid < kTile * kOutPad)
      st_cluster(&next_q[it & 1][rank - 1][tid], 0u, ok ? O[tid] : __int_as_float(0x7fc00000));
    cluster_arrive();
    cluster_wait();
    if (rank != 0) continue;
    if (!ok) continue;
    // y = r + gamma (1 - term) Q_target(s', argmax_a Q_online(s', a));
    // dL/dQ(s, a) = clip(Q(s, a) - y, -1, 1) / B, back through the head's combine
    if (tid < kTile) {
      float qv[5], qn[5];
      const int astar = (int)greedy_action(&next_q[it & 1][0][tid * kOutPad], nullptr, L.plain);
      greedy_action(&next_q[it & 1][1][tid * kOutPad], qn, L.plain);
      greedy_action(O + tid * kOutPad, qv, L.plain);
      float* dO = DO + tid * kOutPad;
      float gq = 0.0f, hl = 0.0f;
#pragma unroll
      for (int k = 0; k < kOutPad; ++k) dO[k] = 0.0f;
      if (e >= 0) {
        float qs = qn[0], qa = qv[0];
#pragma unroll
        for (int k = 1; k < 5; ++k) {
          if (k == astar) qs = qn[k];
          if (k == act) qa = qv[k];
        }
        const float y = rwd + gamma * nt * qs;
        float d;
        if (act >= 5) {
          // outside the action table: no loss term, and no update this step
          atomicOr(fail, kTdFailAction);
          act = 0;
          d = __int_as_float(0x7fc00000);
        } else {
          d = qa - y;
        }
        const float ad = fabsf(d);
        hl = ad <= 1.0f ? 0.5f * d * d : ad - 0.5f;
        // a NaN target stays NaN through the clip
        gq = (isnan(d) ? d : fminf(fmaxf(d, -1.0f), 1.0f)) / (float)batch;
        if (L.plain) {
          for (int k = 0; k < 5; ++k) dO[k] = k == act ? gq : 0.0f;
        } else {
          dO[0] = gq;
          for (int k = 0; k < 5; ++k) dO[1 + k] = (k == act ? gq : 0.0f) - gq / 5.0f;
        }
      }
      hub[tid] = hl;
    }
    __syncthreads();
    float* vec = f.vec + (long long)tile * kVecLd;
    // the head's gradient on the CUDA cores (FP32), half of the threads each:
    // dW3[o][j] = sum_s dO[s][o] H2[s][j] and db3, the Huber sum; dH2 = dO W3
    // masked by the ReLU into dZ2, db2
    if (tid < kHid) {
      float acc[kOut];
#pragma unroll
      for (int o = 0; o < kOut; ++o) acc[o] = 0.0f;
#pragma unroll 4
      for (int s = 0; s < kTile; ++s) {
        const float h = __bfloat162float(H2[s * kLdh + tid]);
        float d[kOutPad];
        load_do(DO + s * kOutPad, d);
#pragma unroll
        for (int o = 0; o < kOut; ++o) acc[o] += d[o] * h;
      }
#pragma unroll
      for (int o = 0; o < kOut; ++o) vec[kVecW3 + o * kHid + tid] = acc[o];
      if (tid < kOut) {
        float b3 = 0.0f;
        for (int s = 0; s < kTile; ++s) b3 += DO[s * kOutPad + tid];
        vec[kVecB3 + tid] = b3;
      }
      if (tid == kHid - 1) {
        float h = 0.0f;
        for (int s = 0; s < kTile; ++s) h += hub[s];
        vec[kVecHub] = h;
      }
    } else {
      const int j = tid - kHid;
      float w3[kOut];
#pragma unroll
      for (int o = 0; o < kOut; ++o) w3[o] = __bfloat162float(w.W3[o * kLdh + j]);
      float db2 = 0.0f;
#pragma unroll 4
      for (int s = 0; s < kTile; ++s) {
        float dh = 0.0f, d[kOutPad];
        load_do(DO + s * kOutPad, d);
#pragma unroll
        for (int o = 0; o < kOut; ++o) dh += d[o] * w3[o];
        const float v = __bfloat162float(H2[s * kLdh + j]) > 0.0f ? dh : 0.0f;
        Z2[s * kLdh + j] = __float2bfloat16_rn(v);
        db2 += v;
      }
      vec[kVecDb2 + j] = db2;
    }
    __syncthreads();
    uint32_t r4[4];
    load_a_col(r4, Z2, kLdh, 16 * warp, 0, lane);
    f.z2[((long long)tile * 16 + warp) * 32 + lane] = make_uint4(r4[0], r4[1], r4[2], r4[3]);
    ldsm_x4_t(r4, H1 + ((lane & 7) + ((lane >> 3) & 1) * 8) * kLdh + 16 * warp + (lane >> 4) * 8);
    f.h1[((long long)tile * 16 + warp) * 32 + lane] = make_uint4(r4[0], r4[1], r4[2], r4[3]);
    // dH1 = dZ2 W2, masked by the ReLU into dZ1 (over H2), db1 from the FP32 values
    {
      const int u0 = 16 * warp;
      float c[2][4] = {};
#pragma unroll 4
      for (int k0 = 0; k0 < kHid; k0 += 16) {
        uint32_t a[4], x[4];
        load_a_col(a, w.W2, kLdh, u0, k0, lane);
        load_x16(x, Z2, kLdh, k0, lane);
        mma_bf16(c[0], a, x[0], x[1]);
        mma_bf16(c[1], a, x[2], x[3]);
      }
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int at = (8 * t + 2 * q + (j & 1)) * kLdh + u0 + g + (j >> 1) * 8;
          if (!(__bfloat162float(H1[at]) > 0.f)) c[t][j] = 0.f;
          H2[at] = __float2bfloat16_rn(c[t][j]);
        }
      // the 16 samples of a unit: s and s + 8, then a tree over s mod 8
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float v = (c[0][2 * h] + c[1][2 * h]) + (c[0][2 * h + 1] + c[1][2 * h + 1]);
        v += __shfl_xor_sync(kFull, v, 1);
        v += __shfl_xor_sync(kFull, v, 2);
        if (q == 0) vec[u0 + g + 8 * h] = v;
      }
    }
    __syncthreads();
    load_a_col(r4, H2, kLdh, 16 * warp, 0, lane);
    f.z1[((long long)tile * 16 + warp) * 32 + lane] = make_uint4(r4[0], r4[1], r4[2], r4[3]);
    const int nx = L.k1 / 16;
    if (warp < nx) {
      ldsm_x4_t(r4, X + ((lane & 7) + ((lane >> 3) & 1) * 8) * L.ld1 + 16 * warp + (lane >> 4) * 8);
      f.x[((long long)tile * nx + warp) * 32 + lane] = make_uint4(r4[0], r4[1], r4[2], r4[3]);
    }
    __syncthreads();  // X and the activations are rewritten by the next tile
  }
  if (!ok && tid == 0) {
    // no update this step; a copy that timed out may still be writing: one
    // more bounded wait for each before the CTA exits
    atomicOr(fail, kTdFailCopy);
    mbar_wait(&bar_w1, phase, kTcTries);
    mbar_wait(&bar_w2, phase, kTcTries);
    if (kRanks > 1 && rank != 0) mbar_wait(&bar_steps, 0u, kTcTries);
  }
}

// The weight gradients from k_td_tile's fragments, and the update, one item per
// CTA: a 16 x 16 block of W2 or W1 (per tile two MMAs, a 16-sample outer
// product from zero), or 64 entries of the vectors.  Every warp takes a run of
// consecutive tiles.  Up to 16 tiles each tile's product has a slot of its own
// in shared memory (four warps, one round of loads each); above, each warp adds
// its tiles up (eight warps).  A thread then adds the slots of two neighbouring
// parameters in order, in FP32, and updates both.  No gradient goes through
// memory: bound by the latency of the loads (old values before the wait) and of
// one Adam update; with one warp a block that had eight updates in a row
// it took 16 K cycles at batch 256, now 4 K (a whole step 23.0 -> 16.6 us).
constexpr int kTuItem = 256;  // floats of an item
constexpr int kTuSlots = 16;
template <int kWarps, bool kSlots>
__global__ void __launch_bounds__(32 * kWarps) k_td_update(TdUpdate u, TdFrag f, int ntiles) {
  __shared__ float sum[kSlots ? kTuSlots : kWarps][kTuItem];
  pdl_launch_dependents();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, t = threadIdx.x;
  const int nx = u.L.k1 / 16, n2 = 256, n1 = 16 * nx;
  const int item = blockIdx.x;
  const bool w2 = item < n2, mat = item < n2 + n1;
  const int mb = w2 ? item >> 4 : (item - n2) / nx, nb = w2 ? item & 15 : (item - n2) % nx;
  // this thread's parameters: columns k, k + 1 of row r, or vector entry ve
  const int r = mb * 16 + t / 8, k = nb * 16 + 2 * (t % 8), ve = (item - n2 - n1) * 64 + t;
  int at = 0;
  bool live[2];
  if (mat) {
    at = w2 ? u.P.w2 + r * kHid + k : u.P.w1 + r * u.L.n_in + k;
    live[0] = t < 128 && (w2 || k < u.L.n_in);
    live[1] = t < 128 && (w2 || k + 1 < u.L.n_in);
  } else {
    at = ve < kVecDb2 ? u.P.b1 + ve : ve < kVecW3 ? u.P.b2 + (ve - kVecDb2)
                                    : ve < kVecB3 ? u.P.w3 + (ve - kVecW3) : u.P.b3 + (ve - kVecB3);
    live[0] = t < 64 && ve < kVecHub;
    live[1] = false;
  }
  UpdRun run = upd_begin(u);
  // the old values (nothing before this launch writes them) before the wait
  float th[2] = {}, m[2] = {}, v[2] = {};
  if (u.lr != 0.0f) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (live[h]) th[h] = u.th[at + h], m[h] = u.m[at + h], v[h] = u.v[at + h];
  }
  pdl_wait();
  const unsigned fail = __ldcg(u.fail);
  const int per = (ntiles + kWarps - 1) / kWarps, t0 = warp * per, t1 = min(ntiles, t0 + per);
  if (mat) {
    const uint4* fa = (w2 ? f.z2 : f.z1) + mb * 32 + lane;
    const uint4* fb = (w2 ? f.h1 : f.x) + nb * 32 + lane;
    const int lb = w2 ? kFragTile : nx * 32;
    const int g = lane >> 2, q = lane & 3;
    float acc[2][4] = {};
    auto put = [&](float* s) {
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int j = 0; j < 2; ++j)
          *reinterpret_cast<float2*>(s + (g + 8 * j) * 16 + 8 * h + 2 * q) = make_float2(acc[h][2 * j], acc[h][2 * j + 1]);
    };
#pragma unroll 4
    for (int i = t0; i < t1; ++i) {
      const uint4 a = __ldcg(fa + (long long)i * kFragTile), b = __ldcg(fb + (long long)i * lb);
      const uint32_t ar[4] = {a.x, a.y, a.z, a.w};
      float d[2][4] = {};
      mma_bf16(d[0], ar, b.x, b.y);
      mma_bf16(d[1], ar, b.z, b.w);
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[h][j] = kSlots ? d[h][j] : acc[h][j] + d[h][j];
      if (kSlots) put(sum[i]);
    }
    if (!kSlots) put(sum[warp]);
  } else {
    const int e = (item - n2 - n1) * 64 + 2 * lane;
    float2 acc = make_float2(0.0f, 0.0f);
    if (e <= kVecHub) {
#pragma unroll 4
      for (int i = t0; i < t1; ++i) {
        const float2 x = __ldcg(reinterpret_cast<const float2*>(f.vec + (long long)i * kVecLd + e));
        acc.x = kSlots ? x.x : acc.x + x.x;
        acc.y = kSlots ? x.y : acc.y + x.y;
        if (kSlots) *reinterpret_cast<float2*>(sum[i] + 2 * lane) = acc;
      }
    }
    if (!kSlots) *reinterpret_cast<float2*>(sum[warp] + 2 * lane) = acc;
  }
  __syncthreads();
  const bool failed = fail != 0u;
  upd_fail(failed, run);
  const int slots = kSlots ? ntiles : kWarps;
  auto total = [&](int i) {
    float g = sum[0][i];
#pragma unroll 4
    for (int s = 1; s < slots; ++s) g += sum[s][i];
    return failed ? __int_as_float(0x7fc00000) : g;
  };
  if (mat) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (!live[h]) continue;
      const float g = total(2 * t + h);
      upd_grad(u, at + h, g);
      if (run.adam) th[h] = upd_adam(u, run, at + h, g, th[h], m[h], v[h]);
      if (run.sync) u.tgt[at + h] = th[h];
    }
    if (live[0]) {
      // the padding column beside an odd last input stays zero
      if (w2)
        upd_images<2, 2>(u, run, r, k, th[0], th[1]);
      else
        upd_images<1, 2>(u, run, r, k, th[0], th[1]);
    }
  } else if (live[0]) {
    upd_one(u, run, at, total(t), th[0], m[0], v[0]);
  } else if (ve == kVecHub && t < 64 && u.loss) {
    *u.loss = total(t) / (float)u.batch;
  }
  upd_end(u, failed);
}
inline int td_update_items(int k1) { return 256 + 16 * (k1 / 16) + (kVecHub + 1 + 63) / 64; }

// The same for the 128-sample learner, whose batches have hundreds of fragment
// tiles: a cluster of kSplit CTAs per item, a run of the tiles each, partial
// sums added in CTA order through distributed shared memory (each CTA updates
// an eighth of the item).  Items: 64 x 64 blocks of W2 and W1 (a warp 16 x 32, so
// that a fragment serves two or four warps; the tiles' operands, contiguous, by
// cp.async in two stages of eight tiles), W3 and b2 of 64 units, the
// remaining vectors.  Nothing here can fail: other items are updated meanwhile,
// so whether the step counts is settled before this kernel (a bulk copy's
// bounded wait would come too late).  Bound by L2 reads (each operand four times) and the
// latency of the chain; 16 x 16 items of one CTA read each operand 16 times,
// 88 MB at batch 4,096 (45.6 us a step, 34.5 now with the rolled epilogues).
constexpr int kSplit = 8, kSplitBlk = 64;
constexpr int kBigB3 = kHid, kBigHub = kBigB3 + kOut;  // vectors of a 128-sample tile: db1 | db3 | Huber sum
inline int td_split_items(int k1) { return 16 + 4 * ((k1 / 16 + 3) / 4) + 4 + 1; }

// x in three BF16 terms (24 bits: exact for a normal x not near the smallest).
__device__ __forceinline__ void split_bf16(float x, float (&t)[3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    t[i] = __bfloat162float(__float2bfloat16_rn(x));
    x -= t[i];
  }
}
// Two floats of another CTA's copy of a shared array.
__device__ __forceinline__ float2 ld_cluster2(const float* p, uint32_t rank) {
  uint32_t a;
  float2 v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];\n" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
  return v;
}

// 16 bytes from global memory (through L2) to shared memory, asynchronously;
// commit groups the copies issued so far, wait1 waits for all groups but the last.
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }

// Operands of a group of fragment tiles in one stage: 2 KB of A, up to 2 KB of B a
// tile; two stages.
constexpr int kStageTile = 4096;
constexpr int kBlkFloats = kSplitBlk * kSplitBlk;
inline constexpr int split_group(int ctas) { return ctas == 1 ? 4 : 8; }
inline constexpr int split_threads(int ctas) { return ctas == 1 ? 512 : 256; }
inline constexpr size_t split_smem(int ctas) {
  return (size_t)kSplit / ctas * kBlkFloats * 4 + (size_t)split_threads(ctas) / 256 * 2 * split_group(ctas) * kStageTile;
}

// kCtas = 1 (a learner with SMs of its own): one CTA takes the kSplit parts of an
// item with the same sums, its two halves of 256 threads (each with stages and a
// barrier of its own) every other part.
template <int kCtas>
__global__ void __cluster_dims__(kCtas, 1, 1) __launch_bounds__(split_threads(kCtas), kCtas == 1 ? 1 : 2)
    k_td_update_split(TdUpdate u, TdFrag f, int ntiles) {
  extern __shared__ __align__(128) uint8_t usm[];
  constexpr int kParts = kSplit / kCtas, kHalves = split_threads(kCtas) / 256, kGroup = split_group(kCtas);
  const int half = kHalves > 1 ? (int)threadIdx.x >> 8 : 0;
  float* blk = reinterpret_cast<float*>(usm);
  uint8_t* stage = usm + kParts * kBlkFloats * 4 + half * 2 * kGroup * kStageTile;
  auto sync = [&]() {
    if (kHalves > 1)
      group_barrier(1 + half, 256);
    else
      __syncthreads();
  };
  pdl_launch_dependents();
  const int t = (int)threadIdx.x & 255, warp = t >> 5, lane = t & 31;
  const int g = lane >> 2, q = lane & 3;
  const int first = kCtas == 1 ? 0 : (int)cluster_rank();
  const int nx = u.L.k1 / 16, nb1 = (nx + 3) / 4, n2 = 16, n1 = 4 * nb1;
  const int item = (int)blockIdx.x / kCtas;
  const bool w2 = item < n2, mat = item < n2 + n1, head = !mat && item < n2 + n1 + 4;
  const int mb = w2 ? item >> 2 : (item - n2) / nb1, nb = w2 ? item & 3 : (item - n2) % nb1, hb = item - n2 - n1;
  // this thread's parameters of a part: columns k, k + 1 of row r; output o of
  // unit n (o = 6: its bias); vector entry ve
  const int k = nb * kSplitBlk + 2 * lane, o = t >> 3;
  constexpr int kVe = (kBigHub + 1 + kSplit - 1) / kSplit;
  int r = 0, n = 0, ve = 0, at = 0;
  bool live[2] = {false, false};
  float w3[kOut] = {};  // the unit's column of W3, before this launch changes it
  float th[2] = {}, m[2] = {}, v[2] = {};
  auto old_values = [&](int part) {
    r = mb * kSplitBlk + 8 * part + warp, n = hb * kSplitBlk + 8 * part + (t & 7), ve = part * kVe + t;
    if (mat) {
      at = w2 ? u.P.w2 + r * kHid + k : u.P.w1 + r * u.L.n_in + k;
      live[0] = w2 || k < u.L.n_in;
      live[1] = w2 || k + 1 < u.L.n_in;
    } else if (head) {
      at = o < kOut ? u.P.w3 + o * kHid + n : u.P.b2 + n;
      live[0] = o <= kOut;
      if (o == kOut) {
#pragma unroll
        for (int i = 0; i < kOut; ++i)
          w3[i] = __bfloat162float(__ldcg(reinterpret_cast<const bf16*>(u.img + u.L.w3) + i * kLdh + n));
      }
    } else {
      at = ve < kBigB3 ? u.P.b1 + ve : u.P.b3 + (ve - kBigB3);
      live[0] = t < kVe && ve < kBigHub;
    }
    if (u.lr != 0.0f) {
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (live[h]) th[h] = u.th[at + h], m[h] = u.m[at + h], v[h] = u.v[at + h];
    }
  };
  UpdRun run = upd_begin(u);
  if (kCtas > 1) old_values(first);
  pdl_wait();
  const bool failed = __ldcg(u.fail) != 0u;
  upd_fail(failed, run);
  // fragment tiles of a part, or the vectors of 128-sample tiles
  const int nt = mat || head ? ntiles : (ntiles + kLtSub - 1) / kLtSub;
  const int per = (nt + kSplit - 1) / kSplit;
  for (int p = half; p < kParts; p += kHalves) {
    float* sums = blk + p * kBlkFloats;
    const int t0 = (first + p) * per, t1 = min(nt, t0 + per);
    if (mat || head) {
      // a tile's operands are contiguous: four 16-unit blocks of A; four (or the
      // rest of) 16-column blocks of B, or the 16 rows of dO
      const int nbk = w2 ? 16 : nx, bblk = min(4, nbk - 4 * nb);
      const uint8_t* ga = reinterpret_cast<const uint8_t*>(head ? f.h2 + 4 * hb * 32 : (w2 ? f.z2 : f.z1) + 4 * mb * 32);
      const uint8_t* gb = head ? reinterpret_cast<const uint8_t*>(f.dout)
                               : reinterpret_cast<const uint8_t*>((w2 ? f.h1 : f.x) + 4 * nb * 32);
      const long long lb = head ? kTile * kOutPad * 4 : nbk * 512;
      const int bb = head ? kTile * kOutPad * 4 : bblk * 512;
      const int ngroups = (t1 - t0 + kGroup - 1) / kGroup;
      // group i into its stage: a 16-byte word per thread and tile, of A by the
      // first four warps, of B by the others
      const bool mine = t < 128 || (t - 128) * 16 < bb;
      auto issue = [&](int i) {
        const int g0 = t0 + i * kGroup, gn = min(kGroup, t1 - g0);
        const uint8_t* src = t < 128 ? ga + (long long)g0 * (kFragTile * 16) + t * 16 : gb + g0 * lb + (t - 128) * 16;
        const long long ld = t < 128 ? kFragTile * 16 : lb;
        uint8_t* dst = stage + (i & 1) * kGroup * kStageTile + t * 16;
        if (mine)
          for (int e = 0; e < gn; ++e) cp_async16(dst + e * kStageTile, src + e * ld);
        cp_async_commit();
      };
      issue(0);
      issue(1);
      const bool have0 = mat && 2 * (warp & 1) < bblk, have1 = mat && 2 * (warp & 1) + 1 < bblk;
      float acc[2][2][4] = {};
      for (int i = 0; i < ngroups; ++i) {
        cp_async_wait1();  // group i (i + 1 stays in flight)
        sync();
        const int gn = min(kGroup, t1 - t0 - i * kGroup);
        const uint8_t* st = stage + (i & 1) * kGroup * kStageTile;
        if (mat) {
#pragma unroll 2
          for (int e = 0; e < gn; ++e, st += kStageTile) {
            const uint4 a = reinterpret_cast<const uint4*>(st + (warp >> 1) * 512)[lane];
            const uint4* pb = reinterpret_cast<const uint4*>(st + 2048 + 2 * (warp & 1) * 512) + lane;
            const uint4 z = make_uint4(0u, 0u, 0u, 0u), b0 = have0 ? pb[0] : z, b1 = have1 ? pb[32] : z;
            const uint32_t ar[4] = {a.x, a.y, a.z, a.w};
            float d[2][2][4] = {};
            mma_bf16(d[0][0], ar, b0.x, b0.y);
            mma_bf16(d[0][1], ar, b0.z, b0.w);
            mma_bf16(d[1][0], ar, b1.x, b1.y);
            mma_bf16(d[1][1], ar, b1.z, b1.w);
#pragma unroll
            for (int b = 0; b < 2; ++b)
#pragma unroll
              for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[b][h][j] += d[b][h][j];
          }
        } else {
          // dW3[o][n] = sum_s dO[s][o] H2[s][n] (warps 0..3) and M[n][o], the same
          // sum over the samples with H2[s][n] > 0, from which db2[n] = sum_o W3[o][n]
          // M[n][o] (warps 4..7).  dO in three BF16 terms against the exact BF16 H2
          // and 0 / 1: FP32 sums of exact products, as on the CUDA cores.
#pragma unroll 2
          for (int e = 0; e < gn; ++e, st += kStageTile) {
            const uint4 a = reinterpret_cast<const uint4*>(st + (warp & 3) * 512)[lane];
            const float* d = reinterpret_cast<const float*>(st + 2048) + 2 * q * kOutPad + g;
            float x[4][3];
            split_bf16(d[0], x[0]);
            split_bf16(d[kOutPad], x[1]);
            split_bf16(d[8 * kOutPad], x[2]);
            split_bf16(d[9 * kOutPad], x[3]);
            uint32_t ar[4] = {a.x, a.y, a.z, a.w};
            if (warp >= 4) {
#pragma unroll
              for (int j = 0; j < 4; ++j)
                ar[j] = ((ar[j] & 0x7FFFu) ? 0x3F80u : 0u) | ((ar[j] & 0x7FFF0000u) ? 0x3F800000u : 0u);
            }
            float sm[4] = {};
#pragma unroll
            for (int c = 2; c >= 0; --c) mma_bf16(sm, ar, pack_bf16x2(x[0][c], x[1][c]), pack_bf16x2(x[2][c], x[3][c]));
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[0][0][j] += sm[j];
          }
        }
        sync();  // these reads before the stage takes another copy
        issue(i + 2);
      }
      if (mat) {
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int j = 0; j < 2; ++j)
              *reinterpret_cast<float2*>(sums + (16 * (warp >> 1) + g + 8 * j) * kSplitBlk + 32 * (warp & 1) + 16 * b + 8 * h + 2 * q) =
                  make_float2(acc[b][h][2 * j], acc[b][h][2 * j + 1]);
      } else {
#pragma unroll
        for (int j = 0; j < 2; ++j)
          *reinterpret_cast<float2*>(sums + (16 * (warp & 3) + g + 8 * j) * 16 + 8 * (warp >> 2) + 2 * q) =
              make_float2(acc[0][0][2 * j], acc[0][0][2 * j + 1]);
      }
    } else {
      for (int e = t; e <= kBigHub; e += 256) {
        float a = 0.0f;
#pragma unroll 4
        for (int i = t0; i < t1; ++i) a += __ldcg(f.vec + (long long)i * kVecLd + e);
        sums[e] = a;
      }
    }
  }
  cluster_arrive();
  cluster_wait();
  // element i (even) and i + 1 of the item
  auto total = [&](int i) {
    float2 x[kSplit];
#pragma unroll
    for (int c = 0; c < kSplit; ++c)
      x[c] = kCtas == 1 ? *reinterpret_cast<const float2*>(blk + c * kBlkFloats + i) : ld_cluster2(blk + i, (uint32_t)c);
    float2 sum = x[0];
#pragma unroll
    for (int c = 1; c < kSplit; ++c) sum.x += x[c].x, sum.y += x[c].y;
    if (failed) sum.x = sum.y = __int_as_float(0x7fc00000);
    return sum;
  };
  for (int p = half; p < kParts; p += kHalves) {
    const int part = first + p;
    if (kCtas == 1) {
      old_values(part);
      sync();  // the part's columns of W3 are read before other threads change them
    }
    if (mat) {
      if (live[0]) {
        const float2 gr = total((8 * part + warp) * kSplitBlk + 2 * lane);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (!live[h]) continue;
          const float gh = h ? gr.y : gr.x;
          upd_grad(u, at + h, gh);
          if (run.adam) th[h] = upd_adam(u, run, at + h, gh, th[h], m[h], v[h]);
          if (run.sync) u.tgt[at + h] = th[h];
        }
        // the padding column beside an odd last input stays zero
        if (w2)
          upd_images<2, 2>(u, run, r, k, th[0], th[1]);
        else
          upd_images<1, 2>(u, run, r, k, th[0], th[1]);
      }
    } else if (head) {
      if (live[0]) {
        const int e = (8 * part + (t & 7)) * 16;
        float gr = 0.0f;
        if (o < kOut) {
          const float2 x = total(e + (o & ~1));
          gr = (o & 1) ? x.y : x.x;
        } else {
#pragma unroll
          for (int i = 0; i < kOut; i += 2) {
            const float2 x = total(e + 8 + i);
            gr += w3[i] * x.x;
            gr += w3[i + 1] * x.y;
          }
        }
        upd_one(u, run, at, gr, th[0], m[0], v[0]);
      }
    } else if (t < kVe && ve <= kBigHub) {
      const float2 x = total(ve & ~1);
      const float gr = (ve & 1) ? x.y : x.x;
      if (ve < kBigHub)
        upd_one(u, run, at, gr, th[0], m[0], v[0]);
      else if (u.loss)
        *u.loss = gr / (float)u.batch;
    }
  }
  upd_end(u, failed);
  cluster_arrive();  // the others' reads of this CTA's sums are done
  cluster_wait();
}

// ------------------------------------------------ tcgen05 learner (large batches)
// The tiles of k_td_tile with 128 samples, on the fifth-generation tensor
// cores: a cluster of three CTAs takes a tile (rank 0 the forward on s and the
// backward pass, ranks 1 and 2 the online and target network's Q(s')), every
// CTA with its network's W1, W2 and W3 resident in shared memory (bulk copies,
// once per launch).  Thread 0 issues the MMAs; 16 warps run the epilogues on
// their lane quarter and 64 columns.  Accumulators are read in the fragment
// shape of mma.sync (tcgen05.ld.16x256b), so that an epilogue packs its BF16
// pairs back into tensor memory as the next layer's A operand
// (tcgen05.st.16x128b) and, with one movmatrix per 8 x 8 block, writes the
// operands that k_td_update sums the weight gradients from:
//   [0, 256)   layer 1, H1 (first half of each 64), head in [32, 48), then dH1
//   [256, 512) layer 2, H2, then dZ2 over it
// dH1 = dZ2 W2 reads W2's shared-memory operand transposed: a K-major tile of R
// rows is, MN-major, the same 128-byte core matrices with SBO = 16 R between
// 8-element MN groups and LBO = 128 between 8-row K groups.
// Bound by the latency of its chain (gather, three layers, dO, dH1, about 18 K
// cycles).  In place of the learner whose jobs streamed W2 through two 32 KB
// buffers, ran a forward for each of two roles a tile and wrote a 330 KB
// gradient row per tile: batch 4,096 76 -> 32.3 us.
// Below this batch the 16-sample learner, whose CTAs spread over more SMs: 24.3
// against 27.2 us at batch 1,024 (35.8 against 31.3 at 2,000, where the line
// stays so that the batches keep their summation order).
constexpr int kLtMinBatch = 2048;

struct LtSmem {
  uint32_t x, w1, w2, w3, dout, bias, w3f, red, next, bytes;
};
__host__ __device__ inline LtSmem lt_smem(int k1) {
  LtSmem t;
  t.x = 0;
  t.w1 = (uint32_t)(kLtRows * k1 * 2);
  t.w2 = t.w1 + (uint32_t)(kHid * k1 * 2);
  t.w3 = t.w2 + (uint32_t)(kHid * kHid * 2);
  t.dout = t.w3 + 16u * kHid * 2u;                       // dO [128][8] float
  t.bias = t.dout + (uint32_t)(kLtRows * kOutPad * 4);   // b1, b2 [256] float
  t.w3f = t.bias + 2u * kHid * 4u;                       // W3 [6][256] float
  t.red = t.w3f + (uint32_t)(kOut * kHid * 4);           // column sums [4][256] float
  t.next = t.red + 4u * kHid * 4u;                       // Q(s') [tile parity][network][128][5] float
  t.bytes = t.next + 2u * 2u * kLtRows * 5u * 4u;
  return t;
}
static_assert(128 * 80 * 2 + 256 * 80 * 2 + 256 * 256 * 2 + 16 * 256 * 2 + 128 * 32 + 2048 + 6144 + 4096 + 10240 <=
                  227 * 1024 - 1024,
              "tcgen05 learner: shared memory");

// Instruction descriptor with the operands' major-ness: trans_a / trans_b = 1
// reads A / B MN-major (bits 15 / 16).
__host__ __device__ constexpr uint32_t idesc_bf16_f32_t(int M, int N, int trans_a, int trans_b) {
  return idesc_bf16_f32(M, N) | ((uint32_t)trans_a << 15) | ((uint32_t)trans_b << 16);
}

// A CTA-wide barrier that also orders the tensor-core work around it.
__device__ __forceinline__ void lt_sync() {
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
}
__device__ __forceinline__ uint32_t movmatrix(uint32_t a) {
  uint32_t d;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;\n" : "=r"(d) : "r"(a));
  return d;
}
// 16 samples x 16 units in C-fragment pairs (p[2 j]: sample g, p[2 j + 1]: g + 8,
// units 8 j + 2 q, + 1) as an operand of k_td_update_split: the A fragment of the
// transpose, or the B fragment.
template <bool kA>
__device__ __forceinline__ void lt_put_frag(uint4* out, const uint32_t (&p)[4], int lane) {
  const uint32_t l0 = movmatrix(p[0]), l1 = movmatrix(p[1]), h0 = movmatrix(p[2]), h1 = movmatrix(p[3]);
  out[lane] = kA ? make_uint4(l0, h0, l1, h1) : make_uint4(l0, l1, h0, h1);
}
// Hidden-layer epilogue of a warp's 32 rows x 64 columns at t, 16 columns at a
// time: bias, ReLU, BF16 pairs back into the first half of the columns (below
// every column still to be read); with kPut != 0 also as fragments (1: B, 2: A)
// to out (the next 16 units 32 words on, the next 16 samples kFragTile), and
// mask[h] bit 8 b + 4 j + e = whether element e of octet j of block b is positive.
// Rolled: the code runs once per tile, so its instruction fetches count.
template <int kPut>
__device__ __forceinline__ void lt_epilogue(uint32_t t, const float* bias, uint4* out, uint32_t (&mask)[2], int lane) {
  const float2* b2 = reinterpret_cast<const float2*>(bias) + (lane & 3);
  mask[0] = mask[1] = 0u;
#pragma unroll 1
  for (int b = 0; b < 4; ++b) {
    uint32_t r[2][8];
    tmem_ld_frag16_nowait(t + 16u * b, r[0]);
    tmem_ld_frag16_nowait(t + (16u << 16) + 16u * b, r[1]);
    const float2 bb[2] = {b2[8 * b], b2[8 * b + 4]};
    tmem_ld_wait();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint32_t p[4], mk = 0u;
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const uint32_t w = pack_bf16x2(fmaxf(__uint_as_float(r[h][4 * j + 2 * e]) + bb[j].x, 0.f),
                                         fmaxf(__uint_as_float(r[h][4 * j + 2 * e + 1]) + bb[j].y, 0.f));
          p[2 * j + e] = w;
          if (kPut) mk |= ((w & 0x7FFFu) ? 1u : 0u) << (4 * j + 2 * e) | ((w & 0x7FFF0000u) ? 2u : 0u) << (4 * j + 2 * e);
        }
      tmem_st_frag8(t + ((uint32_t)(16 * h) << 16) + 8u * b, p);
      if (kPut) {
        lt_put_frag<kPut == 2>(out + h * kFragTile + b * 32, p, lane);
        mask[h] |= mk << (8 * b);
      }
    }
  }
  tmem_st_wait();
}

// kRanks = 1: the three roles of a tile in turn, as in k_td_tile.
template <int kRanks>
__global__ void __cluster_dims__(kRanks, 1, 1) __launch_bounds__(kThreads, 1)
    k_td_tc(const uint8_t* img, const uint8_t* img_t, const uint8_t* timg, const uint8_t* timg_t, ImgLayout L,
            ReplayDev rp, unsigned long long seed, const unsigned long long* step, int batch, float gamma, TdFrag f,
            unsigned* fail) {
  extern __shared__ __align__(1024) uint8_t tsm[];
  __shared__ uint64_t bar_w1, bar_w2, bar_mma;
  __shared__ uint32_t tslot;
  __shared__ int rows_sh[kLtRows];
  __shared__ float dsum_sh[4][kOutPad];
  __shared__ uint64_t bar_steps;
  __shared__ unsigned long long steps_sh[2];
  const LtSmem T = lt_smem(L.k1);
  const TcImg G = tc_img(L.k1);
  uint8_t* xs = tsm + T.x;
  float* dout = reinterpret_cast<float*>(tsm + T.dout);
  float* b1 = reinterpret_cast<float*>(tsm + T.bias);
  float* b2 = b1 + kHid;
  float* w3f = reinterpret_cast<float*>(tsm + T.w3f);
  float* red = reinterpret_cast<float*>(tsm + T.red);
  float* next_q = reinterpret_cast<float*>(tsm + T.next);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, q = lane & 3, quarter = warp & 3, grp = warp >> 2;
  uint32_t rank = kRanks == 1 ? 1u : cluster_rank();
  const int ntiles = (batch + kLtRows - 1) / kLtRows, stride = (int)gridDim.x / kRanks;
  if (tid == kThreads - 1) {
    mbar_init(&bar_w1, 1);
    mbar_init(&bar_w2, 1);
    mbar_init(&bar_mma, 1);
    mbar_init(&bar_steps, 1);
    if (kRanks > 1 && rank != 0) mbar_expect_tx(&bar_steps, 8u);
  }
  __syncwarp();
  cluster_arrive();  // every CTA of the cluster has started before the first remote store
  if (warp == 0) tmem_alloc(&tslot, 512);
  pdl_wait();
  pdl_launch_dependents();
  const unsigned long long tstep = __ldcg(step);
  if (tid == 0) steps_sh[0] = ring_steps(rp);
  auto load_image = [&]() {
    const uint8_t* src = rank == 2 ? timg_t : timg;
    mbar_expect_tx(&bar_w1, G.w2a + 2u * kHid * 4u);
    bulk_g2s(tsm + T.w1, src + G.w1, G.w2a, &bar_w1);
    bulk_g2s(b1, (rank == 2 ? img_t : img) + L.b1, 2u * kHid * 4u, &bar_w1);  // b1 and b2
    mbar_expect_tx(&bar_w2, kHid * kHid * 2u + 16u * kHid * 2u);
    bulk_g2s(tsm + T.w2, src + G.w2f, kHid * kHid * 2u, &bar_w2);
    bulk_g2s(tsm + T.w3, src + G.w3, 16u * kHid * 2u, &bar_w2);
  };
  if (tid == kThreads - 1) load_image();
  lt_sync();
  const uint32_t tacc = tslot, tacc2 = tacc + 256u;
  const uint32_t tw = ((uint32_t)(quarter * 32) << 16) + (uint32_t)(64 * grp);  // this warp's lanes and columns
  const uint32_t sx = smem_u32(xs), sw1 = smem_u32(tsm + T.w1), sw2 = smem_u32(tsm + T.w2),
                 sw3 = smem_u32(tsm + T.w3);
  const int nx = L.k1 / 16;
  float b3[kOut];
  bool ok = true, first = true, mma_out = false;
  uint32_t phase = 0u, wphase = 0u;
  // wait for the MMAs committed last, by every thread
  auto mma_wait = [&]() {
    mma_out = true;
    ok = __syncthreads_and(ok && mbar_wait(&bar_mma, phase, kTcTries));
    phase ^= 1u;
    if (ok) mma_out = false;
    tc_fence_after();
  };
  int tile = (int)blockIdx.x / kRanks;
  uint64_t h = sample_hash(seed, tstep, tile * kLtRows + tid);
  unsigned long long st = steps_sh[0];
  bool agreed = rank == 0 || kRanks == 1;  // st is the cluster's
  for (int turn = 0; tile < ntiles; ++turn, tile += kRanks == 1 && turn % 3 ? 0 : stride) {
    const int it = kRanks == 1 ? turn / 3 : turn;
    if (kRanks == 1) {
      rank = (uint32_t)((turn + 1) % 3);
      if (rank != 1u && ok) {
        // every MMA that read the weights is complete
        fence_async_smem();  // this thread's reads of the biases before the copy overwrites them
        __syncthreads();
        if (tid == kThreads - 1) load_image();
        wphase ^= 1u;
        first = true;
      }
    }
    const uint8_t* im = rank == 2 ? img_t : img;
    if (tid < kLtRows) {
      const int i = tile * kLtRows + tid;
      if (turn > 0) h = sample_hash(seed, tstep, i);
      rows_sh[tid] = i < batch ? (int)sample_entry(h, st, rp) : -1;
    }
    __syncthreads();
    {
      // a row per warp and pass: its floats are contiguous
      const float* src = rank == 0 ? rp.s : rp.s2;
      float v[8][3];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int e = rows_sh[warp * 8 + u];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const int k = lane + 32 * c;
          v[u][c] = e >= 0 && k < L.n_in ? __ldcg(src + (long long)e * L.n_in + k) : 0.0f;
        }
      }
#pragma unroll
      for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int c = 0; c < 3; ++c)
          if (lane + 32 * c < L.k1)
            *reinterpret_cast<bf16*>(xs + kmajor_offset(warp * 8 + u, lane + 32 * c, kLtRows)) =
                __float2bfloat16_rn(v[u][c]);
    }
    fence_async_smem();
    lt_sync();
    int e = -1, act = 0;
    float rwd = 0.0f, nt = 1.0f;
    if (rank == 0 && tid < kLtRows) {
      // this sample's reward, flag and action on their way during the forward
      e = rows_sh[tid];
      if (e >= 0) {
        act = rp.a[e];
        rwd = rp.r[e];
        nt = rp.term[e] ? 0.0f : 1.0f;
      }
    }
    if (tid == 0 && ok && (!first || mbar_wait(&bar_w1, wphase, kTcTries))) {
      tc_fence_after();
      for (int ks = 0; ks < nx; ++ks)
        tc_mma_bf16(tacc, smem_desc(sx + (uint32_t)ks * 2u * kLtRows * 16u, kLtRows * 16u, 128),
                    smem_desc(sw1 + (uint32_t)ks * 2u * kHid * 16u, kHid * 16u, 128), idesc_bf16_f32(kLtRows, kHid),
                    ks > 0 ? 1u : 0u);
      tc_commit(&bar_mma);
    }
    if (rank == 0) {
      // X's B fragments: a core matrix is an 8 x 8 block of 16-byte rows
      for (int w = warp; w < kLtSub * nx; w += kThreads / 32) {
        const int st = w / nx, kb = w % nx, mat = lane >> 3;  // matrices: samples 0-7, 8-15 of inputs 0-7, then 8-15
        uint32_t r4[4];
        ldsm_x4_t(r4, xs + kmajor_offset(st * 16 + (mat & 1) * 8 + (lane & 7), kb * 16 + (mat >> 1) * 8, kLtRows));
        f.x[((long long)(tile * kLtSub + st) * nx + kb) * 32 + lane] = make_uint4(r4[0], r4[1], r4[2], r4[3]);
      }
    }
    mma_wait();
    // this warp's fragment tiles: samples 32 quarter .., units 64 grp ..
    const long long fo = (long long)(tile * kLtSub + 2 * quarter) * kFragTile + 4 * grp * 32;
    uint32_t mask1[2] = {0u, 0u}, mask2[2] = {0u, 0u};
    if (ok && first) mbar_wait(&bar_w1, wphase, kTcTries);  // complete: the biases are visible to this thread
    if (ok) {
      if (rank == 0)
        lt_epilogue<1>(tacc + tw, b1 + 64 * grp, f.h1 + fo, mask1, lane);
      else
        lt_epilogue<0>(tacc + tw, b1 + 64 * grp, nullptr, mask1, lane);
    }
    lt_sync();
    if (tid == 0 && ok && (!first || mbar_wait(&bar_w2, wphase, kTcTries))) {
      tc_fence_after();
      tc_layer_ta(tacc2, tacc, sw2, kHid);
      tc_commit(&bar_mma);
    }
    if (first) {
      // behind layer 2 (with the biases, behind layer 1 they took 1.3 us of batch 4,096)
      if (rank == 0) {
        // W3 in FP32 for dZ2
#pragma unroll
        for (int i = 0; i < kOut * kHid / kThreads; ++i) {
          const int j = tid + i * kThreads;
          w3f[j] = __bfloat162float(__ldcg(reinterpret_cast<const bf16*>(im + L.w3) + (j >> 8) * kLdh + (j & (kHid - 1))));
        }
      }
#pragma unroll
      for (int j = 0; j < kOut; ++j) b3[j] = __ldcg(reinterpret_cast<const float*>(im + L.b3) + j);
    }
    first = false;
    mma_wait();
    if (ok) {
      if (rank == 0)
        lt_epilogue<2>(tacc2 + tw, b2 + 64 * grp, f.h2 + fo, mask2, lane);
      else
        lt_epilogue<0>(tacc2 + tw, b2 + 64 * grp, nullptr, mask2, lane);
    }
    lt_sync();
    if (tid == 0 && ok) {
      tc_layer_ta(tacc + 32u, tacc2, sw3, 16);
      tc_commit(&bar_mma);
    }
    if (kRanks > 1 && turn == 0 && rank == 0 && warp == kOfferWarp) offer_steps(steps_sh, &bar_steps, kRanks);
    mma_wait();
    float qv[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
    if (warp < 4) {
      uint32_t v[8];
      float o[kOut];
      if (ok) {
        tmem_ld8_nowait(tacc + 32u + ((uint32_t)(warp * 32) << 16), v);
        tmem_ld_wait();
      }
#pragma unroll
      for (int j = 0; j < kOut; ++j) o[j] = (ok ? __uint_as_float(v[j]) : __int_as_float(0x7fc00000)) + b3[j];
      greedy_action(o, qv, L.plain);
    }
    if (!agreed) {
      ok = __syncthreads_and(ok && mbar_wait(&bar_steps, 0u, kTcTries));
      agreed = true;
      if (ok && st != steps_sh[1]) {
        // the first CTA read another value: the tile again (its head is read)
        st = steps_sh[1];
        if (tid == 0) ring_steps(rp);  // acquire, as in k_td_tile
        lt_sync();
        turn = -1, tile -= stride;
        continue;
      }
    }
    if (kRanks > 1 && turn == 0 && !(rank == 0 && warp == kOfferWarp)) cluster_wait();  // the start's arrival
    if (rank != 0 && warp < 4) {
#pragma unroll
      for (int a = 0; a < 5; ++a)
        st_cluster(next_q + (((it & 1) * 2 + (int)rank - 1) * kLtRows + tid) * 5 + a, 0u, qv[a]);
    }
    cluster_arrive();
    cluster_wait();
    if (rank != 0 || !ok) {
      lt_sync();  // the head is read before the next tile's layer 1
      continue;
    }
    // double-DQN targets y = r + gamma (1 - term) Q_target(s', argmax_a Q_online(s', a));
    // dL/dQ(s, a) = clip(Q(s, a) - y) / B, back through the head's combine
    if (warp < 4) {
      const float* qo = next_q + ((it & 1) * 2 * kLtRows + tid) * 5;
      const float* qt = qo + kLtRows * 5;
      float d8[kOutPad] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      if (e >= 0) {
        float best = qo[0], qs = qt[0], qa = qv[0];
#pragma unroll
        for (int a = 1; a < 5; ++a) {
          if (qo[a] > best) best = qo[a], qs = qt[a];
          if (act == a) qa = qv[a];
        }
        const float y = isnan(best) ? best : rwd + gamma * nt * qs;  // NaN: a failed next-state forward
        float d;
        if (act >= 5) {
          atomicOr(fail, kTdFailAction);
          act = 0;
          d = __int_as_float(0x7fc00000);
        } else {
          d = qa - y;
        }
        const float ad = fabsf(d);
        const float gq = (isnan(d) ? d : fminf(fmaxf(d, -1.0f), 1.0f)) / (float)batch;
        if (L.plain) {
#pragma unroll
          for (int k = 0; k < 5; ++k) d8[k] = k == act ? gq : 0.0f;
        } else {
          d8[0] = gq;
#pragma unroll
          for (int k = 0; k < 5; ++k) d8[1 + k] = (k == act ? gq : 0.0f) - gq / 5.0f;
        }
        d8[7] = ad <= 1.0f ? 0.5f * d * d : ad - 0.5f;  // the Huber term beside dO
      }
      float4* dO = reinterpret_cast<float4*>(dout + tid * kOutPad);
      float4* dg = reinterpret_cast<float4*>(f.dout + ((long long)tile * kLtRows + tid) * kOutPad);
      dO[0] = dg[0] = make_float4(d8[0], d8[1], d8[2], d8[3]);
      dO[1] = dg[1] = make_float4(d8[4], d8[5], d8[6], d8[7]);
    }
    __syncthreads();
    // dZ2 = (H2 > 0) dO W3 (FP32, then BF16) over H2, and its fragments
    {
      float d[4][kOut];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float* p = dout + (quarter * 32 + 8 * i + g) * kOutPad;
        const float4 a = *reinterpret_cast<const float4*>(p);
        const float2 b = *reinterpret_cast<const float2*>(p + 4);
        d[i][0] = a.x, d[i][1] = a.y, d[i][2] = a.z, d[i][3] = a.w, d[i][4] = b.x, d[i][5] = b.y;
      }
#pragma unroll 1
      for (int b = 0; b < 4; ++b) {
        uint32_t p[2][4];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          float z[4][2] = {};
#pragma unroll
          for (int o = 0; o < kOut; ++o) {
            const float2 w = *reinterpret_cast<const float2*>(w3f + o * kHid + 64 * grp + 16 * b + 8 * j + 2 * q);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              z[i][0] += d[i][o] * w.x;
              z[i][1] += d[i][o] * w.y;
            }
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const uint32_t mk = mask2[i >> 1] >> (8 * b + 4 * j + 2 * (i & 1));
            p[i >> 1][2 * j + (i & 1)] = pack_bf16x2((mk & 1u) ? z[i][0] : 0.0f, (mk & 2u) ? z[i][1] : 0.0f);
          }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          tmem_st_frag8(tacc2 + tw + ((uint32_t)(16 * h) << 16) + 8u * b, p[h]);
          lt_put_frag<true>(f.z2 + fo + h * kFragTile + b * 32, p[h], lane);
        }
      }
      tmem_st_wait();
    }
    lt_sync();
    // dH1 = dZ2 W2 (W2's rows, the units of layer 2, are K: MN-major)
    if (tid == 0) {
      for (int ks = 0; ks < kHid / 16; ++ks)
        tc_mma_bf16_ta(tacc, tacc2 + tf_a_col(ks), smem_desc(sw2 + (uint32_t)ks * 2u * 128u, 128, kHid * 16u),
                       idesc_bf16_f32_t(kLtRows, kHid, 0, 1), ks > 0 ? 1u : 0u);
      tc_commit(&bar_mma);
    }
    float* vec = f.vec + (long long)tile * kVecLd;
    if (warp < 4) {
      // db3 and the Huber sum meanwhile: lanes, then warps in order
      const float* dO = dout + tid * kOutPad;
      float s[kOutPad];
#pragma unroll
      for (int k = 0; k < kOutPad; ++k) {
        s[k] = dO[k];
        for (int off = 16; off > 0; off >>= 1) s[k] += __shfl_xor_sync(kFull, s[k], off);
        if (lane == 0) dsum_sh[warp][k] = s[k];
      }
    }
    mma_wait();
    if (ok) {
      // dZ1 = (H1 > 0) dH1: its fragments (BF16), db1 from the FP32 values
#pragma unroll 1
      for (int b = 0; b < 4; ++b) {
        uint32_t r[2][8];
        tmem_ld_frag16_nowait(tacc + tw + 16u * b, r[0]);
        tmem_ld_frag16_nowait(tacc + tw + (16u << 16) + 16u * b, r[1]);
        tmem_ld_wait();
        float cs[4] = {};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t p[4];
#pragma unroll
          for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const uint32_t mk = mask1[h] >> (8 * b + 4 * j + 2 * i);
              const float x = (mk & 1u) ? __uint_as_float(r[h][4 * j + 2 * i]) : 0.0f;
              const float y = (mk & 2u) ? __uint_as_float(r[h][4 * j + 2 * i + 1]) : 0.0f;
              cs[2 * j] += x;
              cs[2 * j + 1] += y;
              p[2 * j + i] = pack_bf16x2(x, y);
            }
          lt_put_frag<true>(f.z1 + fo + h * kFragTile + b * 32, p, lane);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
#pragma unroll
          for (int off = 4; off < 32; off <<= 1) cs[j] += __shfl_xor_sync(kFull, cs[j], off);
          if (g == 0) red[quarter * kHid + 64 * grp + 16 * b + 8 * (j >> 1) + 2 * q + (j & 1)] = cs[j];
        }
      }
    }
    lt_sync();  // also: tensor memory and X are free for the next tile
    if (ok) {
      if (tid < kHid) {
        vec[tid] = ((red[tid] + red[kHid + tid]) + red[2 * kHid + tid]) + red[3 * kHid + tid];
      } else if (tid < kHid + kOutPad && tid != kHid + kOut) {
        const int k = tid - kHid;
        vec[k < kOut ? kBigB3 + k : kBigHub] =
            ((dsum_sh[0][k] + dsum_sh[1][k]) + dsum_sh[2][k]) + dsum_sh[3][k];
      }
    }
  }
  if (!ok && tid == 0) {
    // no update this step; what is in flight gets one more bounded wait
    atomicOr(fail, kTdFailCopy);
    mbar_wait(&bar_w1, wphase, kTcTries);
    mbar_wait(&bar_w2, wphase, kTcTries);
    if (mma_out) mbar_wait(&bar_mma, phase ^ 1u, kTcTries);
    if (kRanks > 1 && rank != 0) mbar_wait(&bar_steps, 0u, kTcTries);
  }
  lt_sync();
  if (warp == 0) tmem_free(tacc, 512);
}

// ------------------------------------------------------------- host side

namespace {
#define SG_CUDA(call)                                        \
  do {                                                       \
    cudaError_t e_ = (call);                                 \
    if (e_ != cudaSuccess) return sg_set_cuda_error(e_, #call); \
  } while (0)

size_t fwd_smem(const ImgLayout& L, int rows = kTile) {
  return (size_t)L.bytes + (size_t)rows * L.ld1 * 2 + 2ull * rows * kLdh * 2 + (size_t)rows * kOutPad * 4;
}
// The fused rollout's: one activation buffer.
size_t roll_smem(const ImgLayout& L, int rows) { return fwd_smem(L, rows) - (size_t)rows * kLdh * 2; }
size_t grad_smem(const ImgLayout& L) {
  return (size_t)L.bytes + (size_t)kTile * L.ld1 * 2 + 3ull * kTile * kLdh * 2 + 2ull * kTile * kOutPad * 4;
}

int set_smem_attr(const void* fn, size_t bytes) {
  SG_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
  return SG_OK;
}

int rebuild_image(sg_qnet* q, const float* th, uint8_t* img, cudaStream_t st) {
  const int n = image_elems(q->IL);
  k_build_image<<<(n + 255) / 256, 256, 0, st>>>(th, img, q->IL, q->PL);
  SG_CUDA(cudaGetLastError());
  // the copy in the tensor cores' layout (a TD step updates both in place)
  k_tc_image<<<44, 256, 0, st>>>(img, q->IL, img == q->img ? q->img_tc : q->img_tc_t);
  SG_CUDA(cudaGetLastError());
  return SG_OK;
}

void free_qnet(sg_qnet* q) {
  if (!q) return;
  cudaFree(q->master);
  cudaFree(q->target);
  cudaFree(q->adam_m);
  cudaFree(q->adam_v);
  cudaFree(q->img);
  cudaFree(q->img_t);
  cudaFree(q->step);
  cudaFree(q->td_fail);
  cudaFree(q->frag);
  cudaFree(q->img_tc);
  cudaFree(q->img_tc_t);
  delete q;
}
}  // namespace

#ifdef SG_DEBUG_BOUNDS
// This translation unit's debug bounds flag (read and cleared by sg_sim_status).
int sg_take_debug_bounds_qnet(unsigned* v) {
  unsigned z = 0;
  cudaError_t e = cudaMemcpyFromSymbol(v, g_debug_bounds, sizeof(unsigned));
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_debug_bounds, &z, sizeof(unsigned));
  return e == cudaSuccess ? SG_OK : sg_set_cuda_error(e, "debug bounds flag");
}
#endif

extern "C" int sg_qnet_create(int32_t n_in, int32_t arch, int32_t max_batch, uint64_t seed, sg_qnet_t* out) {
  SG_RANGE("sg_qnet_create");
  if (!out || n_in < 1 || n_in > 69 || max_batch < 1 || max_batch > (1 << 16)) return SG_E_INVAL;
  if (arch != SG_QNET_DUELING && arch != SG_QNET_PAPER) return SG_E_INVAL;
  *out = nullptr;
  sg_qnet* q = new (std::nothrow) sg_qnet();
  if (!q) return SG_E_OOM;
  q->n_in = n_in;
  q->arch = arch;
  q->IL = img_layout(n_in, arch == SG_QNET_PAPER ? 1 : 0);
  q->PL = param_layout(n_in);
  q->max_batch = (max_batch + kTile - 1) / kTile * kTile;
  cudaGetDevice(&q->device);
  const size_t P = (size_t)q->PL.total;
  // fragment tiles of the largest batch: whole 128-sample tiles from kLtMinBatch
  const int tiles = q->max_batch >= kLtMinBatch ? (q->max_batch + kLtRows - 1) / kLtRows * kLtSub : q->max_batch / kTile;
  cudaError_t e = cudaSuccess;
  auto alloc = [&](void** p, size_t b) {
    if (e == cudaSuccess) e = cudaMalloc(p, b);
  };
  alloc((void**)&q->master, P * 4);
  alloc((void**)&q->target, P * 4);
  alloc((void**)&q->adam_m, P * 4);
  alloc((void**)&q->adam_v, P * 4);
  alloc((void**)&q->img, (size_t)q->IL.bytes);
  alloc((void**)&q->img_t, (size_t)q->IL.bytes);
  alloc((void**)&q->step, 8);
  alloc((void**)&q->td_fail, 8);
  alloc(&q->frag, td_frag_bytes(tiles, q->IL.k1));
  alloc((void**)&q->img_tc, tc_img(q->IL.k1).bytes);
  alloc((void**)&q->img_tc_t, tc_img(q->IL.k1).bytes);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&q->sms, cudaDevAttrMultiProcessorCount, q->device);
  if (e != cudaSuccess) {
    free_qnet(q);
    sg_set_cuda_error(e, "cudaMalloc");
    return SG_E_OOM;
  }
  int rc = SG_OK;
  if (e == cudaSuccess) e = cudaMemset(q->adam_m, 0, P * 4);
  if (e == cudaSuccess) e = cudaMemset(q->adam_v, 0, P * 4);
  if (e == cudaSuccess) e = cudaMemset(q->step, 0, 8);
  if (e == cudaSuccess) e = cudaMemset(q->td_fail, 0, 8);
  if (e == cudaSuccess) e = cudaMemset(q->img, 0, (size_t)q->IL.bytes);
  if (e == cudaSuccess) e = cudaMemset(q->img_t, 0, (size_t)q->IL.bytes);
  if (e == cudaSuccess) {
    k_init_params<<<((int)P + 255) / 256, 256>>>(q->master, q->PL, n_in, q->IL.plain, seed);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) rc = rebuild_image(q, q->master, q->img, 0);
  if (e == cudaSuccess && rc == SG_OK) e = cudaMemcpy(q->target, q->master, P * 4, cudaMemcpyDeviceToDevice);
  if (e == cudaSuccess && rc == SG_OK) e = cudaMemcpy(q->img_t, q->img, (size_t)q->IL.bytes, cudaMemcpyDeviceToDevice);
  if (e == cudaSuccess && rc == SG_OK)
    e = cudaMemcpy(q->img_tc_t, q->img_tc, tc_img(q->IL.k1).bytes, cudaMemcpyDeviceToDevice);
  if (e == cudaSuccess && rc == SG_OK) e = cudaDeviceSynchronize();
  if (e != cudaSuccess || rc != SG_OK) {
    free_qnet(q);
    return e != cudaSuccess ? sg_set_cuda_error(e, "sg_qnet_create") : rc;
  }
  // The limit is a property of the kernel, shared by every handle: set it for
  // the widest supported input so that a narrower network created later
  // cannot lower it below what a wider one launches with.
  const ImgLayout widest = img_layout(69);
  if ((rc = set_smem_attr((const void*)k_qnet_forward_tc, kTcSmemLaunch)) ||
      (rc = set_smem_attr((const void*)k_rollout_q_tc<false>, qt_smem().bytes)) ||
      (rc = set_smem_attr((const void*)k_rollout_q_tc<true>, qt_smem().bytes)) ||
      (rc = set_smem_attr((const void*)k_rollout_q<1, false, false>, roll_smem(widest, 16))) ||
      (rc = set_smem_attr((const void*)k_rollout_q<1, false, true>, roll_smem(widest, 16))) ||
      (rc = set_smem_attr((const void*)k_rollout_q<2, false, false>, roll_smem(widest, 32))) ||
      (rc = set_smem_attr((const void*)k_rollout_q<2, false, true>, roll_smem(widest, 32))) ||
      (rc = set_smem_attr((const void*)k_rollout_q<1, true, false>, roll_smem(widest, 16))) ||
      (rc = set_smem_attr((const void*)k_rollout_q<1, true, true>, roll_smem(widest, 16))) ||
      (rc = set_smem_attr((const void*)k_rollout_q<2, true, false>, roll_smem(widest, 32))) ||
      (rc = set_smem_attr((const void*)k_rollout_q<2, true, true>, roll_smem(widest, 32))) ||
      (rc = set_smem_attr((const void*)k_td_tile<1>, grad_smem(widest))) ||
      (rc = set_smem_attr((const void*)k_td_tile<kTpRanks>, grad_smem(widest))) ||
      (rc = set_smem_attr((const void*)k_td_tc<1>, lt_smem(80).bytes)) ||
      (rc = set_smem_attr((const void*)k_td_tc<kTpRanks>, lt_smem(80).bytes)) ||
      (rc = set_smem_attr((const void*)k_td_update_split<1>, split_smem(1))) ||
      (rc = set_smem_attr((const void*)k_td_update_split<kSplit>, split_smem(kSplit)))) {
    free_qnet(q);
    return rc;
  }
  // clusters of the learners that run at once (one CTA per SM): more tiles than
  // that loop over a resident grid, which stages its weights once
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(kTpRanks * 64);
  lc.blockDim = dim3(kThreads);
  lc.dynamicSmemBytes = grad_smem(q->IL);
  cudaLaunchAttribute la[1];
  la[0].id = cudaLaunchAttributeClusterDimension;
  la[0].val.clusterDim.x = kTpRanks, la[0].val.clusterDim.y = 1, la[0].val.clusterDim.z = 1;
  lc.attrs = la;
  lc.numAttrs = 1;
  if (cudaOccupancyMaxActiveClusters(&q->td_clusters, k_td_tile<kTpRanks>, &lc) != cudaSuccess || q->td_clusters < 1) {
    cudaGetLastError();
    q->td_clusters = std::max(1, q->sms / (kTpRanks + 1));
  }
  *out = q;
  return SG_OK;
}

extern "C" int sg_qnet_destroy(sg_qnet_t q) {
  SG_RANGE("sg_qnet_destroy");
  if (!q) return SG_E_INVAL;
  cudaDeviceSynchronize();
  free_qnet(q);
  return SG_OK;
}

// The network's own (compact) parameter vector <-> the padded one the
// kernels use (identity for the dueling network).
static int64_t compact_params(const sg_qnet* q) { return q->IL.plain ? paper_params(q->n_in) : q->PL.total; }
static void to_padded(const sg_qnet* q, const float* compact, std::vector<float>& padded) {
  padded.assign((size_t)q->PL.total, 0.0f);
  for (int i = 0; i < q->PL.total; ++i) {
    const int j = q->IL.plain ? paper_index(i, q->PL, q->n_in) : i;
    if (j >= 0) padded[(size_t)i] = compact[j];
  }
}
static void to_compact(const sg_qnet* q, const std::vector<float>& padded, float* compact) {
  for (int i = 0; i < q->PL.total; ++i) {
    const int j = q->IL.plain ? paper_index(i, q->PL, q->n_in) : i;
    if (j >= 0) compact[j] = padded[(size_t)i];
  }
}
static int upload(const sg_qnet* q, float* dev, const float* host) {
  std::vector<float> v;
  to_padded(q, host, v);
  SG_CUDA(cudaMemcpy(dev, v.data(), v.size() * 4, cudaMemcpyHostToDevice));
  return SG_OK;
}
static int download(const sg_qnet* q, const float* dev, float* host) {
  std::vector<float> v((size_t)q->PL.total);
  SG_CUDA(cudaMemcpy(v.data(), dev, v.size() * 4, cudaMemcpyDeviceToHost));
  to_compact(q, v, host);
  return SG_OK;
}

extern "C" int sg_qnet_num_params(sg_qnet_t q, int64_t* n) {
  SG_RANGE("sg_qnet_num_params");
  if (!q || !n) return SG_E_INVAL;
  *n = compact_params(q);
  return SG_OK;
}

extern "C" int sg_qnet_set_params(sg_qnet_t q, const float* host, int64_t n, int32_t which) {
  SG_RANGE("sg_qnet_set_params");
  if (!q || !host || n != compact_params(q) || which < 0 || which > 2) return SG_E_INVAL;
  SG_CUDA(cudaDeviceSynchronize());
  if (which == 0 || which == 2) {
    int rc = upload(q, q->master, host);
    if (!rc) rc = rebuild_image(q, q->master, q->img, 0);
    if (rc) return rc;
  }
  if (which == 1 || which == 2) {
    int rc = upload(q, q->target, host);
    if (!rc) rc = rebuild_image(q, q->target, q->img_t, 0);
    if (rc) return rc;
  }
  SG_CUDA(cudaDeviceSynchronize());
  return SG_OK;
}

extern "C" int sg_qnet_get_params(sg_qnet_t q, float* host, int64_t n, int32_t which) {
  SG_RANGE("sg_qnet_get_params");
  if (!q || !host || n != compact_params(q) || which < 0 || which > 1) return SG_E_INVAL;
  SG_CUDA(cudaDeviceSynchronize());
  return download(q, which == 0 ? q->master : q->target, host);
}

extern "C" int sg_qnet_get_optimizer(sg_qnet_t q, float* m_host, float* v_host, int64_t n, uint64_t* steps) {
  SG_RANGE("sg_qnet_get_optimizer");
  if (!q || n != compact_params(q)) return SG_E_INVAL;
  SG_CUDA(cudaDeviceSynchronize());
  int rc = SG_OK;
  if (m_host) rc = download(q, q->adam_m, m_host);
  if (!rc && v_host) rc = download(q, q->adam_v, v_host);
  if (rc) return rc;
  if (steps) SG_CUDA(cudaMemcpy(steps, q->step, 8, cudaMemcpyDeviceToHost));
  return SG_OK;
}

extern "C" int sg_qnet_set_rollout_rows(sg_qnet_t q, int32_t rows) {
  SG_RANGE("sg_qnet_set_rollout_rows");
  if (!q || (rows != 0 && rows != 16 && rows != 32 && rows != 128)) return SG_E_INVAL;
  q->rollout_mt = rows / 16;
  return SG_OK;
}

extern "C" int sg_qnet_set_grid_limit(sg_qnet_t q, int32_t rollout_ctas, int32_t learner_ctas) {
  SG_RANGE("sg_qnet_set_grid_limit");
  if (!q || rollout_ctas < 0 || learner_ctas < 0) return SG_E_INVAL;
  q->lim_rollout = rollout_ctas;
  q->lim_learner = learner_ctas;
  return SG_OK;
}

extern "C" int sg_qnet_copy_params(sg_qnet_t dst, sg_qnet_t src, sg_stream_t stream) {
  SG_RANGE("sg_qnet_copy_params");
  if (!dst || !src || dst->n_in != src->n_in || dst->arch != src->arch) return SG_E_INVAL;
  const size_t P = (size_t)src->PL.total;
  SG_CUDA(cudaMemcpyAsync(dst->master, src->master, P * 4, cudaMemcpyDeviceToDevice, stream));
  SG_CUDA(cudaMemcpyAsync(dst->img, src->img, (size_t)src->IL.bytes, cudaMemcpyDeviceToDevice, stream));
  SG_CUDA(cudaMemcpyAsync(dst->img_tc, src->img_tc, tc_img(src->IL.k1).bytes, cudaMemcpyDeviceToDevice, stream));
  return SG_OK;
}

extern "C" int sg_qnet_set_optimizer(sg_qnet_t q, const float* m_host, const float* v_host, int64_t n,
                                     uint64_t steps) {
  SG_RANGE("sg_qnet_set_optimizer");
  if (!q || !m_host || !v_host || n != compact_params(q)) return SG_E_INVAL;
  SG_CUDA(cudaDeviceSynchronize());
  int rc = upload(q, q->adam_m, m_host);
  if (!rc) rc = upload(q, q->adam_v, v_host);
  if (rc) return rc;
  const unsigned long long st = steps;
  SG_CUDA(cudaMemcpy(q->step, &st, 8, cudaMemcpyHostToDevice));
  return SG_OK;
}

extern "C" int sg_qnet_forward(sg_qnet_t q, const float* obs_dev, int32_t M, float* q_dev, sg_stream_t stream) {
  SG_RANGE("sg_qnet_forward");
  if (!q || !obs_dev || !q_dev || M < 1) return SG_E_INVAL;
  // a persistent grid over the 128-row tiles
  const int ntiles = (M + kTcRows - 1) / kTcRows;
  k_qnet_forward_tc<<<std::min(ntiles, q->sms), kTfThreads, kTcSmemLaunch, stream>>>(q->img, q->img_tc, q->IL,
                                                                                     obs_dev, M, q_dev);
  SG_CUDA(cudaGetLastError());
  return SG_OK;
}

extern "C" int sg_replay_create(int32_t slots_per_env, int32_t n_envs, int32_t obs_dim, int32_t reserve_slots,
                                sg_replay_t* out) {
  SG_RANGE("sg_replay_create");
  if (!out || slots_per_env < 1 || n_envs < 1 || obs_dim < 1) return SG_E_INVAL;
  if (reserve_slots < 0 || reserve_slots >= slots_per_env) return SG_E_INVAL;
  const long long cap = (long long)slots_per_env * n_envs;
  if (cap > (1ll << 31)) return SG_E_INVAL;
  *out = nullptr;
  sg_replay* r = new (std::nothrow) sg_replay();
  if (!r) return SG_E_OOM;
  r->cap = cap;
  cudaGetDevice(&r->device);
  r->d.slots = slots_per_env;
  r->d.n_envs = n_envs;
  r->d.obs_dim = obs_dim;
  r->d.reserve = reserve_slots;
  r->d.inv_full = ~0ull / ((unsigned long long)(slots_per_env - reserve_slots) * (unsigned long long)n_envs);
  r->d.inv_slots = ~0ull / (unsigned long long)slots_per_env;
  cudaError_t e = cudaSuccess;
  auto alloc = [&](void** p, size_t b) {
    if (e == cudaSuccess) e = cudaMalloc(p, b);
  };
  alloc((void**)&r->d.s, (size_t)cap * obs_dim * 4);
  alloc((void**)&r->d.s2, (size_t)cap * obs_dim * 4);
  alloc((void**)&r->d.a, (size_t)cap);
  alloc((void**)&r->d.r, (size_t)cap * 4);
  alloc((void**)&r->d.term, (size_t)cap);
  alloc((void**)&r->d.steps, 16);
  if (e == cudaSuccess) e = cudaMemset(r->d.steps, 0, 16);
  if (e != cudaSuccess) {
    cudaFree(r->d.s);
    cudaFree(r->d.s2);
    cudaFree(r->d.a);
    cudaFree(r->d.r);
    cudaFree(r->d.term);
    cudaFree(r->d.steps);
    delete r;
    sg_set_cuda_error(e, "cudaMalloc");
    return SG_E_OOM;
  }
  *out = r;
  return SG_OK;
}

extern "C" int sg_replay_destroy(sg_replay_t r) {
  SG_RANGE("sg_replay_destroy");
  if (!r) return SG_E_INVAL;
  cudaDeviceSynchronize();
  cudaFree(r->d.s);
  cudaFree(r->d.s2);
  cudaFree(r->d.a);
  cudaFree(r->d.r);
  cudaFree(r->d.term);
  cudaFree(r->d.steps);
  delete r;
  return SG_OK;
}

extern "C" int sg_replay_info(sg_replay_t r, int64_t* capacity, uint64_t* steps_recorded, void** s_dev, void** s2_dev,
                              void** a_dev, void** r_dev, void** term_dev) {
  SG_RANGE("sg_replay_info");
  if (!r) return SG_E_INVAL;
  if (capacity) *capacity = r->cap;
  if (steps_recorded) {
    SG_CUDA(cudaDeviceSynchronize());
    SG_CUDA(cudaMemcpy(steps_recorded, r->d.steps, 8, cudaMemcpyDeviceToHost));
  }
  if (s_dev) *s_dev = r->d.s;
  if (s2_dev) *s2_dev = r->d.s2;
  if (a_dev) *a_dev = r->d.a;
  if (r_dev) *r_dev = r->d.r;
  if (term_dev) *term_dev = r->d.term;
  return SG_OK;
}

extern "C" int sg_replay_read(sg_replay_t r, int64_t first, int64_t count, float* s_host, float* s2_host,
                              uint8_t* a_host, float* r_host, uint8_t* term_host) {
  SG_RANGE("sg_replay_read");
  if (!r || first < 0 || count < 0 || first + count > r->cap) return SG_E_INVAL;
  SG_CUDA(cudaDeviceSynchronize());
  const size_t od = (size_t)r->d.obs_dim;
  if (s_host) SG_CUDA(cudaMemcpy(s_host, r->d.s + first * od, count * od * 4, cudaMemcpyDeviceToHost));
  if (s2_host) SG_CUDA(cudaMemcpy(s2_host, r->d.s2 + first * od, count * od * 4, cudaMemcpyDeviceToHost));
  if (a_host) SG_CUDA(cudaMemcpy(a_host, r->d.a + first, count, cudaMemcpyDeviceToHost));
  if (r_host) SG_CUDA(cudaMemcpy(r_host, r->d.r + first, count * 4, cudaMemcpyDeviceToHost));
  if (term_host) SG_CUDA(cudaMemcpy(term_host, r->d.term + first, count, cudaMemcpyDeviceToHost));
  return SG_OK;
}

extern "C" int sg_replay_write(sg_replay_t r, int64_t first, int64_t count, const float* s_host, const float* s2_host,
                               const uint8_t* a_host, const float* r_host, const uint8_t* term_host,
                               uint64_t steps_recorded) {
  SG_RANGE("sg_replay_write");
  if (!r || first < 0 || count < 0 || first + count > r->cap) return SG_E_INVAL;
  if (count > 0 && (!s_host || !s2_host || !a_host || !r_host || !term_host)) return SG_E_INVAL;
  SG_CUDA(cudaDeviceSynchronize());
  const size_t od = (size_t)r->d.obs_dim;
  if (count > 0) {
    SG_CUDA(cudaMemcpy(r->d.s + first * od, s_host, count * od * 4, cudaMemcpyHostToDevice));
    SG_CUDA(cudaMemcpy(r->d.s2 + first * od, s2_host, count * od * 4, cudaMemcpyHostToDevice));
    SG_CUDA(cudaMemcpy(r->d.a + first, a_host, count, cudaMemcpyHostToDevice));
    SG_CUDA(cudaMemcpy(r->d.r + first, r_host, count * 4, cudaMemcpyHostToDevice));
    SG_CUDA(cudaMemcpy(r->d.term + first, term_host, count, cudaMemcpyHostToDevice));
  }
  const unsigned long long st = steps_recorded;
  SG_CUDA(cudaMemcpy(r->d.steps, &st, 8, cudaMemcpyHostToDevice));
  return SG_OK;
}

// VEM noise per env at T = n * t (t: env 0's step counter); see sg_vem_eps.
__global__ void k_vem_eps(const uint32_t* __restrict__ t_dev, int n, float e_min, float e_max, double or_start,
                          double or_final, double decay, float* __restrict__ eps) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double T = (double)n * (double)t_dev[0];
  const double frac = T / decay < 1.0 ? T / decay : 1.0;
  const double OR = or_start + (or_final - or_start) * frac;
  const double first = (double)n - OR;
  double e = (double)e_min;
  if ((double)i >= first) e = (double)e_min + (double)e_max * (((double)i - first) / (OR - 1.0));
  eps[i] = (float)e;
}

extern "C" int sg_vem_eps(sg_sim_t sim, float e_min, float e_max, double or_start, double or_final,
                          double decay_steps, float* eps_dev, sg_stream_t stream) {
  SG_RANGE("sg_vem_eps");
  if (!sim || !eps_dev) return SG_E_INVAL;
  const int n = sim->dc.n_envs;
  if (!(or_final >= 2.0 && or_final <= n && or_start >= 2.0 && or_start <= n && decay_steps > 0.0 &&
        e_min >= 0.0f && e_max >= 0.0f))
    return SG_E_INVAL;
  // u is [4][n]: ep_step, ep_id, t, fifo
  k_vem_eps<<<(n + 255) / 256, 256, 0, (cudaStream_t)stream>>>(sim->ustate + 2 * (size_t)n, n, e_min, e_max, or_start,
                                                               or_final, decay_steps, eps_dev);
  SG_CUDA(cudaGetLastError());
  return SG_OK;
}

int sg_rollout_eps_q(sg_sim* sim, int K, sg_qnet* q, const float* eps, sg_replay* rp, float* obs, float* obs_seq,
                     uint8_t* act_seq, float* rew_seq, uint8_t* done_seq, cudaStream_t stream) {
  if (q->n_in != sim->dc.obs_dim) return SG_E_INVAL;
  ReplayDev rd;
  std::memset(&rd, 0, sizeof(rd));
  if (rp) {
    if (rp->d.n_envs != sim->dc.n_envs || rp->d.obs_dim != sim->dc.obs_dim) return SG_E_INVAL;
    rd = rp->d;
  }
  // 32 envs per CTA (two m-tiles) when that fills fewer waves than 16; the
  // shared-memory image limits a CTA to one per SM either way
  int sms = 0;
  SG_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, sim->device));
  const int n = sim->dc.n_envs;
  const int waves16 = ((n + 15) / 16 + sms - 1) / sms, waves32 = ((n + 31) / 32 + sms - 1) / sms;
  // with dynamic obstacles the 32-env CTA (64 registers a thread) spills the
  // disc registers: 16 envs per CTA unless asked otherwise
  const bool dyn = sim->dc.n_dyn > 0;
  // 128 envs per CTA on the tcgen05 kernel when they fill every SM at least
  // once (or when asked for), without dynamic obstacles
  const bool tc = !dyn && (q->rollout_mt == 8 || (q->rollout_mt == 0 && n >= kQtEnvs * sms));
  const int mt = q->rollout_mt > 0 && q->rollout_mt <= 2 ? q->rollout_mt : (!dyn && waves32 < waves16 ? 2 : 1);
  if (tc) {
    // more than one wave of 128-env CTAs: slice the rollout into 4 to 6
    // segments over a resident grid so that no SM idles in a part-empty last
    // wave (the grid within the network's CTA cap, when one is set): the
    // count whose (block, segment) items fill the last round of the grid
    // best (65,536 envs: 5 segments, 429.7 M env-steps/s against 425.8 M
    // with 4, 427.0 M with 6, 413.5 M with 8)
    const int cap = q->lim_rollout > 0 ? std::min(q->lim_rollout, sms) : sms;
    const int nblk = (n + kQtEnvs - 1) / kQtEnvs;
    int seg = 0;
    if (nblk > cap && K >= 4) {
      double best = 0.0;
      for (int ns = 4; ns <= 6 && ns <= K; ++ns) {
        const int sl = (K + ns - 1) / ns;
        const long long items = (long long)nblk * ((K + sl - 1) / sl);
        const long long rounds = (items + cap - 1) / cap;
        const double fill = (double)items / ((double)rounds * cap);
        if (fill > best + 1e-9) {
          best = fill;
          seg = sl;
        }
      }
    }
    int grid = nblk;
    if (seg > 0) {
      grid = std::min(nblk * ((K + seg - 1) / seg), cap);
      SG_CUDA(cudaMemsetAsync(sim->q_sync_dev, 0, sizeof(unsigned) * (size_t)(nblk + 2), stream));
    }
    (sim->dc.scan_fast ? k_rollout_q_tc<true> : k_rollout_q_tc<false>)<<<grid, kQtThreads, qt_smem().bytes, stream>>>(
        sim->dc, sg_sim_ptrs(sim), q->img, q->img_tc, q->IL, K, eps, rd, rp ? 1 : 0, sim->map_order_dev, seg,
        seg > 0 ? sim->q_sync_dev : nullptr, obs, obs_seq, act_seq, rew_seq, done_seq);
  } else {
    // envs per CTA: the full tile, or fewer when the tiles would leave SMs
    // idle (one CTA per SM: the staged image takes the shared memory), down
    // to one: a CTA's steps wait on its slowest env and on its warps' issue
    // slots; 4,096 envs: 152 CTAs of 27 instead of 128 of 32
    const int rows = 16 * mt;
    const int epc = (n + rows - 1) / rows < sms ? (n + sms - 1) / sms : rows;
    const int grid = (n + epc - 1) / epc;
    const bool fast = sim->dc.scan_fast != 0;
    auto kern = mt == 2 ? (dyn ? (fast ? k_rollout_q<2, true, true> : k_rollout_q<2, true, false>)
                               : (fast ? k_rollout_q<2, false, true> : k_rollout_q<2, false, false>))
                        : (dyn ? (fast ? k_rollout_q<1, true, true> : k_rollout_q<1, true, false>)
                               : (fast ? k_rollout_q<1, false, true> : k_rollout_q<1, false, false>));
    kern<<<grid, 512 * mt, roll_smem(q->IL, rows), stream>>>(sim->dc, sg_sim_ptrs(sim), q->img, q->IL, K, eps, rd,
                                                            rp ? 1 : 0, sim->map_order_dev, epc, obs, obs_seq, act_seq,
                                                            rew_seq, done_seq);
  }
  SG_CUDA(cudaGetLastError());
  return SG_OK;
}

extern "C" int sg_td_train_step(sg_qnet_t q, sg_replay_t rp, int32_t batch, float gamma, float lr,
                                int32_t target_every, uint64_t seed, float* loss_dev, float* grad_dev,
                                sg_stream_t stream) {
  SG_RANGE("sg_td_train_step");
  if (!q || !rp || batch < 1 || batch > q->max_batch || rp->d.obs_dim != q->n_in) return SG_E_INVAL;
  if (!(gamma >= 0.0f && gamma <= 1.0f) || !(lr >= 0.0f)) return SG_E_INVAL;
  TdUpdate u;
  u.th = q->master, u.m = q->adam_m, u.v = q->adam_v, u.tgt = q->target;
  u.img = q->img, u.img_t = q->img_t, u.tc = q->img_tc, u.tc_t = q->img_tc_t;
  u.step = q->step, u.fail = q->td_fail, u.tick = q->td_fail + 1;
  u.lr = lr, u.every = target_every, u.loss = loss_dev, u.grad = grad_dev, u.batch = batch;
  u.P = q->PL, u.L = q->IL;
  const bool big = batch >= kLtMinBatch;
  const int rows = big ? kLtRows : kTile, ntiles = (batch + rows - 1) / rows;
  // a cluster per tile, or with a limit single CTAs: a cluster starts only where one
  // GPC has that many SMs free, and what a rollout leaves free is spread over all of
  // them.  The same for the update's clusters of eight up to three SMs a GPC.
  // 65,536 envs x 32 steps beside 16 steps of batch 4,096, learner on 4 / 8 / 12 /
  // 16 / 24 / 48 SMs, ms: clusters 10.9 / 7.2 / 5.4 / 5.2 / 4.4 / 4.4, CTAs for the
  // tiles only 6.9 / 5.2 / 4.8 / 4.4 / 3.62 / 4.36, for both 6.0 / 3.9 / 3.27 / 3.36 /
  // 3.56 / 4.41; one after the other 3.40.  Where the rollout ends early the
  // update's clusters are faster: 19,456 envs x 8 beside 32 steps, 8 / 24 / 48 SMs: 8.7 /
  // 2.79 / 1.77, 4.6 / 2.66 / 1.68, 5.7 / 3.78 / 2.81.
  const bool own = q->lim_learner > 0 && q->lim_learner < q->sms, own_update = own && q->lim_learner < 24;
  const int fit = own ? q->lim_learner : std::max(1, std::min(q->td_clusters, q->sms / kTpRanks));
  // evenly over the rounds
  const int rounds = (ntiles + fit - 1) / fit, grid = (ntiles + rounds - 1) / rounds * (own ? 1 : kTpRanks);
  const int frags = big ? ntiles * kLtSub : ntiles, items = td_update_items(q->IL.k1);
  const TdFrag f = td_frag(q->frag, frags, q->IL.k1);
  const uint8_t *im = q->img, *im_t = q->img_t, *tc = q->img_tc, *tc_t = q->img_tc_t;
  const unsigned long long* step = q->step;
  if (big) {
    const int parts = own_update ? 1 : kSplit;
    SG_CUDA(sg_launch_pdl(own ? k_td_tc<1> : k_td_tc<kTpRanks>, grid, kThreads, lt_smem(q->IL.k1).bytes, stream, im,
                          im_t, tc, tc_t, q->IL, rp->d, seed, step, batch, gamma, f, q->td_fail));
    SG_CUDA(sg_launch_pdl(own_update ? k_td_update_split<1> : k_td_update_split<kSplit>, td_split_items(q->IL.k1) * parts,
                          split_threads(parts), split_smem(parts), stream, u, f, frags));
    return SG_OK;
  }
  SG_CUDA(sg_launch_pdl(own ? k_td_tile<1> : k_td_tile<kTpRanks>, grid, kThreads, grad_smem(q->IL), stream, im, im_t,
                        q->IL, rp->d, seed, step, batch, gamma, f, q->td_fail));
  if (ntiles <= kTuSlots)
    SG_CUDA(sg_launch_pdl(k_td_update<4, true>, items, 128, 0, stream, u, f, ntiles));
  else
    SG_CUDA(sg_launch_pdl(k_td_update<8, false>, items, 256, 0, stream, u, f, ntiles));
  return SG_OK;
}

// ------------------------------------------------------------------------
// TD loss and gradient without any allocation (sg_td_grad_noalloc).
//
// For callers that must not allocate device memory at all -- code running
// under a fixed memory budget, inside another framework's allocator, or in a
// context where cudaMalloc is not allowed -- and so cannot create a Q-network
// handle.  The caller passes the FP32 parameters and the batch; every
// intermediate buffer (BF16 weight images, TD targets, sample indices,
// per-CTA gradient partials) lives in one file-scope device array that each
// GPU holds from the moment the library is loaded until the process exits.
namespace {
constexpr int kNaMaxBatch = 256;
constexpr int kNaMaxIn = 69;
constexpr int kNaMaxBlk = kNaMaxBatch / kTile;
constexpr int kNaImgBytes = kHid * ((kNaMaxIn + 15) / 16 * 16 + 8) * 2 + kHid * kLdh * 2 + kOutPad * kLdh * 2 +
                            2 * kHid * 4 + kOutPad * 4;
constexpr int kNaImgSlot = (kNaImgBytes + 255) / 256 * 256;
// The widest image (69 inputs) is staged by the TD kernels in one mbarrier
// phase, whose transaction count holds at most 2^20 - 1 bytes.
static_assert(kNaImgBytes + 16 < (1 << 20), "one weight image fits an mbarrier phase's transaction count");
constexpr int kNaMaxParams = kHid * kNaMaxIn + kHid + kHid * kHid + kHid + kOut * kHid + kOut;
constexpr long long kNaOffY = 2ll * kNaImgSlot;
constexpr long long kNaOffIdx = kNaOffY + kNaMaxBatch * 4;
constexpr long long kNaOffFail = kNaOffIdx + kNaMaxBatch * 4;
constexpr long long kNaOffPartial = (kNaOffFail + 4 + 255) / 256 * 256;
constexpr long long kNaBytes = kNaOffPartial + (long long)kNaMaxBlk * partial_stride(kNaMaxParams) * 4;
}  // namespace

static __device__ __align__(256) unsigned char g_td_noalloc_scratch[kNaBytes];

// Double-DQN targets for an explicit batch (sample i is row i).
__global__ void __launch_bounds__(kThreads, 1)
    k_td_target_given(const uint8_t* __restrict__ img, const uint8_t* __restrict__ img_t, ImgLayout L, ReplayDev b,
                      int batch, float gamma, float* __restrict__ y, int* __restrict__ idx) {
  extern __shared__ __align__(16) uint8_t smem[];
  uint8_t* sw = smem;
  bf16* X = reinterpret_cast<bf16*>(smem + L.bytes);
  bf16* H1 = X + kTile * L.ld1;
  bf16* H2 = H1 + kTile * kLdh;
  float* O = reinterpret_cast<float*>(H2 + kTile * kLdh);
  __shared__ int rows[kTile];
  __shared__ int astar[kTile];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * kTile + warp;
  if (lane == 0) {
    rows[warp] = i < batch ? i : -1;
    if (i < batch) idx[i] = i;
  }
  stage_image(sw, img, L.bytes);
  __syncthreads();
  gather_tile(X, L.ld1, b.s2, rows, b.obs_dim, warp, lane);
  __syncthreads();
  mlp_tile(qw_at(sw, L), X, H1, H2, O, warp, lane);
  if (lane == 0) astar[warp] = (int)greedy_action(O + warp * kOutPad, nullptr, L.plain);
  __syncthreads();
  stage_image(sw, img_t, L.bytes);
  __syncthreads();
  mlp_tile(qw_at(sw, L), X, H1, H2, O, warp, lane);
  if (lane == 0 && i < batch) {
    float qv[5];
    greedy_action(O + warp * kOutPad, qv, L.plain);
    const float nt = b.term[i] ? 0.0f : 1.0f;
    y[i] = b.r[i] + gamma * nt * qv[astar[warp]];
  }
}

namespace {
constexpr int kNaMaxDevices = 64;
std::mutex g_na_mutex;
unsigned char* g_na_ptr[kNaMaxDevices] = {};

// Once per device, with that device current: the device address of the
// scratch array (in host code its name is only a host-side stand-in) and
// the shared-memory limits of the kernels this path launches.
int na_setup(unsigned char** out) {
  int dev = 0;
  SG_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kNaMaxDevices) return sg_set_error_text("sg_td_grad_noalloc: device ordinal too large", SG_E_INVAL);
  std::lock_guard<std::mutex> lock(g_na_mutex);
  if (!g_na_ptr[dev]) {
    void* p = nullptr;
    SG_CUDA(cudaGetSymbolAddress(&p, g_td_noalloc_scratch));
    const ImgLayout L = img_layout(kNaMaxIn);
    int rc = set_smem_attr((const void*)k_td_target_given, fwd_smem(L));
    if (!rc) rc = set_smem_attr((const void*)k_td_grad, grad_smem(L));
    if (rc) return rc;
    g_na_ptr[dev] = static_cast<unsigned char*>(p);
  }
  *out = g_na_ptr[dev];
  return SG_OK;
}
}  // namespace

extern "C" int sg_td_grad_noalloc(const float* params_dev, const float* target_params_dev, int32_t n_in,
                                  const float* s_dev, const uint8_t* a_dev, const float* r_dev, const float* s2_dev,
                                  const uint8_t* term_dev, int32_t batch, float gamma, float* loss_dev,
                                  float* grad_dev, sg_stream_t stream) {
  SG_RANGE("sg_td_grad_noalloc");
  if (!params_dev || !target_params_dev || !s_dev || !a_dev || !r_dev || !s2_dev || !term_dev || !grad_dev)
    return sg_set_error_text("sg_td_grad_noalloc: a required pointer is NULL", SG_E_INVAL);
  if (n_in < 1 || n_in > kNaMaxIn)
    return sg_set_error_text("sg_td_grad_noalloc: n_in must be in [1, 69] (static scratch limit)", SG_E_INVAL);
  if (batch < 1 || batch > kNaMaxBatch)
    return sg_set_error_text("sg_td_grad_noalloc: batch must be in [1, 256] (static scratch limit)", SG_E_INVAL);
  if (!(gamma >= 0.0f && gamma <= 1.0f)) return sg_set_error_text("sg_td_grad_noalloc: gamma outside [0, 1]", SG_E_INVAL);
  unsigned char* base = nullptr;
  int rc = na_setup(&base);
  if (rc) return rc;
  const ImgLayout IL = img_layout(n_in);
  const ParamLayout PL = param_layout(n_in);
  uint8_t* img = base;
  uint8_t* img_t = base + kNaImgSlot;
  float* y = reinterpret_cast<float*>(base + kNaOffY);
  int* idx = reinterpret_cast<int*>(base + kNaOffIdx);
  float* partial = reinterpret_cast<float*>(base + kNaOffPartial);
  unsigned* fail = reinterpret_cast<unsigned*>(base + kNaOffFail);
  ReplayDev b;
  std::memset(&b, 0, sizeof(b));
  b.s = const_cast<float*>(s_dev);
  b.s2 = const_cast<float*>(s2_dev);
  b.a = const_cast<uint8_t*>(a_dev);
  b.r = const_cast<float*>(r_dev);
  b.term = const_cast<uint8_t*>(term_dev);
  b.slots = 1;
  b.n_envs = batch;
  b.obs_dim = n_in;
  const int ne = image_elems(IL);
  k_build_image<<<(ne + 255) / 256, 256, 0, stream>>>(params_dev, img, IL, PL);
  SG_CUDA(cudaGetLastError());
  k_build_image<<<(ne + 255) / 256, 256, 0, stream>>>(target_params_dev, img_t, IL, PL);
  SG_CUDA(cudaGetLastError());
  const int nblk = (batch + kTile - 1) / kTile;
  SG_CUDA(cudaMemsetAsync(fail, 0, 4, stream));
  k_td_target_given<<<nblk, kThreads, fwd_smem(IL), stream>>>(img, img_t, IL, b, batch, gamma, y, idx);
  SG_CUDA(cudaGetLastError());
  k_td_grad<<<nblk, kThreads, grad_smem(IL), stream>>>(img, IL, PL, b, idx, y, batch, partial, fail);
  SG_CUDA(cudaGetLastError());
  TdUpdate u;
  std::memset(&u, 0, sizeof(u));  // no parameters: loss and gradient only
  u.fail = fail;
  u.loss = loss_dev, u.grad = grad_dev, u.batch = batch;
  u.P = PL, u.L = IL;
  k_grad_sum<<<(PL.total + 256) / 256, 256, 0, stream>>>(u, partial, nblk);
  SG_CUDA(cudaGetLastError());
  return SG_OK;
}
