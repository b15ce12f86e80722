// Training pass of the closure network on the 5th-generation tensor cores
// (tcgen05): for a batch X [M][288] (BF16) with targets T [M][32], the
// forward pass y = W3 tanh(W2 tanh(W1 x + b1) + b2) + b3, the loss
// sum over rows and used outputs of (y - t)^2, its gradient dy = 2 (y - t) /
// (17 M) on the used outputs, the back-propagated dh2 = (dy W3) (1 - h2^2),
// dh1 = (dh2 W2) (1 - h1^2), and every weight and bias gradient, as per-block
// partial sums that mlp_reduce_adam_kernel adds in block order.
//
// One persistent block per SM walks 128-row tiles; thread r and r + 128 own
// row r (TMEM lane r), each half of its columns. Per tile one thread issues,
// in turn: layer 1 (X W1^T), layer 2, layer 3, the two backward products
// (dy W3, dh2 W2) and the three weight-gradient products, each committed to
// one mbarrier that all threads wait on (bounded). Operands are BF16 tiles in
// shared memory: the weights, one bulk copy, and the hidden rows and gradients
// in the canonical layout without swizzle (8-row x 16-byte core matrices), the
// rows of X by TMA in boxes of 64 columns with 128-byte swizzle. The weight
// gradients read the same tiles transposed, as MN-major operands (the transpose
// bits of the instruction descriptor; without swizzle the leading byte offset is
// then the stride between core matrices along K, the batch rows, and the stride
// byte offset the one along M or N):
//   gW1^T [288 x 64] = X^T dh1    (three M = 128 blocks over the features)
//   gW2^T [64 x 64]  = h1^T dh2   gW3^T [64 x 32] = h2^T dy
// with M = 128 rows of which the rows past 288 / 64 are discarded. Their FP32
// accumulators stay in tensor memory over all tiles of the block. The bias
// gradients are FP32 column sums of dy, dh2, dh1 (warp shuffles, then per-warp
// sums in shared memory in a fixed order), so repeated runs agree bit for bit.
//
// A batch of 8192 is 64 tiles, one to a block: the chain through a tile bounds
// it, 33000 cycles of which 13000 went by until the weights and then the rows
// had been copied by the threads, 10000 in column sums by a full butterfly for
// each column and targets read when they were needed. Now both copies are
// asynchronous and start together, the targets are read ahead, a butterfly
// halves its columns at every step (the same sums), and the column sums and the
// gradients of W3 and W2 run beside the products that the chain waits for:
// 22.3 -> 11.8 us.
//
// TMEM (512 columns, 64-column blocks): gW1^T at 0 .. 191, gW2^T at 192,
// gW3^T at 256; layer 1 at 320, then h1 in FP32 (for 1 - h1^2); layer 2 at
// 384, then h2 in FP32, then dh2 W2; layer 3 at 448, then dy W3.
#include <cstdint>

#include "lbrr_chain.cuh"
#include "lbrr_launch.h"
#include "lbrr_mlp.h"
#include "lbrr_act.cuh"
#include "lbrr_tc.cuh"

namespace lbrr {

namespace {

using namespace tc;

constexpr int kRows = kMlpTrainRows;  // 128
constexpr int kThreads = 2 * kRows;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kColG1 = 0, kColG2 = 192, kColG3 = 256, kColL1 = 320, kColL2 = 384,
                   kColL3 = 448;

// shared memory (bytes); every tile but X in the canonical K-major layout of its rows
constexpr uint32_t kSmW1 = 0;                                     // [64][288]
constexpr uint32_t kSmW2 = kSmW1 + kMlpW1Bytes;                  // [64][64]
constexpr uint32_t kSmW3 = kSmW2 + kMlpW2Bytes;                  // [32][64]
constexpr uint32_t kSmW2t = kSmW3 + kMlpW3Bytes;                 // [64][64] = W2^T
constexpr uint32_t kSmW3t = kSmW2t + kMlpW2Bytes;                // [64][32] = W3^T
constexpr uint32_t kSmX = kSmW3t + kMlpW3Bytes;                  // 5 boxes [128][64]
constexpr int kBoxCols = 64, kBoxes = (kMlpIn + kBoxCols - 1) / kBoxCols;
constexpr uint32_t kBoxBytes = kRows * kBoxCols * 2;
constexpr uint32_t kSmH1 = kSmX + kBoxes * kBoxBytes;            // [128][64]
constexpr uint32_t kSmH2 = kSmH1 + kRows * kMlpHidden * 2;       // [128][64]
constexpr uint32_t kSmDy = kSmH2 + kRows * kMlpHidden * 2;       // [128][32]
constexpr uint32_t kSmDh2 = kSmDy + kRows * kMlpOut * 2;         // [128][64]
constexpr uint32_t kSmDh1 = kSmDh2 + kRows * kMlpHidden * 2;     // [128][64]
constexpr uint32_t kSmMisc = kSmDh1 + kRows * kMlpHidden * 2;
// misc: mbarriers, TMEM address, biases b1 b2 b3 (160), per-warp column sums of
// dy, dh2, dh1 (8 warps x 80 columns: a warp covers 32 rows and one half of
// the columns) and per-warp loss sums
constexpr int kGbCols = kMlpOut / 2 + kMlpHidden / 2 + kMlpHidden / 2;  // 80 per half
constexpr uint32_t kSmBias = kSmMisc + 64;
constexpr uint32_t kSmGbw = kSmBias + 4 * (2 * kMlpHidden + kMlpOut);
constexpr uint32_t kSmLossw = kSmGbw + 4 * 8 * kGbCols;
constexpr uint32_t kTrainSmem = kSmLossw + 4 * 8;
static_assert(kSmX % 1024 == 0 && kSmMisc % 16 == 0, "alignment");
static_assert(kTrainSmem <= 232448, "fits the shared memory of one block");
// the transposed reads with M = 128 run past the 288 (X) or 64 (h1, h2) real
// rows into the next tile's bytes (discarded rows): they stay inside the block
static_assert(kSmX + (kBoxes + 1) * kBoxBytes <= kTrainSmem, "X^T reads");
static_assert(kSmH2 + 15 * 1024 + 15 * 128 + 1024 + 128 <= kTrainSmem, "h^T reads");

__host__ __device__ constexpr uint32_t idesc_t(int M, int N) {  // both operands MN-major
  return idesc_bf16(M, N) | (1u << 15) | (1u << 16);
}

// Operand descriptors of a [rows][C] tile (canonical, K-major rows): read
// K-major (K = C, the rows are M or N) or MN-major (K = rows, MN = C).
__device__ __forceinline__ uint64_t kmaj(uint32_t base, int C, int ks) {
  return sdesc(base + 256 * ks, 128, (C / 8) * 128);  // K step ks: 16 columns
}
__device__ __forceinline__ uint64_t mnmaj(uint32_t base, int C, int ks) {
  // K step ks: rows 16 ks .. 16 ks + 15 (two 8-row groups)
  return sdesc(base + 2 * ks * (C / 8) * 128, (C / 8) * 128, 128);
}

// 32 consecutive FP32 TMEM columns of this thread's lane into v
__device__ __forceinline__ void ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t a[16], b[16];
  tmem_ld16_async(taddr, a);
  tmem_ld16_async(taddr + 16, b);
  tmem_wait_ld();
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    v[k] = __uint_as_float(a[k]);
    v[16 + k] = __uint_as_float(b[k]);
  }
}
__device__ __forceinline__ void st32(uint32_t taddr, const float (&v)[32]) {
  uint32_t a[16], b[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    a[k] = __float_as_uint(v[k]);
    b[k] = __float_as_uint(v[16 + k]);
  }
  tmem_st16(taddr, a);
  tmem_st16(taddr + 16, b);
}
// values v[0 .. 8 NC) as BF16 into columns c0 .. of row r of a [rows][C] tile
template <int NC>
__device__ __forceinline__ void put_bf16(unsigned char *tile, int C, int r, int c0,
                                         const float *v) {
#pragma unroll
  for (int k = 0; k < 8 * NC; k += 8)
    *reinterpret_cast<uint4 *>(tile + cm_offset(r, c0 + k, C)) =
        make_uint4(pack_bf16(v[k], v[k + 1]), pack_bf16(v[k + 2], v[k + 3]),
                   pack_bf16(v[k + 4], v[k + 5]), pack_bf16(v[k + 6], v[k + 7]));
}
// column sums over the warp's 32 rows, added to dst[0 .. N): a butterfly in
// which a lane keeps, at every step, the half of the columns that the step's bit
// of its number names (v is used up)
template <int N, int O = 16, int C = N>
__device__ __forceinline__ void warp_col_sums(float (&v)[N], float *dst, int lane) {
  if constexpr (O > 0) {
    constexpr int kHalf = C > 1 ? C / 2 : 1;
    const bool up = C > 1 && (lane & O);
#pragma unroll
    for (int k = 0; k < kHalf; ++k) {
      const float keep = up ? v[k + C / 2] : v[k], send = up ? v[k] : v[k + C / 2];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, send, O);
    }
    warp_col_sums<N, O / 2, kHalf>(v, dst, lane);
  } else if (lane % (32 / N) == 0) {
    dst[lane / (32 / N)] += v[0];
  }
}

template <bool TRACE>
__global__ void __launch_bounds__(kThreads, 1)
    mlp_train_tc_kernel(MlpDevice p, const __grid_constant__ CUtensorMap x_map,
                        const float *T, long long M, float *gpart, float *lpart, int *status,
                        float *trace) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int r = tid & (kRows - 1), half = tid >> 7;
  // products done, weights landed, rows landed, drain
  uint64_t *mbar = reinterpret_cast<uint64_t *>(smem + kSmMisc);
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + kSmMisc + 32);
  float *sb = reinterpret_cast<float *>(smem + kSmBias);
  float *gbw = reinterpret_cast<float *>(smem + kSmGbw) + warp * kGbCols;
  float *lossw = reinterpret_cast<float *>(smem + kSmLossw);
  const uint32_t mbar_a = smem_u32(mbar), mbar_w = smem_u32(mbar + 1);
  const uint32_t mbar_x = smem_u32(mbar + 2), mbar_d = smem_u32(mbar + 3);
  const long long ntiles = (M + kRows - 1) / kRows;

  // ---- weights (and the transposed copies of W2, W3), rows of the first tile
  auto request = [&](long long tile) {  // rows past M are zero
    mbar_expect_tx(mbar_x, kBoxes * kBoxBytes);
#pragma unroll
    for (int k = 0; k < kBoxes; ++k)
      tma_load_2d(smem_u32(smem + kSmX) + k * kBoxBytes, &x_map, k * kBoxCols, (int)(tile * kRows),
                  mbar_x);
  };
  if (tid == 0) {
    for (int k = 0; k < 4; ++k) mbar_init(smem_u32(mbar + k), 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    fence_async_smem();
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  chain_wait();
  if (tid == 0) {
    request(blockIdx.x);  // the launcher starts no block without a tile
    mbar_expect_tx(mbar_w, kMlpWeightBytes);
    bulk_load(smem_u32(smem + kSmW1), p.w1, kMlpWeightBytes, mbar_w);
  }
  for (int c = tid; c < 2 * kMlpHidden + kMlpOut; c += kThreads)
    sb[c] = c < kMlpHidden ? p.b1[c] : (c < 2 * kMlpHidden ? p.b2[c - kMlpHidden]
                                                           : p.b3[c - 2 * kMlpHidden]);
  for (int c = tid; c < 8 * kGbCols; c += kThreads)
    reinterpret_cast<float *>(smem + kSmGbw)[c] = 0.f;
  if (tid < 8) lossw[tid] = 0.f;
  fence_async_smem();
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t lane_addr = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
  const uint32_t sw1 = smem_u32(smem + kSmW1), sw2 = smem_u32(smem + kSmW2);
  const uint32_t sw3 = smem_u32(smem + kSmW3), sw2t = smem_u32(smem + kSmW2t);
  const uint32_t sw3t = smem_u32(smem + kSmW3t), sx = smem_u32(smem + kSmX);
  const uint32_t sh1 = smem_u32(smem + kSmH1), sh2 = smem_u32(smem + kSmH2);
  const uint32_t sdy = smem_u32(smem + kSmDy), sdh2 = smem_u32(smem + kSmDh2);
  const uint32_t sdh1 = smem_u32(smem + kSmDh1);
  const uint32_t lim = wait_limit(status);
  const float inv_n = 1.0f / ((float)M * (float)kMlpOutUsed);
  uint32_t phase = 0, xphase = 0;
  bool ok = true, requested = true;
  // all threads wait for the MMAs committed so far (the same decision in every thread)
  auto sync_mma = [&]() {
    ok = !__syncthreads_or(!mbar_wait(mbar_a, phase, lim));
    if (ok) phase ^= 1;
    fence_after();
    return ok;
  };
  auto handoff = [&]() {  // shared-memory and TMEM writes of every thread before the next MMAs
    tmem_wait_st();
    fence_async_smem();
    fence_before();
    __syncthreads();
    fence_after();
  };

  for (long long tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
    const bool first = tile == blockIdx.x;
    const long long row = tile * kRows + r;
    const bool valid = row < M;
    float *trow = TRACE && valid ? trace + row * kMlpTrace : nullptr;
    // ---- this thread's targets, needed after layer 3; rows
    float t[16];
#pragma unroll
    for (int k = 0; k < 16; ++k)
      t[k] = valid && 16 * half + k < kMlpOutUsed ? T[row * kMlpOut + 16 * half + k] : 0.f;
    if (!first) {
      if (tid == 0) request(tile);
      requested = true;
    }
    ok = !__syncthreads_or(!(mbar_wait(mbar_w, 0, lim) && mbar_wait(mbar_x, xphase, lim)));
    if (!ok) break;
    xphase ^= 1;
    requested = false;
    fence_after();
    // ---- layer 1
    if (tid == 0) {
#pragma unroll 1
      for (int ks = 0; ks < kMlpIn / 16; ++ks)
        umma(tmem + kColL1,
             sdesc_swizzled(sx + (ks / 4) * kBoxBytes + 32 * (ks % 4), 16, 1024, true),
             kmaj(sw1, kMlpIn, ks),
             idesc_bf16(128, kMlpHidden), ks > 0);
      umma_commit(mbar_a);
    }
    if (!sync_mma()) break;
    float v[32];
    ld32(lane_addr + kColL1 + 32 * half, v);
#pragma unroll
    for (int k = 0; k < 32; ++k) v[k] = tanh_approx(v[k] + sb[32 * half + k]);
    st32(lane_addr + kColL1 + 32 * half, v);  // h1 in FP32, for 1 - h1^2
    put_bf16<4>(smem + kSmH1, kMlpHidden, r, 32 * half, v);
    if (TRACE && trow)
#pragma unroll
      for (int k = 0; k < 32; ++k) trow[kTraceH1 + 32 * half + k] = v[k];
    handoff();
    // ---- layer 2
    if (tid == 0) {
#pragma unroll
      for (int ks = 0; ks < kMlpHidden / 16; ++ks)
        umma(tmem + kColL2, kmaj(sh1, kMlpHidden, ks), kmaj(sw2, kMlpHidden, ks),
             idesc_bf16(128, kMlpHidden), ks > 0);
      umma_commit(mbar_a);
    }
    if (!sync_mma()) break;
    ld32(lane_addr + kColL2 + 32 * half, v);
#pragma unroll
    for (int k = 0; k < 32; ++k) v[k] = tanh_approx(v[k] + sb[kMlpHidden + 32 * half + k]);
    st32(lane_addr + kColL2 + 32 * half, v);  // h2 in FP32
    put_bf16<4>(smem + kSmH2, kMlpHidden, r, 32 * half, v);
    if (TRACE && trow)
#pragma unroll
      for (int k = 0; k < 32; ++k) trow[kTraceH2 + 32 * half + k] = v[k];
    handoff();
    // ---- layer 3, loss and dy (this thread: outputs 16 half .. 16 half + 15)
    if (tid == 0) {
#pragma unroll
      for (int ks = 0; ks < kMlpHidden / 16; ++ks)
        umma(tmem + kColL3, kmaj(sh2, kMlpHidden, ks), kmaj(sw3, kMlpHidden, ks),
             idesc_bf16(128, kMlpOut), ks > 0);
      umma_commit(mbar_a);
    }
    if (!sync_mma()) break;
    {
      uint32_t a[16];
      tmem_ld16_async(lane_addr + kColL3 + 16 * half, a);
      tmem_wait_ld();
      float dy[16], lsum = 0.f;
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const int o = 16 * half + k;
        const float y = __uint_as_float(a[k]) + sb[2 * kMlpHidden + o];
        const float d = valid && o < kMlpOutUsed ? y - t[k] : 0.f;
        lsum = fmaf(d, d, lsum);
        dy[k] = 2.0f * d * inv_n;
        if (TRACE && trow) {
          trow[kTraceY + o] = y;
          trow[kTraceDy + o] = dy[k];
        }
      }
      put_bf16<2>(smem + kSmDy, kMlpOut, r, 16 * half, dy);
      handoff();
      // ---- dh2 = (dy W3) (1 - h2^2): K = 32 over the outputs, into layer 3's
      // columns; behind it the gradient of W3, K = the tile's 128 rows
      if (tid == 0) {
#pragma unroll
        for (int ks = 0; ks < kMlpOut / 16; ++ks)
          umma(tmem + kColL3, kmaj(sdy, kMlpOut, ks), kmaj(sw3t, kMlpOut, ks),
               idesc_bf16(128, kMlpHidden), ks > 0);
        umma_commit(mbar_a);
#pragma unroll 1
        for (int ks = 0; ks < kRows / 16; ++ks)
          umma(tmem + kColG3, mnmaj(sh2, kMlpHidden, ks), mnmaj(sdy, kMlpOut, ks),
               idesc_t(128, kMlpOut), !first || ks > 0);
      }
      warp_col_sums<16>(dy, gbw, lane);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
      if (lane == 0) lossw[warp] += lsum;
    }
    if (!sync_mma()) break;
    {
      float hv[32];
      ld32(lane_addr + kColL3 + 32 * half, v);
      ld32(lane_addr + kColL2 + 32 * half, hv);
#pragma unroll
      for (int k = 0; k < 32; ++k) v[k] *= 1.0f - hv[k] * hv[k];
      put_bf16<4>(smem + kSmDh2, kMlpHidden, r, 32 * half, v);
      if (TRACE && trow)
#pragma unroll
        for (int k = 0; k < 32; ++k) trow[kTraceDh2 + 32 * half + k] = v[k];
    }
    handoff();
    // ---- dh1 = (dh2 W2) (1 - h1^2), into layer 2's columns (h2 is no longer
    // needed); behind it the gradient of W2
    if (tid == 0) {
#pragma unroll
      for (int ks = 0; ks < kMlpHidden / 16; ++ks)
        umma(tmem + kColL2, kmaj(sdh2, kMlpHidden, ks), kmaj(sw2t, kMlpHidden, ks),
             idesc_bf16(128, kMlpHidden), ks > 0);
      umma_commit(mbar_a);
#pragma unroll 1
      for (int ks = 0; ks < kRows / 16; ++ks)
        umma(tmem + kColG2, mnmaj(sh1, kMlpHidden, ks), mnmaj(sdh2, kMlpHidden, ks),
             idesc_t(128, kMlpHidden), !first || ks > 0);
    }
    warp_col_sums<32>(v, gbw + kMlpOut / 2, lane);
    if (!sync_mma()) break;
    {
      float hv[32];
      ld32(lane_addr + kColL2 + 32 * half, v);
      ld32(lane_addr + kColL1 + 32 * half, hv);
#pragma unroll
      for (int k = 0; k < 32; ++k) v[k] *= 1.0f - hv[k] * hv[k];
      put_bf16<4>(smem + kSmDh1, kMlpHidden, r, 32 * half, v);
      if (TRACE && trow)
#pragma unroll
        for (int k = 0; k < 32; ++k) trow[kTraceDh1 + 32 * half + k] = v[k];
    }
    handoff();
    // ---- the gradient of W1; with it all gradients, accumulated over the tiles
    if (tid == 0) {
#pragma unroll 1
      for (int ks = 0; ks < kRows / 16; ++ks)
#pragma unroll
        for (int q = 0; q < 3; ++q)  // features 128 q ..: boxes 2 q, 2 q + 1, rows 16 ks ..
          umma(tmem + kColG1 + 64 * q,
               sdesc_swizzled(sx + 2 * q * kBoxBytes + 2048 * ks, kBoxBytes, 1024, true),
               mnmaj(sdh1, kMlpHidden, ks), idesc_t(128, kMlpHidden), !first || ks > 0);
      umma_commit(mbar_a);
    }
    warp_col_sums<32>(v, gbw + kMlpOut / 2 + kMlpHidden / 2, lane);
    if (!sync_mma()) break;  // the next tile overwrites the operand tiles
  }

  if (ok) {
    // ---- block partials in the packed parameter order: thread (r, half)
    // holds lane r of each accumulator and half of its columns
    float *o = gpart + (long long)blockIdx.x * kMlpParams;
    float v[32];
#pragma unroll 1
    for (int q = 0; q < 3; ++q) {  // gW1[j][f], f = 128 q + r
      ld32(lane_addr + kColG1 + 64 * q + 32 * half, v);
      const int f = 128 * q + r;
      if (f < kMlpIn)
#pragma unroll
        for (int k = 0; k < 32; ++k) o[kOffW1 + (32 * half + k) * kMlpIn + f] = v[k];
    }
    ld32(lane_addr + kColG2 + 32 * half, v);  // gW2[j][i], i = r
    if (r < kMlpHidden)
#pragma unroll
      for (int k = 0; k < 32; ++k) o[kOffW2 + (32 * half + k) * kMlpHidden + r] = v[k];
    {
      uint32_t a[16];  // gW3[o][j], j = r
      tmem_ld16_async(lane_addr + kColG3 + 16 * half, a);
      tmem_wait_ld();
      if (r < kMlpHidden)
#pragma unroll
        for (int k = 0; k < 16; ++k)
          o[kOffW3 + (16 * half + k) * kMlpHidden + r] = __uint_as_float(a[k]);
    }
    __syncthreads();
    // bias gradients: the four row warps of each half, in order
    const float *g = reinterpret_cast<const float *>(smem + kSmGbw);
    for (int c = tid; c < 2 * kGbCols; c += kThreads) {
      const int h = c / kGbCols, k = c - h * kGbCols;
      const float s = ((g[(4 * h + 0) * kGbCols + k] + g[(4 * h + 1) * kGbCols + k]) +
                       g[(4 * h + 2) * kGbCols + k]) +
                      g[(4 * h + 3) * kGbCols + k];
      if (k < kMlpOut / 2)
        o[kOffB3 + 16 * h + k] = s;
      else if (k < kMlpOut / 2 + kMlpHidden / 2)
        o[kOffB2 + 32 * h + k - kMlpOut / 2] = s;
      else
        o[kOffB1 + 32 * h + k - kMlpOut / 2 - kMlpHidden / 2] = s;
    }
    if (tid == 0)
      lpart[blockIdx.x] = (((lossw[0] + lossw[1]) + (lossw[2] + lossw[3])) +
                           ((lossw[4] + lossw[5]) + (lossw[6] + lossw[7])));
  } else {
    // copies and MMAs still in flight finish before the memory goes away
    if (tid == 0) {
      atomicExch(status, 1);
      umma_commit(mbar_d);
      mbar_wait(mbar_d, 0);
    }
    mbar_wait(mbar_w, 0);
    if (requested) mbar_wait(mbar_x, xphase);
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                 "r"(kTmemCols)
                 : "memory");
}

}  // namespace

cudaError_t launch_mlp_train(const MlpDevice &p, const void *X, const float *T, long long M,
                             float *gpart, float *lpart, int *status, int nblocks,
                             cudaStream_t st, float *trace) {
  if (!T || M < 1) return cudaErrorInvalidValue;
  auto kern = trace ? mlp_train_tc_kernel<true> : mlp_train_tc_kernel<false>;
  cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTrainSmem);
  if (e != cudaSuccess) return e;
  const long long tiles = (M + kRows - 1) / kRows;
  const int nb = (int)(tiles < nblocks ? tiles : nblocks);
  CUtensorMap map;
  e = make_row_map(X, M, kBoxCols, CU_TENSOR_MAP_SWIZZLE_128B, &map);
  if (e != cudaSuccess) return e;
  return launch_chained(kern, nb, kThreads, kTrainSmem, st, p, map, T, M, gpart, lpart, status,
                        trace);
}

}  // namespace lbrr
