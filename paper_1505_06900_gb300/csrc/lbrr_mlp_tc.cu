// Forward pass of the closure network on the 5th-generation tensor cores
// (tcgen05, sm_100-family): y = W3 tanh(W2 tanh(W1 x + b1) + b2) + b3 for
// tiles of 128 rows, BF16 operands in shared memory, FP32 accumulators in
// tensor memory (TMEM).
//
// One block per SM (persistent), in two groups of 256 threads that take
// alternate tiles. The BF16 weights are staged once into shared memory in the
// canonical K-major layout without swizzle: 8 x 8 "core matrices" of 128
// contiguous bytes (8 rows of 16 bytes), adjacent core matrices along K 128
// bytes apart (leading byte offset) and adjacent 8-row groups K/8 * 128 bytes
// apart (stride byte offset), as they lie in memory. A tile's 128 input rows
// come by TMA in boxes of 64 columns in the layout with 128-byte swizzle, the
// last 32 with 64-byte swizzle; one thread of the group issues the MMAs of a
// layer (M = 128, N = 64, 64, 32) and commits them to the group's mbarrier; the
// threads, two to a row (TMEM lane), then read the accumulator (tcgen05.ld 32x32b), add the bias, apply
// tanh and write the BF16 row back into TMEM (tcgen05.st), the A operand of the
// next layer.
//
// Reading X (576 B a row) bounds it. One tile after another, loads, three
// products and epilogues in turn, 262144 rows took 101 us; now the rows of a
// group's next tile are requested as soon as layer 1 has read the present one's,
// and the two groups' chains overlap: 39 us (62 with the rows copied by the
// threads, 16 bytes each, whose issue alone held a tile up for 4400 to 9000
// cycles). Outputs go through shared memory, a row of 128 bytes to a store.
//
// Every mbarrier wait is bounded: on expiry the group records a timeout in
// *status and waits (bounded) for its MMAs to drain before the block frees its
// TMEM and returns.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <cstdint>

#include "lbrr_launch.h"
#include "lbrr_mlp.h"
#include "lbrr_act.cuh"
#include "lbrr_tc.cuh"

namespace lbrr {

namespace {

using namespace tc;

constexpr int kTcRows = 128;
constexpr int kGroupThreads = 256;  // two threads per row; warps w and w + 4 share TMEM lanes
constexpr int kTcGroups = 2;
constexpr int kTcThreads = kTcGroups * kGroupThreads;
// TMEM columns of a group: layer 1 then 3, layer 2, the BF16 rows between them
constexpr uint32_t kColGroup = 192, kCol1 = 0, kCol2 = 64, kColH = 128;
constexpr uint32_t kTmemCols = 512;

// shared-memory plan (bytes, all 1024-aligned up to the output rows)
constexpr uint32_t kA1Bytes = kTcRows * kMlpIn * 2;           // 73728
constexpr int kYRow = kMlpOut + 1;                            // odd: no bank conflicts
constexpr uint32_t kYBytes = kTcRows * kYRow * 4;             // 16896
constexpr uint32_t kOffSW1 = 0;
constexpr uint32_t kOffSW2 = kOffSW1 + kMlpW1Bytes;
constexpr uint32_t kOffSW3 = kOffSW2 + kMlpW2Bytes;
constexpr uint32_t kOffSA1 = kOffSW3 + kMlpW3Bytes;
constexpr uint32_t kOffY = kOffSA1 + kTcGroups * kA1Bytes;
constexpr uint32_t kOffMisc = kOffY + kTcGroups * kYBytes;  // mbarriers, TMEM address, biases
constexpr uint32_t kTcSmem = kOffMisc + 1024;
// the boxes of a tile in A1
constexpr int kBoxCols = 64, kBoxes = kMlpIn / kBoxCols, kLastCols = kMlpIn - kBoxes * kBoxCols;
constexpr uint32_t kBoxBytes = kTcRows * kBoxCols * 2;
static_assert(kLastCols == 32, "64-byte rows");
static_assert(kOffSA1 % 1024 == 0 && kA1Bytes % 1024 == 0, "swizzle atoms");

__device__ __forceinline__ void group_sync(int g) {
  asm volatile("bar.sync %0, %1;\n" ::"r"(1 + g), "n"(kGroupThreads) : "memory");
}
// the same, returning whether any thread of the group passed pred = true
__device__ __forceinline__ bool group_any(int g, bool pred) {
  uint32_t r;
  asm volatile(
      "{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbar.red.or.pred q, %2, %3, p;\n"
      "selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((uint32_t)pred), "r"(1 + g), "n"(kGroupThreads)
      : "memory");
  return r != 0;
}

__device__ __forceinline__ uint32_t pack2(float lo, float hi) { return pack_bf16(lo, hi); }

// Layer epilogue: tanh(acc + bias) of columns 32 half .. 32 half + 31, as BF16
// into the 16 TMEM columns at dst; with TRACE also the FP32 values into
// hrow[64].
template <bool TRACE = false>
__device__ __forceinline__ void hidden_epilogue(uint32_t taddr, const float *bias, uint32_t dst,
                                                int half, float *hrow = nullptr) {
  uint32_t q[16];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int c0 = 32 * half + 16 * i;
    float v[16];
    tmem_ld16(taddr + c0, v);
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = tanh_approx(v[k] + bias[c0 + k]);
    if (TRACE && hrow)
#pragma unroll
      for (int k = 0; k < 16; k += 4)
        *reinterpret_cast<float4 *>(hrow + c0 + k) =
            make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
#pragma unroll
    for (int k = 0; k < 16; k += 2) q[8 * i + k / 2] = pack2(v[k], v[k + 1]);
  }
  tmem_st16(dst, q);
  tmem_wait_st();
}

// Standardised features of row r from the moment field in global memory.
__device__ __forceinline__ void features_gather(const MlpDevice &p, const float *mom,
                                                const Grid &g, long long cell,
                                                unsigned char *a1, int r, int half) {
  int x, y, z;
  cell_coords(cell, g, x, y, z);
  const long long n = g.n;
#pragma unroll 1
  for (int nb = half ? 14 : 0; nb < (half ? 27 : 14); ++nb) {
    const int dx = nb % 3 - 1, dy = (nb / 3) % 3 - 1, dz = nb / 9 - 1;
    const long long c = ((long long)wrap_add(z, dz, g.nz) * g.ny + wrap_add(y, dy, g.ny)) * g.nx +
                        wrap_add(x, dx, g.nx);
#pragma unroll
    for (int k = 0; k < kMlpMoments; k += 2) {
      const float v0 = (__ldg(mom + k * n + c) - p.in_mean[k]) * p.in_inv_std[k];
      const float v1 = (__ldg(mom + (k + 1) * n + c) - p.in_mean[k + 1]) * p.in_inv_std[k + 1];
      *reinterpret_cast<uint32_t *>(a1 + cm_offset(r, kMlpMoments * nb + k, kMlpIn)) =
          pack2(v0, v1);
    }
  }
  if (half)
    for (int f = kMlpInUsed; f < kMlpIn; f += 2)
      *reinterpret_cast<uint32_t *>(a1 + cm_offset(r, f, kMlpIn)) = 0u;
}

// FROM_MOM: rows are the cells of a grid and their features are built from
// the moment field mom [10][N]; outputs y[k][cell] for the 17 used outputs.
// (Small grids only: lbrr_mlp_conv.cu takes the others.)
// Otherwise rows are X [M][288] (BF16) and outputs Y [M][32].
// TRACE (rows X only): also H[row][0..63] and H[row][64..127], the FP32
// activations of layers 1 and 2 before their BF16 rounding.
template <bool FROM_MOM, bool TRACE = false>
__global__ void __launch_bounds__(kTcThreads, 1)
    mlp_tc_kernel(MlpDevice p, const __grid_constant__ CUtensorMap x_map,
                  const __grid_constant__ CUtensorMap x_last, const float *__restrict__ mom,
                  const Grid g, long long M, float *__restrict__ Y, int *status, float *__restrict__ H) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const int tid = threadIdx.x, warp = tid >> 5;
  const int gr = tid / kGroupThreads, gt = tid % kGroupThreads;
  const int r = gt & (kTcRows - 1), half = gt >> 7;  // row, and which half of its work
  // of each group: MMAs done, rows landed; then the weights landed
  uint64_t *mbar = reinterpret_cast<uint64_t *>(smem + kOffMisc);
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + kOffMisc + 16 * kTcGroups + 8);
  float *sb = reinterpret_cast<float *>(smem + kOffMisc + 64);  // b1, b2, b3 (160)
  unsigned char *a1 = smem + kOffSA1 + gr * kA1Bytes;
  float *ys = reinterpret_cast<float *>(smem + kOffY + gr * kYBytes);
  const uint32_t mbar_a = smem_u32(mbar + gr), mbar_x = smem_u32(mbar + kTcGroups + gr);
  const long long ntiles = (M + kTcRows - 1) / kTcRows;
  const long long stride = (long long)kTcGroups * gridDim.x;

  long long tile = blockIdx.x + (long long)gr * gridDim.x;
  bool requested = false;
  // rows of X into the A1 tile (zeros past M)
  auto request = [&](long long t) {
    requested = true;
    if (gt != 0) return;
    mbar_expect_tx(mbar_x, kA1Bytes);
    const uint32_t dst = smem_u32(a1);
#pragma unroll
    for (int k = 0; k < kBoxes; ++k)
      tma_load_2d(dst + k * kBoxBytes, &x_map, k * kBoxCols, (int)(t * kTcRows), mbar_x);
    tma_load_2d(dst + kBoxes * kBoxBytes, &x_last, kBoxes * kBoxCols, (int)(t * kTcRows), mbar_x);
  };
  const uint32_t mbar_w = smem_u32(mbar + 2 * kTcGroups);
  if (tid == 0) {
    for (int k = 0; k <= 2 * kTcGroups; ++k) mbar_init(smem_u32(mbar + k), 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    fence_async_smem();
    mbar_expect_tx(mbar_w, kOffSA1);
    bulk_load(smem_u32(smem), p.w1, kOffSA1, mbar_w);
  }
  __syncthreads();
  if (!FROM_MOM && tile < ntiles) request(tile);
  // ---- biases
  for (int c = tid; c < 2 * kMlpHidden + kMlpOut; c += kTcThreads)
    sb[c] = c < kMlpHidden ? p.b1[c] : (c < 2 * kMlpHidden ? p.b2[c - kMlpHidden]
                                                           : p.b3[c - 2 * kMlpHidden]);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  fence_async_smem();
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot + kColGroup * gr;
  // TMEM lanes of this warp: 32 (warp % 4) ..
  const uint32_t lane_addr = tmem + ((uint32_t)(32 * (warp & 3)) << 16);

  const uint32_t sw1 = smem_u32(smem + kOffSW1), sw2 = smem_u32(smem + kOffSW2);
  const uint32_t sw3 = smem_u32(smem + kOffSW3), sa1 = smem_u32(a1);
  uint32_t phase = 0, xphase = 0;
  bool ok = true;
  // the group's threads wait for the MMAs committed so far (the same decision in each)
  auto sync_mma = [&]() {
    ok = !group_any(gr, !mbar_wait(mbar_a, phase));
    phase ^= 1;
    fence_after();
    return ok;
  };
  auto handoff = [&]() {  // the group's writes before the next MMAs
    fence_before();
    group_sync(gr);
    fence_after();
  };

  ok = !group_any(gr, !mbar_wait(mbar_w, 0));
  for (; tile < ntiles && ok; tile += stride) {
    const long long row = tile * kTcRows + r;
    const bool valid = row < M;
    // ---- input rows
    if (FROM_MOM) {
      if (valid) {
        features_gather(p, mom, g, row, a1, r, half);
      } else {
        for (int kb = half * (kMlpIn / 16); kb < (half + 1) * (kMlpIn / 16); ++kb)
          *reinterpret_cast<uint4 *>(a1 + cm_offset(r, 8 * kb, kMlpIn)) =
              make_uint4(0u, 0u, 0u, 0u);
      }
      fence_async_smem();
    } else {
      ok = !group_any(gr, !mbar_wait(mbar_x, xphase));
      if (!ok) break;
      xphase ^= 1;
      requested = false;
    }
    handoff();
    // ---- layer 1: D[128 x 64] = A1[128 x 288] W1^T
    if (gt == 0) {
#pragma unroll 1
      for (int ks = 0; ks < kMlpIn / 16; ++ks)
        umma(tmem + kCol1,
             FROM_MOM ? sdesc(sa1 + 256 * ks, 128, (kMlpIn / 8) * 128)
                      : sdesc_swizzled(sa1 + (ks / 4) * kBoxBytes + 32 * (ks % 4), 16,
                                       ks / 4 < kBoxes ? 1024 : 512, ks / 4 < kBoxes),
             sdesc(sw1 + 256 * ks, 128, (kMlpIn / 8) * 128), idesc_bf16(128, 64), ks > 0);
      umma_commit(mbar_a);
    }
    if (!sync_mma()) break;
    if (!FROM_MOM && tile + stride < ntiles) request(tile + stride);  // A1 has been read
    hidden_epilogue<TRACE>(lane_addr + kCol1, sb, lane_addr + kColH + 16 * half, half,
                           TRACE && valid ? H + row * (2 * kMlpHidden) : nullptr);
    handoff();
    // ---- layer 2
    if (gt == 0) {
#pragma unroll
      for (int ks = 0; ks < kMlpHidden / 16; ++ks)
        umma_ts(tmem + kCol2, tmem + kColH + 8 * ks,
                sdesc(sw2 + 256 * ks, 128, (kMlpHidden / 8) * 128), idesc_bf16(128, 64), ks > 0);
      umma_commit(mbar_a);
    }
    if (!sync_mma()) break;
    hidden_epilogue<TRACE>(lane_addr + kCol2, sb + kMlpHidden, lane_addr + kColH + 16 * half, half,
                           TRACE && valid ? H + row * (2 * kMlpHidden) + kMlpHidden : nullptr);
    handoff();
    // ---- layer 3: each half reads 16 of the 32 columns
    if (gt == 0) {
#pragma unroll
      for (int ks = 0; ks < kMlpHidden / 16; ++ks)
        umma_ts(tmem + kCol1, tmem + kColH + 8 * ks,
                sdesc(sw3 + 256 * ks, 128, (kMlpHidden / 8) * 128), idesc_bf16(128, 32), ks > 0);
      umma_commit(mbar_a);
    }
    if (!sync_mma()) break;
    float y[16];
    tmem_ld16(lane_addr + kCol1 + 16 * half, y);
    const float *b3 = sb + 2 * kMlpHidden + 16 * half;
    if (FROM_MOM) {
      if (valid) {
#pragma unroll
        for (int k = 0; k < 16; ++k)
          if (16 * half + k < kMlpOutUsed) Y[(16 * half + k) * M + row] = y[k] + b3[k];
      }
    } else {
#pragma unroll
      for (int k = 0; k < 16; ++k) ys[r * kYRow + 16 * half + k] = y[k] + b3[k];
      group_sync(gr);
      const long long row0 = tile * kTcRows;
      const int lane = tid & 31;
#pragma unroll
      for (int k = 0; k < kTcRows; k += kGroupThreads / 32) {
        const int q = k + gt / 32;
        if (row0 + q < M) Y[(row0 + q) * kMlpOut + lane] = ys[q * kYRow + lane];
      }
    }
    // the accumulators and, over the next tile's barriers, ys have been read
    fence_before();
  }

  if (!ok) {
    if (gt == 0) atomicExch(status, 1);
    // let copies and MMAs still in flight finish before the memory goes away
    // (at the last phase waited for)
    mbar_wait(mbar_w, 0);
    if (requested) mbar_wait(mbar_x, xphase);
    mbar_wait(mbar_a, phase ^ 1);
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

cudaError_t make_row_map(const void *X, long long M, int cols, CUtensorMapSwizzle swizzle,
                         CUtensorMap *map) {
  PFN_cuTensorMapEncodeTiled_v12000 encode = tensor_map_encoder();
  if (!encode) return cudaErrorNotSupported;
  const cuuint64_t dims[2] = {kMlpIn, (cuuint64_t)M}, strides[1] = {kMlpIn * 2};
  const cuuint32_t box[2] = {(cuuint32_t)cols, kTcRows}, estr[2] = {1, 1};
  const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(X), dims,
                            strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t launch_mlp_tc(const MlpDevice &p, const void *X, const float *mom, const Grid *g,
                          long long M, float *Y, int *status, int nblocks, cudaStream_t st,
                          float *H) {
  const bool from_mom = mom != nullptr;
  if (from_mom && H) return cudaErrorInvalidValue;
  auto kern = from_mom ? mlp_tc_kernel<true> : (H ? mlp_tc_kernel<false, true>
                                                  : mlp_tc_kernel<false>);
  cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTcSmem);
  if (e != cudaSuccess) return e;
  CUtensorMap map{}, last{};
  if (!from_mom) {
    e = make_row_map(X, M, kBoxCols, CU_TENSOR_MAP_SWIZZLE_128B, &map);
    if (e == cudaSuccess) e = make_row_map(X, M, kLastCols, CU_TENSOR_MAP_SWIZZLE_64B, &last);
    if (e != cudaSuccess) return e;
  }
  const long long tiles = (M + kTcRows - 1) / kTcRows;
  const int nb = (int)(tiles < nblocks ? tiles : nblocks);
  const Grid gg = g ? *g : Grid{1, 1, 1, M};
  kern<<<nb, kTcThreads, kTcSmem, st>>>(p, map, last, mom, gg, M, Y, status, H);
  return cudaGetLastError();
}

}  // namespace lbrr
