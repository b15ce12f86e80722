// Learned closure on the RR step (an extension; the paper has no learned
// component): moment field, standardised features and targets for training,
// 2x2x2 coarsening of a fine run, and the update of a coarse D3Q27 FP32 store
// in which the network's prediction of the order 3..6 off-equilibrium
// coefficients is added to the recursion's before the (1 - 1/tau)
// relaxation.
//
// Feature of a cell: the moments (rho - 1, u, Pi1) of the cell and its 26
// periodic neighbours, standardised per moment kind, neighbour index
// (dx+1) + 3(dy+1) + 9(dz+1), feature 10 * neighbour + moment, zero padded
// to 288. Target: the order 3..6 Hermite coefficients of (f - f_RR), f_RR the
// RR reconstruction from the cell's own moments, divided by out_scale, in the
// order xxy, xxz, xyy, xzz, yzz, yyz, xyz, xxyy, xxzz, yyzz, xyzz, xyyz, xxyz,
// xxyzz, xxyyz, xyyzz, xxyyzz, zero padded to 32.
#include "lbrr_launch.h"
#include "lbrr_mlp.h"
#include "lbrr_act.cuh"

namespace lbrr {

namespace {

constexpr int kAux = 128;

// --------------------------------------------------------------- moments --
__global__ void __launch_bounds__(kAux)
    moment_field_kernel(const float *__restrict__ f, const Grid g, const int parity,
                        float *__restrict__ mom) {
  const long long cell = (long long)blockIdx.x * kAux + threadIdx.x;
  if (cell >= g.n) return;
  int x, y, z;
  cell_coords(cell, g, x, y, z);
  float df[27];
  load_logical<27, 0>(f, g, parity, x, y, z, df);
  const Macro m = Lattice<27>::moments(df);
  const long long n = g.n;
  const float v[kMlpMoments] = {m.drho, m.ux, m.uy, m.uz, m.pxx, m.pxy, m.pxz, m.pyy, m.pyz, m.pzz};
#pragma unroll
  for (int k = 0; k < kMlpMoments; ++k) mom[k * n + cell] = v[k];
}

// -------------------------------------------------------------- features --
// Bound by its output: 576 B a cell against 40 B of moments. With a thread
// writing its cell's row 4 bytes at a time the lines of 32 rows were open at
// once and 64^3 took 315 us. So a block takes kFeatX cells of kFeatY rows of
// a plane, forms the standardised moments of these and their neighbours once,
// packed two to a word as the features hold them, and then kFeatChunks threads
// to a cell each gather 4 words of their own fixed place in the feature row:
// 16-byte stores, consecutive along the rows. 35 us.
constexpr int kFeatX = 32, kFeatY = 4;                // cells of a block
constexpr int kFeatChunks = kMlpIn / 8;               // 16-byte chunks of a feature row
constexpr int kFeatThreads = 8 * kFeatChunks;         // 8 cells at a time
constexpr int kFeatPairs = kMlpMoments / 2;           // words of a cell
constexpr int kFeatRow = (kFeatX + 2) * kFeatPairs;   // words of a staged row
static_assert(kFeatX % 8 == 0, "the cells taken at a time lie in one row");

__global__ void __launch_bounds__(kFeatThreads)
    features_kernel(MlpDevice p, const float *__restrict__ mom, const Grid g, const int tiles_x,
                    const int tiles_y, uint4 *__restrict__ X) {
  __shared__ uint32_t words[3 * (kFeatY + 2) * kFeatRow];
  const long long n = g.n;
  const unsigned b = blockIdx.x, bx = b % (unsigned)tiles_x, byz = b / (unsigned)tiles_x;
  const int x0 = (int)bx * kFeatX, y0 = (int)(byz % (unsigned)tiles_y) * kFeatY;
  const int z = (int)(byz / (unsigned)tiles_y);
  const int nx = min(kFeatX, g.nx - x0), ny = min(kFeatY, g.ny - y0);
  for (int q = threadIdx.x; q < 3 * (kFeatY + 2) * (kFeatX + 2); q += kFeatThreads) {
    const int row = q / (kFeatX + 2), px = q - row * (kFeatX + 2);
    const int pz = row / (kFeatY + 2), py = row - pz * (kFeatY + 2);
    if (px > nx + 1 || py > ny + 1) continue;
    const int x = x0 + px - 1, y = y0 + py - 1;
    const long long c = ((long long)wrap_add(z, pz - 1, g.nz) * g.ny +
                         (y < 0 ? g.ny - 1 : y == g.ny ? 0 : y)) * g.nx +
                        (x < 0 ? g.nx - 1 : x == g.nx ? 0 : x);
#pragma unroll
    for (int k = 0; k < kMlpMoments; k += 2) {
      const float v0 = (__ldg(mom + k * n + c) - p.in_mean[k]) * p.in_inv_std[k];
      const float v1 = (__ldg(mom + (k + 1) * n + c) - p.in_mean[k + 1]) * p.in_inv_std[k + 1];
      words[row * kFeatRow + px * kFeatPairs + k / 2] = pack_bf16(v0, v1);
    }
  }
  __syncthreads();
  const bool wide = reinterpret_cast<uintptr_t>(X) % 16 == 0;  // else 4-byte stores
  const int chunk = threadIdx.x % kFeatChunks, first = threadIdx.x / kFeatChunks;
  int place[4];  // of the chunk's words, from the staged row and position of the cell's (-1, -1, -1)
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int w = 4 * chunk + k, nb = w / kFeatPairs;
    place[k] = nb < 27 ? ((nb / 9) * (kFeatY + 2) + (nb / 3) % 3) * kFeatRow +
                             (nb % 3) * kFeatPairs + w - nb * kFeatPairs
                       : -1;  // zero padding
  }
  for (int q = first; q < kFeatX * kFeatY; q += kFeatThreads / kFeatChunks) {
    const int x = q % kFeatX, y = q / kFeatX;
    if (x >= nx || y >= ny) continue;
    const uint32_t *w = words + y * kFeatRow + x * kFeatPairs;
    uint4 v;
    v.x = place[0] < 0 ? 0u : w[place[0]];
    v.y = place[1] < 0 ? 0u : w[place[1]];
    v.z = place[2] < 0 ? 0u : w[place[2]];
    v.w = place[3] < 0 ? 0u : w[place[3]];
    uint4 *dst = X + (((long long)z * g.ny + y0 + y) * g.nx + x0 + x) * kFeatChunks + chunk;
    if (wide) {
      *dst = v;
    } else {
      uint32_t *d = reinterpret_cast<uint32_t *>(dst);
      d[0] = v.x, d[1] = v.y, d[2] = v.z, d[3] = v.w;
    }
  }
}

// --------------------------------------------------------------- targets --
// 1-D Hermite analysis of a line d(-1), d(0), d(+1): sums of H0 = 1,
// H1 = xi, H2 = xi^2 - 1/3 times d.
__device__ __forceinline__ void ana1(float dm, float dz, float dp, float &e0, float &e1,
                                     float &e2) {
  e0 = dm + dz + dp;
  e1 = dp - dm;
  e2 = fmaf(2.0f / 3.0f, dm + dp, -dz / 3.0f);
}

// Hermite coefficients A[a][b][c] = sum_i H_a(xi_x) H_b(xi_y) H_c(xi_z) d_i of
// a D3Q27 population vector (separable: x lines, then y, then z).
__device__ __forceinline__ void hermite_analysis(const float (&d)[27], float (&A)[3][3][3]) {
  float ax[3][9];  // [a][line (iy, iz)]
#pragma unroll
  for (int l = 0; l < 9; ++l) ana1(d[3 * l], d[3 * l + 1], d[3 * l + 2], ax[0][l], ax[1][l], ax[2][l]);
  float axy[3][3][3];  // [a][b][iz]
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int iz = 0; iz < 3; ++iz)
      ana1(ax[a][3 * iz], ax[a][3 * iz + 1], ax[a][3 * iz + 2], axy[a][0][iz], axy[a][1][iz],
           axy[a][2][iz]);
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b)
      ana1(axy[a][b][0], axy[a][b][1], axy[a][b][2], A[a][b][0], A[a][b][1], A[a][b][2]);
}

// The target rows of a warp's 32 cells first .. first + 31 (those below n), the
// order 3..6 coefficients of A divided by div * out_scale, zero padded. They go
// through shared memory, so that a store writes one row of 128 bytes: with each
// thread storing its own row, step_targets_kernel took 74 us at 64^3; 43.
__device__ __forceinline__ void write_targets(const MlpDevice &p, const float (&A)[3][3][3],
                                              float div, long long first, long long n,
                                              float *__restrict__ T) {
  __shared__ float rows[kAux / 32][32][kMlpOutUsed];  // odd row length: no bank conflicts
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
#pragma unroll
  for (int k = 0; k < kMlpOutUsed; ++k)
    rows[warp][lane][k] = A[hi_pow(k, 0)][hi_pow(k, 1)][hi_pow(k, 2)] / (div * p.out_scale[k]);
  __syncwarp();
  const int count = n - first < 32 ? (int)(n - first) : 32;
  float *dst = T + first * kMlpOut + lane;
#pragma unroll 8
  for (int k = 0; k < count; ++k) dst[k * kMlpOut] = lane < kMlpOutUsed ? rows[warp][k][lane] : 0.f;
}

__global__ void __launch_bounds__(kAux)
    targets_kernel(MlpDevice p, const float *__restrict__ f, const Grid g, const int parity,
                   float *__restrict__ T) {
  const long long first = (long long)blockIdx.x * kAux + (threadIdx.x & ~31u);  // of the warp
  if (first >= g.n) return;
  const long long cell = min(first + threadIdx.x % 32, g.n - 1);
  int x, y, z;
  cell_coords(cell, g, x, y, z);
  float df[27], rr[27];
  load_logical<27, 0>(f, g, parity, x, y, z, df);
  const Macro m = Lattice<27>::moments(df);
  Lattice<27>::synth<0>(m, 1.0f, rr);  // f_RR - w (tau -> infinity)
#pragma unroll
  for (int i = 0; i < 27; ++i) rr[i] = df[i] - rr[i];
  float A[3][3][3];
  hermite_analysis(rr, A);
  write_targets(p, A, 1.0f, first, g.n, T);
}

// Step-matching targets of coarse cell x: P_i(x) = post_i(x + xi_i) (logical
// populations; in the AA store, parity 0: slot i of x + xi_i, parity 1: slot
// opp(i) of x itself), R = the RR post-collision of pre's cell x; the order
// 3..6 coefficients of (P - R) / om1. Shifted values throughout: the weights
// cancel in the difference.
__global__ void __launch_bounds__(kAux)
    step_targets_kernel(MlpDevice p, const float *__restrict__ fpre, const int ppre,
                        const float *__restrict__ fpost, const int ppost, const Grid g,
                        const float om1, float *__restrict__ T) {
  const long long first = (long long)blockIdx.x * kAux + (threadIdx.x & ~31u);  // of the warp
  if (first >= g.n) return;
  const long long cell = min(first + threadIdx.x % 32, g.n - 1);
  int x, y, z;
  cell_coords(cell, g, x, y, z);
  float df[27], r[27];
  load_logical<27, 0>(fpre, g, ppre, x, y, z, df);
  const Macro m = Lattice<27>::moments(df);
  Lattice<27>::synth<0>(m, om1, r);
  const long long n = g.n;
#pragma unroll
  for (int i = 0; i < 27; ++i) {
    float pi;
    if (ppost == 0) {
      const long long dst = ((long long)wrap_add(z, vel(i, 2), g.nz) * g.ny +
                             wrap_add(y, vel(i, 1), g.ny)) * g.nx + wrap_add(x, vel(i, 0), g.nx);
      pi = __ldg(fpost + i * n + dst);
    } else {
      pi = __ldg(fpost + (26 - i) * n + cell);
    }
    r[i] = pi - r[i];
  }
  float A[3][3][3];
  hermite_analysis(r, A);
  write_targets(p, A, om1, first, g.n, T);
}

// -------------------------------------------------------------- coarsen --
// RESCALE: the off-equilibrium part of the average is scaled,
// f0(rho, u) + scale (fbar - f0(rho, u)) with rho, u the moments of fbar.
template <int SF, int SC, bool RESCALE = false>
__global__ void __launch_bounds__(kAux)
    coarsen_kernel(const typename Storage<SF>::T *__restrict__ ff, const Grid gf, const int parity,
                   typename Storage<SC>::T *__restrict__ fc, const Grid gc, const float scale) {
  const long long cell = (long long)blockIdx.x * kAux + threadIdx.x;
  if (cell >= gc.n) return;
  int x, y, z;
  cell_coords(cell, gc, x, y, z);
  float acc[27] = {};
#pragma unroll 1
  for (int s = 0; s < 8; ++s) {
    float df[27];
    load_logical<27, SF>(ff, gf, parity, 2 * x + (s & 1), 2 * y + ((s >> 1) & 1),
                         2 * z + (s >> 2), df);
#pragma unroll
    for (int i = 0; i < 27; ++i) acc[i] += df[i];
  }
#pragma unroll
  for (int i = 0; i < 27; ++i) acc[i] *= 0.125f;
  if (RESCALE) {
    const Macro m = Lattice<27>::moments(acc);
    float eq[27];
    Lattice<27>::synth<0>(m, 0.0f, eq);  // f0 - w
#pragma unroll
    for (int i = 0; i < 27; ++i) acc[i] = fmaf(scale, acc[i] - eq[i], eq[i]);
  }
#pragma unroll
  for (int i = 0; i < 27; ++i) Storage<SC>::template store<27>(fc + i * gc.n + cell, i, acc[i]);
}

// ---------------------------------------------------------- closure step --
// One thread per cell (blocks along x, AA parity as in lbrr_step.cu): RR
// coefficients plus (1 - 1/tau) times the network's correction, RR alone for
// a cell whose standardised prediction exceeds the bound or whose corrected
// populations are not all positive (counted).
constexpr int kDT = 128;

template <int PARITY>
__global__ void __launch_bounds__(kDT)
    rr_step_delta_kernel(MlpDevice p, float *__restrict__ f, const Grid g, const float om1,
                         const float *__restrict__ ystd, unsigned long long *fallbacks,
                         const float bound, const float dead_zone) {
  const int x = blockIdx.x * kDT + threadIdx.x;
  if (x >= g.nx) return;
  const int y = blockIdx.y, z = blockIdx.z;
  const long long cell = ((long long)z * g.ny + y) * g.nx + x;
  float yk[kMlpOutUsed];
#pragma unroll
  for (int k = 0; k < kMlpOutUsed; ++k) yk[k] = __ldg(ystd + k * g.n + cell);
  closure_update_cell<PARITY>(p, f, g, om1, x, y, z, yk, fallbacks, bound, dead_zone);
}

}  // namespace

cudaError_t launch_moment_field(int storage, const void *f, const Grid &g, int parity, float *mom,
                                cudaStream_t st) {
  if (storage != 0) return cudaErrorInvalidValue;
  moment_field_kernel<<<(unsigned)((g.n + kAux - 1) / kAux), kAux, 0, st>>>(
      static_cast<const float *>(f), g, parity, mom);
  return cudaGetLastError();
}

cudaError_t launch_features(const MlpDevice &p, const float *mom, const Grid &g, void *X,
                            cudaStream_t st) {
  const int tx = (g.nx + kFeatX - 1) / kFeatX, ty = (g.ny + kFeatY - 1) / kFeatY;
  features_kernel<<<(unsigned)((long long)tx * ty * g.nz), kFeatThreads, 0, st>>>(
      p, mom, g, tx, ty, static_cast<uint4 *>(X));
  return cudaGetLastError();
}

cudaError_t launch_targets(const MlpDevice &p, int storage, const void *f, const Grid &g,
                           int parity, float *T, cudaStream_t st) {
  if (storage != 0) return cudaErrorInvalidValue;
  targets_kernel<<<(unsigned)((g.n + kAux - 1) / kAux), kAux, 0, st>>>(
      p, static_cast<const float *>(f), g, parity, T);
  return cudaGetLastError();
}

cudaError_t launch_coarsen(int storage_f, const void *ff, const Grid &gf, int parity_f,
                           int storage_c, void *fc, const Grid &gc, cudaStream_t st,
                           float neq_scale) {
  const unsigned nb = (unsigned)((gc.n + kAux - 1) / kAux);
  if (storage_f != 0 || storage_c != 0) return cudaErrorInvalidValue;
  if (neq_scale == 1.0f)
    coarsen_kernel<0, 0><<<nb, kAux, 0, st>>>(static_cast<const float *>(ff), gf, parity_f,
                                              static_cast<float *>(fc), gc, 1.0f);
  else
    coarsen_kernel<0, 0, true><<<nb, kAux, 0, st>>>(static_cast<const float *>(ff), gf, parity_f,
                                                    static_cast<float *>(fc), gc, neq_scale);
  return cudaGetLastError();
}

cudaError_t launch_step_targets(const MlpDevice &p, const float *fpre, int ppre,
                                const float *fpost, int ppost, const Grid &g, float om1, float *T,
                                cudaStream_t st) {
  step_targets_kernel<<<(unsigned)((g.n + kAux - 1) / kAux), kAux, 0, st>>>(p, fpre, ppre, fpost,
                                                                           ppost, g, om1, T);
  return cudaGetLastError();
}

cudaError_t launch_step_delta(const MlpDevice &p, float *f, const Grid &g, float om1, int parity,
                              const float *ystd, unsigned long long *fallbacks, float bound,
                              float dead_zone, cudaStream_t st) {
  const dim3 grid((g.nx + kDT - 1) / kDT, g.ny, g.nz);
  if (parity == 0)
    rr_step_delta_kernel<0><<<grid, kDT, 0, st>>>(p, f, g, om1, ystd, fallbacks, bound,
                                                 dead_zone);
  else
    rr_step_delta_kernel<1><<<grid, kDT, 0, st>>>(p, f, g, om1, ystd, fallbacks, bound,
                                                 dead_zone);
  return cudaGetLastError();
}

}  // namespace lbrr
