// Runs of updates of a periodic 3-D FP32 grid carried out on its moments.
//
// The regularized collision (RR and its order-2 form) replaces the
// populations of a cell by a function of ten numbers: rho - 1, rho u and the
// second moments, from which Pi^(1) follows (Sec. 3.5). So between the first and
// the last of a run of updates the state need not be kept as Q populations: an
// update reads the ten moments of every cell, forms the post-collision
// populations, streams them inside the chip and reduces them to the ten moments
// of the next state, 80 bytes a cell instead of 2 Q 4 (216 for D3Q27). The run
// starts with the moments of the AA store and ends with its last collision
// streamed into the store, in the layout the same number of single updates would
// leave. Every value is computed by the operations of the single updates in
// their order (the moments' sums over x, y, then z are split by z component), so
// the result is theirs bit for bit, underflow and the signs of zeros included,
// while the velocities are finite numbers.
#include "lbrr_launch.h"
#include "lbrr_quot.cuh"

namespace lbrr {

namespace {

constexpr int kFields = 10;  // rho - 1, rho u (3), second moments (xx, xy, xz, yy, yz, zz)
constexpr int kTX = 32, kEX = kTX + 2;  // cells of a tile row, with its neighbours

// Tile of a block, one block per SM: as many threads as the registers allow
// without spills (80 and 72 a thread: 24 and 28 warps), since the ring of
// recomputed cells around the tile shrinks with its size. Measured at 256^3
// (D3Q27 / D3Q19, GLUPS over 20 updates): 16 rows 47.1 / 55.3, 20 rows 49.0 /
// 58.6, 24 rows 44.7 (72 registers) / 61.4, two blocks of 9 rows 46.8 / 57.3 (all
// with the populations of D3Q27 at twice their value or more inside the chip,
// which saved factors of 1/2 but rounded what underflows differently; 47.7 / 60.8
// as it is).
template <int Q>
struct Tile {
  static constexpr int TY = Q == 27 ? 20 : 24, EY = TY + 2, E = kEX * EY;
  static constexpr int kCells = kTX * TY;
  // threads: one per cell of the tile, then one per cell of the ring around it
  static constexpr int kThreads = (E + 31) / 32 * 32;
};

// Directions by column (cx, cy): column c = (cx + 1) + 3 (cy + 1). The
// populations of a column with z component -1, 0 and +1 come from the same
// cell, and are kept together: the outer two as one float2 where the lattice
// has them. Column 4, (0, 0), never leaves its cell's thread.
template <int Q>
__host__ __device__ constexpr bool has_outer(int c) {  // z components -1 and +1
  return Q == 27 || c % 2 == 1 || c == 4;
}
template <int Q>
__host__ __device__ constexpr int group_size(int cz) {
  return Q == 27 || cz == 0 ? 9 : 5;
}
template <int Q>
__host__ __device__ constexpr int in_group(int c, int cz) {  // place within the z component
  return Q == 27 || cz == 0 ? c : (c == 1 ? 0 : (c == 3 ? 1 : (c == 4 ? 2 : (c == 5 ? 3 : 4))));
}
template <int Q>
__host__ __device__ constexpr int dir_of(int c, int cz) {
  return in_group<Q>(c, cz) + (cz < 0 ? 0 : (cz == 0 ? group_size<Q>(-1)
                                                     : group_size<Q>(-1) + group_size<Q>(0)));
}
template <int Q>
__host__ __device__ constexpr int outer_index(int c) {
  return Q == 27 ? (c < 4 ? c : c - 1) : c / 2;
}
template <int Q>
constexpr int outers() {
  return Q == 27 ? 8 : 4;
}
template <int Q>
constexpr int plane_shared() {  // floats of one plane in shared memory
  return (2 * outers<Q>() + 8) * Tile<Q>::E;
}

// The sums of one z component: x lines, then y (sum, first and second moments
// of total order <= 2), as moments_d3q27 and moments_d3q19 form them.
struct Part {
  float s, x, y, xx, yy, xy;
};
__device__ __forceinline__ Part part(const float (&f)[9]) {
  float x0[3], x1[3], x2[3], t0, t1, t2;
#pragma unroll
  for (int l = 0; l < 3; ++l)
    mom3<false>(f[3 * l], f[3 * l + 1], f[3 * l + 2], x0[l], x1[l], x2[l]);
  Part p;
  mom3<false>(x0[0], x0[1], x0[2], p.s, p.y, p.yy);
  mom3<false>(x1[0], x1[1], x1[2], p.x, p.xy, t0);
  mom3<false>(x2[0], x2[1], x2[2], p.xx, t1, t2);
  return p;
}
// the cross (0,-1), (-1,0), (0,0), (1,0), (0,1) of a D3Q19 plane z = +-1
__device__ __forceinline__ Part part(const float (&f)[5]) {
  Part p;
  p.xx = f[1] + f[3];
  p.yy = f[0] + f[4];
  p.s = (p.xx + p.yy) + f[2];
  p.x = f[3] - f[1];
  p.y = f[4] - f[0];
  p.xy = 0.0f;
  return p;
}
// What a cell carries from update to update: rho - 1, rho u and its raw second
// moments.
struct Mom3 {
  float drho, jx, jy, jz, xx, xy, xz, yy, yz, zz;
};

// a / b correctly rounded, from nr = minus the correctly rounded 1 / b: one
// correction of the quotient by its exact remainder (P. Markstein, IBM J. Res.
// Dev. 34, 1990; taken so that a zero keeps its sign). One reciprocal serves the
// three components of a velocity.
__device__ __forceinline__ float quot(float a, float b, float nr) {
  const float q = __fmul_rn(-a, nr);
  return __fmaf_rn(__fmaf_rn(b, q, -a), nr, q);
}
// Macroscopic values as macro_from_moments forms them. A single update rounds a
// product j_a u_b before it takes it from the second moment where its synthesis
// uses the product too (order-2 form: all; D3Q19: the diagonal ones); elsewhere
// the difference is one fused operation.
template <int Q, int MODEL>
__device__ __forceinline__ Macro macro_of(const Mom3 &v) {
  Macro m;
  m.drho = v.drho;
  m.rho = 1.0f + v.drho;
  m.jx = v.jx;
  m.jy = v.jy;
  m.jz = v.jz;
  const float nr = minus_reciprocal(m.rho);
  m.ux = quot(m.jx, m.rho, nr);
  m.uy = quot(m.jy, m.rho, nr);
  m.uz = quot(m.jz, m.rho, nr);
  if (!(fminf(fminf(fabsf(m.ux), fabsf(m.uy)), fabsf(m.uz)) >= kLeastQuotient)) {
    if (needs_division(m.jx, m.ux) || needs_division(m.jy, m.uy) || needs_division(m.jz, m.uz)) {
      m.ux = __fdiv_rn(m.jx, m.rho);
      m.uy = __fdiv_rn(m.jy, m.rho);
      m.uz = __fdiv_rn(m.jz, m.rho);
    }
  }
  auto less = [](bool round, float p, float j, float u) {
    return round ? __fsub_rn(p, __fmul_rn(j, u)) : __fmaf_rn(-j, u, p);
  };
  constexpr bool off = Q == 27 && MODEL == 1, diag = off || Q == 19;
  m.pxx = less(diag, __fmaf_rn(-kCs2, m.drho, v.xx), m.jx, m.ux);
  m.pyy = less(diag, __fmaf_rn(-kCs2, m.drho, v.yy), m.jy, m.uy);
  m.pzz = less(diag, __fmaf_rn(-kCs2, m.drho, v.zz), m.jz, m.uz);
  m.pxy = less(off, v.xy, m.jx, m.uy);
  m.pxz = less(off, v.xz, m.jx, m.uz);
  m.pyz = less(off, v.yz, m.jy, m.uz);
  return m;
}

// Moments from the sums of z component -1 (m), 0 (z) and +1 (p).
template <int Q>
__device__ __forceinline__ Mom3 combine(const Part &m, const Part &z, const Part &p) {
  auto sum = [](float a, float b, float c) { return (a + c) + b; };
  return {sum(m.s, z.s, p.s), sum(m.x, z.x, p.x), sum(m.y, z.y, p.y), p.s - m.s,
          sum(m.xx, z.xx, p.xx), Q == 27 ? sum(m.xy, z.xy, p.xy) : z.xy, p.x - m.x,
          sum(m.yy, z.yy, p.yy), p.y - m.y, m.s + p.s};
}
template <int Q>
__device__ __forceinline__ Mom3 moments_of(const float (&f)[Q]) {
  float gm[group_size<Q>(-1)], gz[group_size<Q>(0)], gp[group_size<Q>(1)];
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    constexpr int o = group_size<Q>(-1), w = o + group_size<Q>(0);
    (i < o ? gm[i] : (i < w ? gz[i - o] : gp[i - w])) = f[i];
  }
  return combine<Q>(part(gm), part(gz), part(gp));
}

// Layout of the moments: rows in blocks of 32 cells; of a block first the
// fields 0 .. 3 of its cells as float4, then 4 .. 7, then 8 and 9 as float2.
// A cell is moved in three accesses at one address and two constant offsets,
// a row's 32 cells are 1280 bytes in one piece.
constexpr int kBlockF = 32 * kFields;
__host__ __device__ __forceinline__ int blocks_x(const Grid &g) { return (g.nx + 31) / 32; }
__host__ __device__ __forceinline__ long long plane_floats(const Grid &g) {
  return (long long)blocks_x(g) * g.ny * kBlockF;
}
__device__ __forceinline__ uint32_t cell_float(const Grid &g, int x, int y) {
  return (uint32_t)(y * blocks_x(g) + (x >> 5)) * kBlockF + 4 * (x & 31);
}
// the two float2 fields of a cell, from its float4 address and x
__device__ __forceinline__ int tail_float(int x) { return 256 - 2 * (x & 31); }
__device__ __forceinline__ Mom3 load_fields(const float *p, int tail) {
  const float4 u = __ldg(reinterpret_cast<const float4 *>(p));
  const float4 w = __ldg(reinterpret_cast<const float4 *>(p + 128));
  const float2 r = __ldg(reinterpret_cast<const float2 *>(p + tail));
  return {u.x, u.y, u.z, u.w, w.x, w.y, w.z, w.w, r.x, r.y};
}
__device__ __forceinline__ void store_fields(float *p, int tail, const Mom3 &m) {
  *reinterpret_cast<float4 *>(p) = make_float4(m.drho, m.jx, m.jy, m.jz);
  *reinterpret_cast<float4 *>(p + 128) = make_float4(m.xx, m.xy, m.xz, m.yy);
  *reinterpret_cast<float2 *>(p + tail) = make_float2(m.yz, m.zz);
}

// One update of the moments a -> b. A block walks the planes of a z segment
// of a tile: per plane it forms the post-collision populations of plane p + 1
// of the tile and its ring of neighbours into shared memory, and gathers those
// of plane p (one barrier a plane, two planes in shared memory); the sums of
// the three z components of a cell meet in registers. 512^3, GB300: 2.59 ms an
// update for D3Q27 over a run of 20 (51.7 GLUPS, single updates 30.7). It moves
// 80 bytes a cell through HBM at 4.0 TB/s; the bound is the instructions
// issued (547 a cell, 74% of the issue slots of the active SMs, three ready
// warps waiting for every one that issues). What mattered on the way:
// single 4-byte accesses to the moments (47.4 GLUPS where 53.4 were reached over
// 20 updates), 4-byte shared-memory accesses only and columns (0, 0) exchanged
// too (41.8), and any spill, since shared memory leaves the L1 cache little.
template <int Q, int MODEL>
__global__ void __launch_bounds__(Tile<Q>::kThreads, 1)
    rr_moment_step_kernel(const float *__restrict__ a, float *__restrict__ b, const Grid g,
                          const float om1, const int tiles_x, const int tiles_y, const int seg) {
  constexpr int kTY = Tile<Q>::TY, kEY = Tile<Q>::EY, kE = Tile<Q>::E, kTile = Tile<Q>::kCells;
  extern __shared__ __align__(128) float sm[];
  const int t = threadIdx.x;
  const int tile = blockIdx.x % (tiles_x * tiles_y), zi = blockIdx.x / (tiles_x * tiles_y);
  const int x0 = tile % tiles_x * kTX, y0 = tile / tiles_x * kTY;
  const int z0 = zi * seg, z1 = min(z0 + seg, g.nz);
  const long long plane = plane_floats(g);

  // cell (ex, ey) of the extended tile
  int ex = t % kTX + 1, ey = t / kTX + 1;
  if (t >= kTile) {  // rows 0 and kEY - 1 of the tile's columns, then the two outer columns
    const int r = t - kTile, c = r - 2 * kTX;
    ex = c < 0 ? r % kTX + 1 : (c & 1) * (kEX - 1);
    ey = c < 0 ? r / kTX * (kEY - 1) : c >> 1;
  }
  const bool active = t < kE, inner = t < kTile;
  int x = x0 + ex - 1, y = y0 + ey - 1;
  const bool in = inner && x < g.nx && y < g.ny;
  x = x < 0 ? x + g.nx : (x < g.nx ? x : x % g.nx);
  y = y < 0 ? y + g.ny : (y < g.ny ? y : y % g.ny);
  const uint32_t cell = cell_float(g, x, y);
  const int tail = tail_float(x);
  const int e = ey * kEX + ex;

  Mom3 mv;
  float own[3], next[3];  // the populations of velocity (0, 0, *), which stay in their column
  auto fetch = [&](int p) {
    const int zp = p < 0 ? p + g.nz : (p >= g.nz ? p - g.nz : p);
    mv = load_fields(a + zp * plane + cell, tail);
  };
  auto post = [&](int p) {
    float df[Q];
    Lattice<Q>::template synth<MODEL>(macro_of<Q, MODEL>(mv), om1, df);
    float *dst = sm + (p & 1) * plane_shared<Q>();
#pragma unroll
    for (int c = 0; c < 9; ++c) {
      if (c == 4) continue;
      if (has_outer<Q>(c))
        reinterpret_cast<float2 *>(dst)[outer_index<Q>(c) * kE + e] =
            make_float2(df[dir_of<Q>(c, -1)], df[dir_of<Q>(c, 1)]);
      dst[(2 * outers<Q>() + (c < 4 ? c : c - 1)) * kE + e] = df[dir_of<Q>(c, 0)];
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) next[k] = df[dir_of<Q>(4, k - 1)];
  };

  if (active) {
    fetch(z0 - 1);
    post(z0 - 1);
    fetch(z0);
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) own[k] = next[k];
  __syncthreads();
  Part c1{}, c2{}, d1{};  // sums of component +1 of planes p - 1, p - 2; of 0 of plane p - 1
  for (int p = z0 - 1; p <= z1; ++p) {
    if (active && p < z1) {
      post(p + 1);
      if (p + 2 <= z1) fetch(p + 2);
    }
    if (inner) {
      float gm[group_size<Q>(-1)], gz[group_size<Q>(0)], gp[group_size<Q>(1)];
      const float *src = sm + (p & 1) * plane_shared<Q>();
#pragma unroll
      for (int c = 0; c < 9; ++c) {
        const int o = e - (c / 3 - 1) * kEX - (c % 3 - 1);
        if (has_outer<Q>(c)) {
          const float2 v = c == 4 ? make_float2(own[0], own[2])
                                  : reinterpret_cast<const float2 *>(
                                        src)[outer_index<Q>(c) * kE + o];
          gm[in_group<Q>(c, -1)] = v.x;
          gp[in_group<Q>(c, 1)] = v.y;
        }
        gz[c] = c == 4 ? own[1] : src[(2 * outers<Q>() + (c < 4 ? c : c - 1)) * kE + o];
      }
      if (p > z0 && in) {
        store_fields(b + (p - 1) * plane + cell, tail,
                     combine<Q>(part(gm), d1, c2));
      }
      c2 = c1;
      c1 = part(gp);
      d1 = part(gz);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) own[k] = next[k];
    __syncthreads();
  }
}

constexpr int kCellThreads = 128;

// Moments of the logical populations of an AA store of either parity.
template <int Q>
__global__ void __launch_bounds__(kCellThreads)
    moments_of_store_kernel(const float *__restrict__ f, const Grid g, const int parity,
                            float *__restrict__ b) {
  const int x = blockIdx.x * kCellThreads + threadIdx.x;
  if (x >= g.nx) return;
  float df[Q];
  load_logical<Q, 0>(f, g, parity, x, blockIdx.y, blockIdx.z, df);
  store_fields(b + blockIdx.z * plane_floats(g) + cell_float(g, x, blockIdx.y), tail_float(x),
               moments_of<Q>(df));
}

// The update that ends a run: collision from the moments into the AA store, at
// parity 1 into the cell's own slots (population i in slot opp(i)), at parity 0
// streamed to slot i of x + xi_i.
template <int Q, int MODEL, int PARITY>
__global__ void __launch_bounds__(kCellThreads)
    store_of_moments_kernel(const float *__restrict__ a, const Grid g, const float om1,
                            float *__restrict__ f) {
  const int x = blockIdx.x * kCellThreads + threadIdx.x;
  if (x >= g.nx) return;
  const int y = blockIdx.y, z = blockIdx.z;
  const long long cell = ((long long)z * g.ny + y) * g.nx + x;
  float df[Q];
  const Mom3 v = load_fields(a + z * plane_floats(g) + cell_float(g, x, y), tail_float(x));
  Lattice<Q>::template synth<MODEL>(macro_of<Q, MODEL>(v), om1, df);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    if (PARITY == 1) {
      f[(Q - 1 - i) * g.n + cell] = df[i];
    } else {
      const long long row = (long long)wrap_add(z, vel_q<Q>(i, 2), g.nz) * g.ny +
                            wrap_add(y, vel_q<Q>(i, 1), g.ny);
      f[i * g.n + row * g.nx + wrap_add(x, vel_q<Q>(i, 0), g.nx)] = df[i];
    }
  }
}

// z segments of the blocks: the fewest plane iterations of the busiest SM (a
// segment costs two planes more than it holds).
struct RunPlan {
  int tiles_x, tiles_y, seg;
  unsigned blocks;
  long long planes;  // plane iterations of the busiest SM
};
RunPlan plan_of(int ty, const Grid &g, int sms) {
  RunPlan r;
  r.tiles_x = (g.nx + kTX - 1) / kTX;
  r.tiles_y = (g.ny + ty - 1) / ty;
  const long long tiles = (long long)r.tiles_x * r.tiles_y;
  r.planes = -1;
  for (int s = 1; s <= g.nz && s <= 64; ++s) {
    const int len = (g.nz + s - 1) / s, segs = (g.nz + len - 1) / len;
    const long long c = (tiles * segs + sms - 1) / sms * (len + 2);
    if (r.planes < 0 || c < r.planes) {
      r.planes = c;
      r.seg = len;
      r.blocks = (unsigned)(tiles * segs);
    }
  }
  return r;
}

template <int Q, int MODEL>
cudaError_t run_t(float *f, float *m0, float *m1, const Grid &g, float om1, int parity, int steps,
                  int sms, cudaStream_t st) {
  auto kern = rr_moment_step_kernel<Q, MODEL>;
  constexpr int smem = 2 * plane_shared<Q>() * 4, threads = Tile<Q>::kThreads;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const RunPlan r = plan_of(Tile<Q>::TY, g, sms);
  const dim3 cells((g.nx + kCellThreads - 1) / kCellThreads, g.ny, g.nz);
  moments_of_store_kernel<Q><<<cells, kCellThreads, 0, st>>>(f, g, parity, m0);
  for (int k = 1; k < steps; ++k) {
    kern<<<r.blocks, threads, smem, st>>>(m0, m1, g, om1, r.tiles_x, r.tiles_y, r.seg);
    float *s = m0;
    m0 = m1;
    m1 = s;
  }
  if ((parity + steps) & 1)
    store_of_moments_kernel<Q, MODEL, 1><<<cells, kCellThreads, 0, st>>>(m0, g, om1, f);
  else
    store_of_moments_kernel<Q, MODEL, 0><<<cells, kCellThreads, 0, st>>>(m0, g, om1, f);
  return cudaGetLastError();
}

}  // namespace

// Where the run on the moments is the faster one: a store that does not fit
// the 129 MB L2 cache (within it the single updates gain, 35 to 39 GLUPS for
// D3Q27, and the pass over the moments does not), and enough updates on a
// grid its tiles fill. In units of a single update of every cell (216 or 152
// bytes a cell at the copy rate), its first and last passes cost 296 / 216 or
// 232 / 152, and an update between them 0.54 (D3Q27) or 0.60 (D3Q19) of the
// cells its plane iterations could hold, which is what the kernel measures at
// 256^3 and 512^3; 0.08 and 0.14 are added on the safe side. Measured on both
// sides of the lines (microseconds an update, single / moments): 96x60x64
// 10.5 / 15.3, 640x130x9 19.3 / 24.3, 128^3 70.3 / 54.8 (40 updates) and 72.7 /
// 69.3 (3), 250x151x101 131 / 97.2; D3Q19 128^3 50.8 / 52.0 (6 updates),
// 160x145x130 73.8 / 70.9 (9).
bool moment_run_supported(int q, int storage, int model, const Grid &g, int steps, int sms) {
  if (q == 9 || model == 2 || storage != 0 || g.walls || steps < 3 ||
      (long long)g.nx * g.ny > (1LL << 26) || 4LL * q * g.n < 128000000LL)
    return false;
  const int ty = q == 27 ? Tile<27>::TY : Tile<19>::TY;
  const double held = (double)plan_of(ty, g, sms).planes * sms * ty * kTX;
  const double ends = q == 27 ? 296.0 / 216.0 : 232.0 / 152.0, rate = q == 27 ? 0.62 : 0.74;
  return ends * (double)g.n + (steps - 1) * rate * held < (double)steps * (double)g.n;
}
size_t moment_run_bytes(const Grid &g) { return 2 * sizeof(float) * (size_t)plane_floats(g) * g.nz; }

cudaError_t launch_moment_run(int q, int model, void *f, void *scratch, const Grid &g, float om1,
                              int parity, int steps, int sms, cudaStream_t st) {
  float *s = static_cast<float *>(f), *m0 = static_cast<float *>(scratch);
  float *m1 = m0 + plane_floats(g) * g.nz;
  if (q == 19)
    return model == 0 ? run_t<19, 0>(s, m0, m1, g, om1, parity, steps, sms, st)
                      : run_t<19, 1>(s, m0, m1, g, om1, parity, steps, sms, st);
  return model == 0 ? run_t<27, 0>(s, m0, m1, g, om1, parity, steps, sms, st)
                    : run_t<27, 1>(s, m0, m1, g, om1, parity, steps, sms, st);
}

}  // namespace lbrr
