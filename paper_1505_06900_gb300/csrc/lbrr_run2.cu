// Runs of updates of a periodic D2Q9 FP32 grid (RR) on the moments of its cells,
// several updates to a pass.
//
// As in lbrr_run3.cu the state between the first and the last of a run of
// updates is six numbers a cell (rho - 1, rho u, the second moments) instead
// of nine populations, and, the grid being flat, a block can carry a tile with
// a halo through several updates before anything goes back to memory. Small
// and medium grids spend their time on launches (1.9 us an update as a graph
// of single updates) and on L2, so here a block holds its tile in registers
// and exchanges populations through shared memory (kernel below); large grids
// take the kernel of lbrr_run2m.cu, which streams rows. The plan of a grid
// (updates a pass, tiles, kernel) minimises an estimate fitted to both kernels.
// Every value is computed by the operations of the single updates in their
// order, so the store comes out bit for bit as theirs, underflow and the signs of
// zeros included, while the velocities are finite numbers. (Grids with walls stay
// with the single updates: the gain there was 5%, 10.1 -> 9.8 us at 1001^2.)
//
// GB300, microseconds an update, single updates / runs: 128^2 1.91 / 1.07 (50
// updates), 251^2 2.14 / 1.69, 1001^2 9.57 / 7.50, 2048^2 46.2 / 28.2,
// 4096x3000 134 / 75.8 (20 updates). The tile kernel issues in 39% (128^2) and
// 45% (1001^2) of the slots of its active SMs: its phases (collision, exchange,
// sums) follow one another in all warps of a block, and one block fills an SM's
// registers.
#include "lbrr_chain.cuh"
#include "lbrr_two.cuh"

namespace lbrr {

namespace {

using namespace two;

// Shape of a block: cells a thread, threads, cells from one row of the extended
// tile to the next and rows at most, and whether the exchange has two buffers
// (one barrier an update instead of two). The guard cells before and after are
// read by the outermost cells.
template <int K_, int NT_, int STRIDE_, int ROWS_, int BUFS_>
struct Shape {
  static constexpr int K = K_, NT = NT_, STRIDE = STRIDE_, ROWS = ROWS_, BUFS = BUFS_;
  static constexpr int kMax = K * NT, GUARD = STRIDE + 1, SLOT = ROWS * STRIDE + 2 * GUARD;
};
using Small = Shape<2, 512, 48, 48, 2>;
using Mid = Shape<2, 1024, 64, 48, 2>;
using Big = Shape<6, 768, 80, 64, 1>;

struct Pass2 {
  int ox, oy, tiles_x;  // tiles of ox x oy cells
  int ex;               // row length of a tile with its halo
  int units;            // updates of the pass, and cells of halo
  int parity;           // of the store a first pass reads or a last pass leaves
};

// One pass of `units` updates: a block holds the moments of a tile and a halo
// of as many cells in registers, and every update exchanges the populations of
// the cells through shared memory; the cells that lack neighbours grow by one
// ring an update, up to the edge of the tile. KIND 0: moments to moments, 1:
// the store's populations to moments, 2: moments to the store, with one
// collision more.
template <class B, int KIND>
__global__ void __launch_bounds__(B::NT, 1)
    rr_moment_pass2_kernel(float *f, const float *a, float *b, const Grid g, const float om1,
                           const Pass2 p) {
  constexpr int K = B::K, NT = B::NT, SLOT = B::SLOT, P = K / 2;
  constexpr int kStride = B::STRIDE, kGuard = B::GUARD;
  extern __shared__ __align__(128) float sm[];
  const int t = threadIdx.x;
  const int x0 = (int)(blockIdx.x % p.tiles_x) * p.ox, y0 = (int)(blockIdx.x / p.tiles_x) * p.oy;
  const long long n = g.n;
  const int xa = x0 - p.units, ya = y0 - p.units;  // the extended tile
  const int ex = p.ex, cells = ex * (p.oy + 2 * p.units);
  Mom2 m[P];
  uint32_t e[P];  // the places of both cells of a pair, 16 bits each
  auto place = [&](int j, int &x, int &y) {  // cell j of the thread, not wrapped
    const int c = t + j * NT, ey = c / ex;
    x = xa + c - ey * ex;
    y = ya + ey;
    return c < cells;
  };
  chain_wait();
#pragma unroll
  for (int j = 0; j < K; ++j) {
    int x, y;
    Mom2 &mj = m[j / 2];
    const int k = j & 1;
    if (!k) e[j / 2] = 0;
    uint32_t at = kGuard;
    lane(mj.drho, k) = lane(mj.jx, k) = lane(mj.jy, k) = 0.0f;
    lane(mj.xx, k) = lane(mj.xy, k) = lane(mj.yy, k) = 0.0f;
    const bool used = place(j, x, y);
    if (used) at = kGuard + (y - ya) * kStride + (x - xa);
    e[j / 2] |= at << (16 * k);
    if (!used) continue;
    x = x < 0 ? x + g.nx : (x < g.nx ? x : x - g.nx);
    y = y < 0 ? y + g.ny : (y < g.ny ? y : y - g.ny);
    if (x < 0 || x >= g.nx) x = (x % g.nx + g.nx) % g.nx;
    if (y < 0 || y >= g.ny) y = (y % g.ny + g.ny) % g.ny;
    if (KIND == 1) {
      float df[9];
      load_logical<9, 0>(f, g, p.parity, x, y, 0, df);
      V v[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) v[i] = bc(df[i]);
      Mom2 q = moments_of(v);
      lane(mj.drho, k) = q.drho.x;
      lane(mj.jx, k) = q.jx.x;
      lane(mj.jy, k) = q.jy.x;
      lane(mj.xx, k) = q.xx.x;
      lane(mj.xy, k) = q.xy.x;
      lane(mj.yy, k) = q.yy.x;
    } else {
      const float *src = a + block2(g, x, y);
      const float4 u = reinterpret_cast<const float4 *>(src)[x & 31];
      const float2 w = reinterpret_cast<const float2 *>(src + 128)[x & 31];
      lane(mj.drho, k) = u.x;
      lane(mj.jx, k) = u.y;
      lane(mj.jy, k) = u.z;
      lane(mj.xx, k) = u.w;
      lane(mj.xy, k) = w.x;
      lane(mj.yy, k) = w.y;
    }
  }
  for (int s = 0; s < p.units; ++s) {
    float *buf = sm + (B::BUFS == 2 ? (s & 1) * (8 * SLOT) : 0);
    V own[P];
#pragma unroll
    for (int j = 0; j < P; ++j) {
      if (2 * j * NT >= cells) continue;
      V q[9];
      post_collision(macro_of(m[j]), om1, q);
#pragma unroll
      for (int k = 0; k < 2; ++k)
        if (t + (2 * j + k) * NT < cells) {
#pragma unroll
          for (int i = 0; i < 9; ++i)
            if (i != 4)
              buf[(i < 4 ? i : i - 1) * SLOT + (k ? e[j] >> 16 : e[j] & 0xFFFFu)] = lane(q[i], k);
        }
      own[j] = q[4];
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < P; ++j) {
      if (2 * j * NT >= cells) continue;
      V q[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        const int o = (i < 4 ? i : i - 1) * SLOT - vel(i, 1) * kStride - vel(i, 0);
        q[i] = i == 4 ? own[j]
                      : make_float2((buf + (e[j] & 0xFFFFu))[o], (buf + (e[j] >> 16))[o]);
      }
      m[j] = moments_of(q);
    }
    if (B::BUFS == 1) __syncthreads();
  }
#pragma unroll
  for (int j = 0; j < P; ++j) {
    V q[9];
    if (KIND == 2) post_collision(macro_of(m[j]), om1, q);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      int x, y;
      if (!place(2 * j + k, x, y) || x < x0 || y < y0 || x >= x0 + p.ox || y >= y0 + p.oy ||
          x >= g.nx || y >= g.ny)
        continue;
      if (KIND == 2) {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          const float v = lane(q[i], k);
          if (p.parity == 1)
            f[(8 - i) * n + (long long)y * g.nx + x] = v;
          else
            f[i * n + (long long)wrap_add(y, vel(i, 1), g.ny) * g.nx +
              wrap_add(x, vel(i, 0), g.nx)] = v;
        }
      } else {
        float *dst = b + block2(g, x, y);
        reinterpret_cast<float4 *>(dst)[x & 31] =
            make_float4(lane(m[j].drho, k), lane(m[j].jx, k), lane(m[j].jy, k), lane(m[j].xx, k));
        reinterpret_cast<float2 *>(dst + 128)[x & 31] =
            make_float2(lane(m[j].xy, k), lane(m[j].yy, k));
      }
    }
  }
}

template <class B>
bool fits(int ex, int rows) {
  return ex <= B::STRIDE && rows <= B::ROWS && ex * rows <= B::kMax;
}

// The tiles of a pass of `halo` updates: of the row lengths a block can hold,
// and for each of the numbers of waves over the SMs, the one estimated fastest.
Plan2 plan2(const Grid &g, int halo, int sms) {
  Plan2 best{};
  best.us = -1;
  int prev = 0;
  for (int w = Big::STRIDE - 2 * halo; w >= 4; --w) {
    const int tiles_x = (g.nx + w - 1) / w, ox = (g.nx + tiles_x - 1) / tiles_x;
    if (ox == prev) continue;
    prev = ox;
    const int ex = ox + 2 * halo;
    int my = Big::kMax / ex;
    if (my > Big::ROWS) my = Big::ROWS;
    const int mo = my - 2 * halo;
    if (mo < 1) continue;
    const long long least = (long long)tiles_x * ((g.ny + mo - 1) / mo);
    for (long long waves = (least + sms - 1) / sms, k = 0; k < 3; ++k, ++waves) {
      long long ty = waves * sms / tiles_x;
      if (ty > g.ny) ty = g.ny;
      const int oy = (int)((g.ny + ty - 1) / ty), tiles_y = (g.ny + oy - 1) / oy;
      const int rows = oy + 2 * halo, cells = ex * rows;
      const long long wv = ((long long)tiles_x * tiles_y + sms - 1) / sms;
      const double update = fits<Small>(ex, rows)  ? 0.30 + cells * 0.5e-3
                            : fits<Mid>(ex, rows) ? 0.35 + cells * 0.5e-3
                                                  : 0.40 + cells * 0.66e-3;
      const double c = wv * (2.0 + halo * update) + 2.0;
      if (best.us < 0 || c < best.us) best = {tiles_x, tiles_y, ox, oy, ex, cells, c};
    }
  }
  return best;
}

template <class B, int KIND>
cudaError_t pass2_t(float *f, const float *a, float *b, const Grid &g, float om1, const Pass2 &p,
                    unsigned blocks, cudaStream_t st) {
  auto kern = rr_moment_pass2_kernel<B, KIND>;
  constexpr int smem = B::BUFS * 8 * B::SLOT * 4;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  return launch_chained(kern, blocks, B::NT, smem, st, f, a, b, g, om1, p);
}
template <int KIND>
cudaError_t pass2_k(float *f, const float *a, float *b, const Grid &g, float om1, const Pass2 &p,
                    unsigned blocks, cudaStream_t st) {
  const int rows = p.oy + 2 * p.units;
  if (fits<Small>(p.ex, rows)) return pass2_t<Small, KIND>(f, a, b, g, om1, p, blocks, st);
  if (fits<Mid>(p.ex, rows)) return pass2_t<Mid, KIND>(f, a, b, g, om1, p, blocks, st);
  return pass2_t<Big, KIND>(f, a, b, g, om1, p, blocks, st);
}

}  // namespace

// Fewer than six updates do not pay for the first and last passes, which touch
// the store (1001^2: 12.3 us an update singly, 15.4 as a run of 4, 9.8 as one
// of 6), except on small grids, where launches count (128^2, 4 updates: 4.2 /
// 3.2).
bool moment_run2_supported(int q, int storage, int model, const Grid &g, int steps) {
  if (q != 9 || storage != 0 || model != 0 || g.walls) return false;
  return steps >= 6 || (steps >= 4 && g.n <= (1 << 19));
}
size_t moment_run2_bytes(const Grid &g) {
  return 2 * sizeof(float) * 192 * (size_t)blocks2_x(g) * (size_t)g.ny;
}
void plan_moment_run2(const Grid &g, int sms, Run2Plans *plans) {
  for (int h = 0; h <= kRun2Units; ++h) {
    plans->tile[h] = plan2(g, h, sms);
    plans->march[h] = plan_march(g, h, sms);
  }
  plans->ready = true;
}

cudaError_t launch_moment_run2(void *f, void *scratch, const Grid &g, float om1, int parity,
                               int steps, const Run2Plans &plans, bool *rows, cudaStream_t st) {
  float *s = static_cast<float *>(f), *m0 = static_cast<float *>(scratch);
  float *m1 = m0 + 192 * (size_t)blocks2_x(g) * (size_t)g.ny;
  // updates a pass: the cheapest by the estimate, shared out evenly; the last
  // pass ends with its collision written to the store, one update more
  const int moving = steps - 1;
  int passes = 0;
  bool march = false;
  double cost = -1;
  for (int t = 1; t <= kRun2Units; ++t) {
    int k = (moving + t - 1) / t;
    if (k < 2) k = 2;
    const int per = (moving + k - 1) / k, least = moving / k;
    for (int w = 0; w < 2; ++w) {
      const double us = w ? plans.march[per].us : plans.tile[per].us;
      if (us < 0 || (w ? plans.march[least].us : plans.tile[least].us) < 0) continue;
      if (cost < 0 || k * us < cost) {
        cost = k * us;
        passes = k;
        march = w;
      }
    }
  }
  *rows = march;
  if (cost < 0) return cudaErrorInvalidValue;
  int done = 0;
  for (int k = 0; k < passes; ++k) {
    const int units = (int)((long long)moving * (k + 1) / passes) - done;
    const bool last = k == passes - 1;
    const int kind = k == 0 ? 1 : (last ? 2 : 0), par = last ? (parity + steps) & 1 : parity;
    cudaError_t e;
    if (march) {
      e = launch_march(kind, s, m0, m1, g, om1, plans.march[units], units, par, st);
    } else {
      const Plan2 &q = plans.tile[units];
      const Pass2 p{q.ox, q.oy, q.tiles_x, q.ex, units, par};
      const unsigned n = (unsigned)q.tiles_x * (unsigned)q.tiles_y;
      e = kind == 0   ? pass2_k<0>(s, m0, m1, g, om1, p, n, st)
          : kind == 1 ? pass2_k<1>(s, m0, m1, g, om1, p, n, st)
                      : pass2_k<2>(s, m0, m1, g, om1, p, n, st);
    }
    if (e != cudaSuccess) return e;
    float *x = m0;
    m0 = m1;
    m1 = x;
    done += units;
  }
  return cudaSuccess;
}

}  // namespace lbrr
