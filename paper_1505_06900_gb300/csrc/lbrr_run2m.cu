// Runs of updates of a large D2Q9 FP32 grid on its moments (see lbrr_run2.cu):
// several updates to a pass, streaming rows.
//
// A block walks down a column of the grid; group u of its threads carries out
// update u + 1 on rows that are two behind those of group u - 1, the rows
// passing from group to group through shared memory (one barrier a row). So
// only the columns overlap (by the number of updates on either side) and the
// ends of a segment; memory is read and written once a pass, 48 bytes a cell
// for three to eight updates. A thread has two cells, half a row apart, in
// packed arithmetic: accesses stay coalesced and free of bank conflicts.
// 2048^2, 50 updates: 28.2 us an update (149 GLUPS) against 46.2 of the single
// updates at 0.96 of the copy rate. Bound: the FMA pipe (packed operations
// issue at half rate; 53% busy over a pass that starts cold, and the warps wait
// for it, for the row's barrier and for their dependent chains in about equal
// parts) at 24 warps an SM;
// with one cell a thread the same walk took 33.3 us (200 instructions a cell
// instead of 139), with loads one row ahead instead of kAhead 45.6.
#include "lbrr_chain.cuh"
#include "lbrr_two.cuh"

namespace lbrr {

namespace {

using namespace two;

template <int BYTES>
__device__ __forceinline__ void copy_async(uint32_t dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(BYTES)
               : "memory");
}

constexpr int kAhead = 6;  // rows in flight from memory
constexpr int kThreads2 = 384;  // two blocks of 12 warps an SM at 80 registers

struct PassM {
  int units;           // updates of the pass
  int tiles_x, ox;     // columns of ox cells
  int seg;             // rows of a segment
  int parity;          // of the store a first pass reads or a last pass leaves
};

// One pass of `units` updates over a segment of a column of EX cells: groups
// 0 .. units of EX / 2 threads. Group 0 takes the rows from memory and collides
// them, group u gathers what group u - 1 collided, reduces it to moments and
// collides it again, the last group gives its moments back. KIND 0: moments to
// moments, 1: the store's populations to moments, 2: moments to the store,
// with one collision more.
template <int EX, int KIND>
__global__ void __launch_bounds__(kThreads2, 2)
    rr_moment_march_kernel(float *f, const float *a, float *b, const Grid g, const float om1,
                           const PassM p) {
  constexpr int H = EX / 2;
  constexpr int RS = EX + 4;      // a row of one population, with guard cells at its ends
  constexpr int BUF = 9 * RS;     // one row of all populations
  extern __shared__ __align__(128) float sm[];
  const int ex = threadIdx.x % H, u = threadIdx.x / H, U = p.units;
  const int x0 = (int)(blockIdx.x % p.tiles_x) * p.ox, y0 = (int)(blockIdx.x / p.tiles_x) * p.seg;
  const int y1 = min(y0 + p.seg, g.ny);
  const long long n = g.n;
  int xu[2], x[2];
  bool out[2];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    xu[c] = x0 + ex + c * H - U;
    x[c] = ((xu[c] % g.nx) + g.nx) % g.nx;
    out[c] = ex + c * H >= U && ex + c * H < U + p.ox && xu[c] < g.nx;
  }

  float *ring = sm + u * 2 * BUF + ex + 1;                               // of this group's update
  const float *prev = ring - 2 * BUF;                                    // of the one before
  const int ys = y0 - U, rounds = y1 - y0 + 3 * U, rows = y1 - y0 + 2 * U;

  // Group 0 copies the rows it starts from kAhead rows ahead, each thread its
  // own cells, into shared memory.
  float *stage = sm + U * 2 * BUF;
  int yl = ((ys % g.ny) + g.ny) % g.ny, fetched = 0;
  auto fetch = [&]() {
    if (fetched < rows) {
      float *to = stage + (fetched % kAhead) * (9 * EX);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        if (KIND == 1) {
          const int ya = yl == 0 ? g.ny - 1 : yl - 1, yb = yl + 1 == g.ny ? 0 : yl + 1;
          const int xa = x[c] == 0 ? g.nx - 1 : x[c] - 1, xb = x[c] + 1 == g.nx ? 0 : x[c] + 1;
          const uint32_t dst = (uint32_t)__cvta_generic_to_shared(to + ex + c * H);
#pragma unroll
          for (int i = 0; i < 9; ++i) {  // population i of the cell (load_logical)
            const int sl = p.parity ? 8 - i : i;
            const int xx = !p.parity || vel(i, 0) == 0 ? x[c] : (vel(i, 0) > 0 ? xa : xb);
            const int yy = !p.parity || vel(i, 1) == 0 ? yl : (vel(i, 1) > 0 ? ya : yb);
            copy_async<4>(dst + i * EX * 4, f + sl * n + (long long)yy * g.nx + xx);
          }
        } else {
          const float *src = a + block2(g, x[c], yl);
          copy_async<16>((uint32_t)__cvta_generic_to_shared(to + 4 * (ex + c * H)),
                         src + 4 * (x[c] & 31));
          copy_async<8>((uint32_t)__cvta_generic_to_shared(to + 4 * EX + 2 * (ex + c * H)),
                        src + 128 + 2 * (x[c] & 31));
        }
      }
      ++fetched;
      yl = yl + 1 == g.ny ? 0 : yl + 1;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  chain_wait();
  if (u == 0)
    for (int k = 0; k < kAhead - 1; ++k) fetch();

  V c1[3] = {}, c2[3] = {}, d1[3] = {};  // rows' lines cy = +1 (last, one before), 0 (last)
  for (int k = 0; k < rounds; ++k) {
    Mom2 m;
    if (u == 0) {
      fetch();
      asm volatile("cp.async.wait_group %0;" ::"n"(kAhead - 1) : "memory");
      const float *from = stage + (k % kAhead) * (9 * EX);
      if (KIND == 1) {
        V df[9];
#pragma unroll
        for (int i = 0; i < 9; ++i)
          df[i] = make_float2(from[i * EX + ex], from[i * EX + ex + H]);
        m = moments_of(df);
      } else {
        const float4 *q4 = reinterpret_cast<const float4 *>(from) + ex;
        const float2 *q2 = reinterpret_cast<const float2 *>(from + 4 * EX) + ex;
        const float4 v = q4[0], w = q4[H];
        const float2 r = q2[0], t = q2[H];
        m = {make_float2(v.x, w.x), make_float2(v.y, w.y), make_float2(v.z, w.z),
             make_float2(v.w, w.w), make_float2(r.x, t.x), make_float2(r.y, t.y)};
      }
    } else {
      const float *src = prev + ((k + 1) & 1) * BUF;
      auto get = [&](int i) {
        const float *q = src + i * RS - vel(i, 0);
        return make_float2(q[0], q[H]);
      };
      V df[9];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        df[i] = get(i);
        df[i + 3] = d1[i];
        df[i + 6] = c2[i];
        c2[i] = c1[i];
        d1[i] = get(i + 3);
        c1[i] = get(i + 6);
      }
      m = moments_of(df);
    }
    if (u < U || KIND == 2) {
      V q[9];
      post_collision(macro_of(m), om1, q);
      if (u < U) {
        float *dst = ring + (k & 1) * BUF;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          dst[i * RS] = q[i].x;
          dst[i * RS + H] = q[i].y;
        }
      } else {
        const int y = ys + k - 2 * U;
#pragma unroll
        for (int c = 0; c < 2; ++c)
          if (out[c] && y >= y0 && y < y1) {
#pragma unroll
            for (int i = 0; i < 9; ++i) {
              const float v = lane(q[i], c);
              if (p.parity == 1)
                f[(8 - i) * n + (long long)y * g.nx + xu[c]] = v;
              else
                f[i * n + (long long)wrap_add(y, vel(i, 1), g.ny) * g.nx +
                  wrap_add(xu[c], vel(i, 0), g.nx)] = v;
            }
          }
      }
    } else {
      const int y = ys + k - 2 * U;
#pragma unroll
      for (int c = 0; c < 2; ++c)
        if (out[c] && y >= y0 && y < y1) {
          float *dst = b + block2(g, xu[c], y);
          reinterpret_cast<float4 *>(dst)[xu[c] & 31] =
              make_float4(lane(m.drho, c), lane(m.jx, c), lane(m.jy, c), lane(m.xx, c));
          reinterpret_cast<float2 *>(dst + 128)[xu[c] & 31] =
              make_float2(lane(m.xy, c), lane(m.yy, c));
        }
    }
    __syncthreads();
  }
}

// The columns and segments of a pass of `units` updates: the row length and
// the number of waves estimated fastest (a round takes 0.22 us and 0.88 ns a
// thread on the SM, measured from 256 to 768 threads; rows of 64 cells, one
// warp a group, 7% more).
PlanM planm(const Grid &g, int units, int sms) {
  PlanM best{};
  best.us = -1;
  for (int ex = 64; ex <= 256; ex *= 2) {
    const int threads = ex / 2 * (units + 1), most = ex - 2 * units;
    if (threads > kThreads2 || most < ex / 4) continue;
    const int tiles_x = (g.nx + most - 1) / most, ox = (g.nx + tiles_x - 1) / tiles_x;
    const int per_sm = 768 / threads < 6 ? 768 / threads : 6;
    for (long long slots = 1; slots <= per_sm; ++slots) {
      for (long long waves = 1; waves <= 8; ++waves) {
        long long ty = waves * slots * sms / tiles_x;
        if (ty < 1) continue;
        if (ty > g.ny) ty = g.ny;
        const int seg = (int)((g.ny + ty - 1) / ty), tiles_y = (g.ny + seg - 1) / seg;
        const double wv =
            (double)(((long long)tiles_x * tiles_y + slots * sms - 1) / (slots * sms));
        const double round = (ex == 64 ? 1.07 : 1.0) * (0.22 + slots * threads * 0.88e-3);
        const double c = wv * (1.5 + (seg + 3 * units) * round) + 1.5;
        if (best.us < 0 || c < best.us) best = {ex, tiles_x, ox, seg, tiles_x * tiles_y, c};
      }
    }
  }
  return best;
}

template <int EX, int KIND>
cudaError_t passm_t(float *f, const float *a, float *b, const Grid &g, float om1, const PassM &p,
                    unsigned blocks, cudaStream_t st) {
  auto kern = rr_moment_march_kernel<EX, KIND>;
  const int smem = (p.units * 2 * 9 * (EX + 4) + kAhead * 9 * EX) * 4;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
  }
  return launch_chained(kern, blocks, EX / 2 * (p.units + 1), smem, st, f, a, b, g, om1, p);
}
template <int KIND>
cudaError_t passm_k(int ex, float *f, const float *a, float *b, const Grid &g, float om1,
                    const PassM &p, unsigned blocks, cudaStream_t st) {
  if (ex == 64) return passm_t<64, KIND>(f, a, b, g, om1, p, blocks, st);
  if (ex == 128) return passm_t<128, KIND>(f, a, b, g, om1, p, blocks, st);
  return passm_t<256, KIND>(f, a, b, g, om1, p, blocks, st);
}

}  // namespace

PlanM plan_march(const Grid &g, int units, int sms) {
  if (units > 0) return planm(g, units, sms);
  PlanM none{};
  none.us = -1;
  return none;
}

cudaError_t launch_march(int kind, float *f, const float *a, float *b, const Grid &g, float om1,
                         const PlanM &q, int units, int parity, cudaStream_t st) {
  const PassM p{units, q.tiles_x, q.ox, q.seg, parity};
  const unsigned n = (unsigned)q.blocks;
  return kind == 0   ? passm_k<0>(q.ex, f, a, b, g, om1, p, n, st)
         : kind == 1 ? passm_k<1>(q.ex, f, a, b, g, om1, p, n, st)
                     : passm_k<2>(q.ex, f, a, b, g, om1, p, n, st);
}

}  // namespace lbrr
