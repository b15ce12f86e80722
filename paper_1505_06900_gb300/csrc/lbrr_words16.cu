// Collide-and-stream kernel of the 16-bit population stores for rows that are
// not whole 16-byte chunks, two neighbouring cells to a thread.
//
// AA pattern and arithmetic as in lbrr_step.cu (one cell after the other in
// scalar FP32, so the populations are the same bit for bit). With one cell to
// a thread a warp's access is 64 bytes and too few bytes are in flight: D3Q19
// BF16 on 250 x 150 x 101 took 74 us in the even update and 70 in the odd one,
// which also spent three quarters of its issue slots, half of them on
// addresses; 288 MB take 43 at the rate of a copy. Here a slot that is not
// shifted along x moves as one 32-bit word of two cells, the shifted slots of
// the odd update, whose pairs straddle words, as two halves, and addresses are
// 32-bit offsets wherever the store is below 4 GB. The two cells' populations
// stay packed in their words while a cell is computed. 50 and 60 us, now
// bound by the issue of the scalar arithmetic (70 to 75% of the slots); FP16
// D3Q27 on 250 x 150 x 100 99 -> 81 a step, D2Q9 on 2050 x 2050 31.3 -> 27.9.
//
// The even update is a walk over words whatever the rows (cell count even); the
// odd one takes rows of an even number of cells.
#include <algorithm>

#include "lbrr_launch.h"

namespace lbrr {

namespace {

constexpr int kWordThreads = 128;  // at most

// Post-collision populations of the word's two cells in place of theirs: twice
// the low half, each time moving the other half down and the result on top. The
// loop is kept: with both cells' work in one stretch of code they are computed
// side by side, in up to twice the registers.
template <int Q, int S, int MODEL>
__device__ __forceinline__ void collide_words(uint32_t (&w)[Q], float om1) {
  using St = Storage<S>;
  using T = typename St::T;
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    float df[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const uint16_t b = (uint16_t)w[i];
      df[i] = St::template load<Q>(reinterpret_cast<const T *>(&b), i);
    }
    const Macro m = Lattice<Q>::moments(df);
    Lattice<Q>::template synth<MODEL>(m, om1, df);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      T v;
      St::template store<Q>(&v, i, df[i]);
      w[i] = __byte_perm(w[i], *reinterpret_cast<const uint16_t *>(&v), 0x5432);
    }
  }
}

// Value of type U at byte offset off of slot s, the offsets within a slot being
// below 2^32; SIZE: unsigned where the whole store's are.
template <typename U, typename SIZE>
__device__ __forceinline__ U &at(char *f, int s, SIZE slot_bytes, unsigned off) {
  return *reinterpret_cast<U *>(f + (s * slot_bytes + off));
}

template <int Q, int S, int MODEL>
__global__ void __launch_bounds__(kWordThreads)
    rr_step_words16_even_kernel(char *__restrict__ f, const unsigned nw, const float om1) {
  const unsigned c = blockIdx.x * kWordThreads + threadIdx.x;
  if (c >= nw) return;
  const size_t slot = 4 * (size_t)nw;
  uint32_t w[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) w[i] = at<uint32_t>(f, i, slot, 4 * c);
  collide_words<Q, S, MODEL>(w, om1);
  unsigned out = 4 * c;
  asm volatile("" : "+r"(out));  // addresses anew, not kept across the collision
#pragma unroll
  for (int i = 0; i < Q; ++i) at<uint32_t>(f, Q - 1 - i, slot, out) = w[i];
}

// Byte offsets, within a slot, around the cells x and x + 1 of row (y, z).
template <int Q>
struct Place {
  unsigned xm, x0, x1, xp;  // of the cells x - 1 .. x + 2
  unsigned rows[3][3];      // [1 + cz][1 + cy] of the rows
  __device__ __forceinline__ Place(const Grid &g, int x, int y, int z) {
    constexpr bool k3 = Lattice<Q>::D == 3;
    x0 = 2 * x;
    x1 = x0 + 2;
    xm = x == 0 ? 2 * g.nx - 2 : x0 - 2;
    xp = x + 2 == g.nx ? 0 : x0 + 4;
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int b = 0; b < 3; ++b)
        rows[c][b] = 2u * (unsigned)g.nx *
                     ((unsigned)(k3 ? wrap_add(z, c - 1, g.nz) : 0) * (unsigned)g.ny +
                      (unsigned)wrap_add(y, b - 1, g.ny));
  }
  // hides from the compiler what the values were computed from
  __device__ __forceinline__ void forget() {
    asm volatile("" : "+r"(xm), "+r"(x0), "+r"(x1), "+r"(xp));
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int b = 0; b < 3; ++b)
        if (Lattice<Q>::D == 3 || c == 1) asm volatile("" : "+r"(rows[c][b]));
  }
  // the row to which population s goes
  __device__ __forceinline__ unsigned row(int s) const {
    return rows[Lattice<Q>::D == 3 ? 1 + vel_q<Q>(s, 2) : 1][1 + vel_q<Q>(s, 1)];
  }
};

// A block covers blockDim.x pairs of blockDim.y rows.
template <int Q, int S, int MODEL, typename SIZE>
__global__ void __launch_bounds__(kWordThreads)
    rr_step_words16_odd_kernel(char *__restrict__ f, const Grid g, const float om1) {
  const int x = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
  const int y = blockIdx.y * blockDim.y + threadIdx.y, z = blockIdx.z;
  if (x >= g.nx || y >= g.ny) return;
  const SIZE slot = 2 * (SIZE)g.n;
  Place<Q> p(g, x, y, z);
  uint32_t w[Q];
  // population i of cell c lives in slot opp(i) of c - xi_i, in that slot's row
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int s = Q - 1 - i, cx = vel_q<Q>(s, 0);
    const unsigned r = p.row(s);
    if (cx == 0)
      w[i] = at<uint32_t>(f, s, slot, r + p.x0);
    else
      w[i] = (uint32_t)at<uint16_t>(f, s, slot, r + (cx > 0 ? p.x1 : p.xm)) |
             (uint32_t)at<uint16_t>(f, s, slot, r + (cx > 0 ? p.xp : p.x0)) << 16;
  }
  collide_words<Q, S, MODEL>(w, om1);
  p.forget();  // the sums anew, not kept across the collision
#pragma unroll
  for (int s = 0; s < Q; ++s) {
    const int cx = vel_q<Q>(s, 0);
    const unsigned r = p.row(s);
    if (cx == 0) {
      at<uint32_t>(f, s, slot, r + p.x0) = w[s];
    } else {
      at<uint16_t>(f, s, slot, r + (cx > 0 ? p.x1 : p.xm)) = (uint16_t)w[s];
      at<uint16_t>(f, s, slot, r + (cx > 0 ? p.xp : p.x0)) = (uint16_t)(w[s] >> 16);
    }
  }
}

template <int Q, int S, int MODEL>
cudaError_t words_t(void *f, const Grid &g, float om1, int parity, cudaStream_t st) {
  if (parity == 0) {
    const unsigned nw = (unsigned)(g.n / 2);
    rr_step_words16_even_kernel<Q, S, MODEL>
        <<<(nw + kWordThreads - 1) / kWordThreads, kWordThreads, 0, st>>>(
            static_cast<char *>(f), nw, om1);
  } else {
    // equal parts of a row, and as many rows as fit beside each other
    const int pairs = g.nx / 2, parts = (pairs + kWordThreads - 1) / kWordThreads;
    const dim3 block((pairs + parts - 1) / parts,
                     std::min(g.ny, kWordThreads / ((pairs + parts - 1) / parts)));
    const dim3 grid(parts, (g.ny + block.y - 1) / block.y, g.nz);
    if (2 * Q * g.n < (1LL << 32))
      rr_step_words16_odd_kernel<Q, S, MODEL, unsigned>
          <<<grid, block, 0, st>>>(static_cast<char *>(f), g, om1);
    else
      rr_step_words16_odd_kernel<Q, S, MODEL, size_t>
          <<<grid, block, 0, st>>>(static_cast<char *>(f), g, om1);
  }
  return cudaGetLastError();
}

template <int Q, int S>
cudaError_t words_m(int model, void *f, const Grid &g, float om1, int parity, cudaStream_t st) {
  switch (model) {
    case 0: return words_t<Q, S, 0>(f, g, om1, parity, st);
    case 1: return words_t<Q, S, 1>(f, g, om1, parity, st);
    default: return words_t<Q, S, 2>(f, g, om1, parity, st);
  }
}

}  // namespace

// A thread takes twice as long, so a store must be large enough to fill the GPU
// with half the threads. us an update, this and one cell to a thread: D3Q27 of
// 34^3 cells (1.1 million populations) 3.8 and 4.2, 26^3 (0.5) 2.9 and 2.6; D3Q19
// of 42^3 (1.4) 3.2 and 4.2, 34^3 (0.7) 3.2 and 2.9; D2Q9 of 450^2 (1.8) 3.2 and
// 3.5, 350^2 (1.1) 2.9 and 2.6.
constexpr long long kMinPopulations = 1250000;

bool words16_supported(int q, const Grid &g, int parity) {
  return g.walls == 0 && (parity ? g.nx : g.n) % 2 == 0 && g.n < (1LL << 31) &&
         q * g.n >= kMinPopulations;
}

cudaError_t launch_step_words16(int q, int storage, int model, void *f, const Grid &g, float om1,
                                int parity, cudaStream_t st) {
  if (q == 9)
    return storage == 1 ? words_m<9, 1>(model, f, g, om1, parity, st)
                        : words_m<9, 2>(model, f, g, om1, parity, st);
  if (q == 19)
    return storage == 1 ? words_m<19, 1>(model, f, g, om1, parity, st)
                        : words_m<19, 2>(model, f, g, om1, parity, st);
  return storage == 1 ? words_m<27, 1>(model, f, g, om1, parity, st)
                      : words_m<27, 2>(model, f, g, om1, parity, st);
}

}  // namespace lbrr
