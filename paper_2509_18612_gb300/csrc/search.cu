// Combinatorial companions of the solver on the same device graph:
//
//  * the greedy MaxCut comparator (App. C.1): a run fixes a vertex ordering,
//    puts the first vertex in S and every later one on the side that cuts
//    more edges to the vertices already placed (ties: S).  Run b uses the
//    random ordering pi_b of [0, n): a balanced 4-round Feistel network on
//    [0, 4^h) whose round function is word 0 of Philox counter
//    (R, b, round, STREAM_ORDER), with cycle walking onto [0, n).  One warp
//    per run; the runs are independent.
//
//  * 1-flip local search on rounded vectors (bit-packed, n x ceil(B/32)
//    words): every round computes the cut change of flipping each node alone,
//    gain_v = sum_u w_vu s_u s_v (s = +-1 side), and flips every node whose
//    gain is positive and larger than the gain of each neighbour with a
//    positive gain (equal gains: the lower index wins).  Those nodes are
//    pairwise non-adjacent, so the cut grows by the sum of their gains; the
//    search ends at a 1-flip local optimum or after max_rounds rounds.  A
//    device flag per round lets the remaining rounds return at once.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "api_util.cuh"
#include "deco_internal.cuh"
#include "slab.cuh"

namespace cg = cooperative_groups;

namespace deco {

int device_sm_count();

namespace {

struct Feistel {
  int h;            // bits per half
  uint32_t mask;    // 2^h - 1
  uint32_t n;
  uint32_t k0, k1;

  __device__ __forceinline__ uint32_t net(uint32_t x, uint32_t b) const {
    uint32_t L = x >> h, R = x & mask;
#pragma unroll
    for (uint32_t i = 0; i < 4; ++i) {
      const uint4 f = philox4x32_10(make_uint4(R, b, i, STREAM_ORDER), k0, k1);
      const uint32_t t = R;
      R = L ^ (f.x & mask);
      L = t;
    }
    return (L << h) | R;
  }
};

// order[b n + k] = pi_b(k).  TABLE: the round function of run b takes 2^h
// values of R in each of the 4 rounds, so the block tabulates them (4 x 2^h
// Philox calls instead of four per step of every walk) in shared memory.  A
// thread walks one item after another, so that a warp is not held by its
// longest walk.  Measured, 5 000 x 256 items: 19 us; Philox in every step 129.
constexpr int ORDER_MAX_H = 12;   // 4 x 2^12 16-bit words: 32 KB

template <bool TABLE>
__global__ void __launch_bounds__(256) k_orders(Feistel F, int32_t B, int32_t* order) {
  extern __shared__ uint16_t tab[];
  const uint32_t b = blockIdx.x, half = F.mask + 1u;
  if (TABLE) {
    for (uint32_t i = threadIdx.x; i < 4u * half; i += blockDim.x)
      tab[i] = (uint16_t)(philox4x32_10(make_uint4(i & F.mask, b, i >> F.h, STREAM_ORDER), F.k0, F.k1).x & F.mask);
    __syncthreads();
  }
  const uint32_t step = gridDim.y * blockDim.x;
  uint32_t k = blockIdx.y * blockDim.x + threadIdx.x;
  if (k >= F.n) return;
  uint32_t x = k;
  for (;;) {
    // a cycle of the bijection on [0, 4^h) passes through [0, n): every walk ends
    if (TABLE) {
      uint32_t L = x >> F.h, R = x & F.mask;
#pragma unroll
      for (uint32_t i = 0; i < 4; ++i) {
        const uint32_t t = R;
        R = L ^ tab[i * half + R];
        L = t;
      }
      x = (L << F.h) | R;
    } else {
      x = F.net(x, b);
    }
    if (x >= F.n) continue;
    order[(size_t)b * F.n + k] = (int32_t)x;
    if (F.n - k <= step) return;
    x = k += step;
  }
}

// One run per block places its vertices in order: warp 0 places, warp 1 loads
// ahead of it.  Bound by the chain of n dependent placements: a shared load of
// the neighbours' sides (2: not placed), a warp reduction, a shared store.
// Warp 1 fills the list of the next WIN vertices (vertex, row, first 64
// entries) in shared memory while warp 0 works on this one; of longer rows the
// rest is read in place, several loads at once.  The sides of a run are a byte
// or two bits per vertex in shared memory, which go to the run's part of
// `order` at the end (it has consumed it; 4 n bytes of stride), or column b of
// z: greedy_plan.  Measured, degree 10, 256 runs of 5 000 vertices: 0.54 ms;
// loading ahead from the same warp 1.07, with the whole chain of loads in each
// placement 4.28.  Degree 300, one run: 4.0 ms; one load after another on long
// rows 8.9.
enum GreedySides : int { GREEDY_BYTES = 0, GREEDY_BITS = 1, GREEDY_COLUMN = 2 };

template <bool WT, int WIN>
struct GreedyWindow {
  int4 row[WIN];                                  // vertex, first entry, entries
  int32_t u[WIN][64];                             // neighbours (-1: none)
  int32_t w[WT ? WIN : 1][64];
};

template <bool WT, int SIDES, int WIN>
__global__ void __launch_bounds__(64) k_greedy(int32_t n, int32_t B, const int32_t* __restrict__ row_ptr,
                                               const int32_t* __restrict__ col_idx, const int32_t* __restrict__ wint,
                                               int32_t* order, uint8_t* z) {
  extern __shared__ __align__(16) uint8_t sides[];
  __shared__ GreedyWindow<WT, WIN> win[2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int32_t b = blockIdx.x;
  int32_t* const ord = order + (size_t)b * n;
  uint32_t* const words = reinterpret_cast<uint32_t*>(sides);
  if (SIDES != GREEDY_COLUMN)
    for (int i = threadIdx.x; i < (SIDES == GREEDY_BYTES ? (n + 3) / 4 : (n + 15) / 16); i += 64)
      words[i] = SIDES == GREEDY_BYTES ? 0x02020202u : 0xAAAAAAAAu;
  // rows of the window after the next, one per lane (warp 1)
  int32_t v = -1, e0 = 0, d = 0;
  auto rows = [&](int32_t k) {
    v = lane < WIN && k + lane < n ? ord[k + lane] : -1;
    e0 = v >= 0 ? __ldg(row_ptr + v) : 0;
    d = v >= 0 ? __ldg(row_ptr + v + 1) - e0 : 0;
  };
  auto fill = [&](GreedyWindow<WT, WIN>& g) {
    if (lane < WIN) g.row[lane] = make_int4(v, e0, d, 0);
    int32_t u[WIN][2], w[WT ? WIN : 1][2];
#pragma unroll
    for (int j = 0; j < WIN; ++j) {
      const int32_t ej = __shfl_sync(0xFFFFFFFFu, e0, j), dj = __shfl_sync(0xFFFFFFFFu, d, j);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        u[j][h] = -1;
        if (WT) w[WT ? j : 0][h] = 0;
        if (32 * h + lane < dj) {
          u[j][h] = __ldg(col_idx + ej + 32 * h + lane);
          if (WT) w[WT ? j : 0][h] = __ldg(wint + ej + 32 * h + lane);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < WIN; ++j)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        g.u[j][32 * h + lane] = u[j][h];
        if (WT) g.w[WT ? j : 0][32 * h + lane] = w[WT ? j : 0][h];
      }
  };
  if (warp == 1) {
    rows(0);
    fill(win[0]);
    rows(WIN);
  }
  __syncthreads();
  for (int32_t k0 = 0, s = 0; k0 < n; k0 += WIN, s ^= 1) {
    if (warp == 1) {
      fill(win[s ^ 1]);
      rows(k0 + 2 * WIN);
    } else {
      const GreedyWindow<WT, WIN>& g = win[s];
      const int cnt = min(WIN, n - k0);
      auto vote = [&](int32_t u, int32_t w) -> int32_t {
        // w if the neighbour is in S-bar (placing v in S cuts the edge), -w if in S, 0 if not placed
        int x = 2;
        if (u >= 0)
          x = SIDES == GREEDY_BYTES ? sides[u] : SIDES == GREEDY_BITS ? (words[u >> 4] >> (2 * (u & 15))) & 3u
                                                                        : z[(size_t)u * B + b];
        return x == 0 ? w : x == 1 ? -w : 0;
      };
      int4 r = g.row[0];
      int32_t u0 = g.u[0][lane], w0 = WT ? g.w[0][lane] : 1;
      for (int j = 0; j < cnt; ++j) {
        const int4 cur = r;
        const int32_t u = u0, w = w0;
        const int jn = j + 1 < cnt ? j + 1 : j;
        int32_t t = vote(u, w);
        r = g.row[jn];                                    // the next vertex's list, meanwhile
        u0 = g.u[jn][lane];
        if (WT) w0 = g.w[WT ? jn : 0][lane];
        if (cur.z > 32) {
          t += vote(g.u[j][32 + lane], WT ? g.w[WT ? j : 0][32 + lane] : 1);
          // the entries from x on: 32 N at a time while more than `over` are left
          int32_t x = 64;
          auto tail = [&](auto count, int32_t over) {
            constexpr int N = decltype(count)::value;
            for (; cur.z - x > over; x += 32 * N) {
              int32_t ux[N], wx[N];
#pragma unroll
              for (int q = 0; q < N; ++q) {
                const int32_t at = x + 32 * q + lane;
                ux[q] = at < cur.z ? __ldg(col_idx + cur.y + at) : -1;
                wx[q] = WT && at < cur.z ? __ldg(wint + cur.y + at) : 1;
              }
#pragma unroll
              for (int q = 0; q < N; ++q) t += vote(ux[q], wx[q]);
            }
          };
          tail(std::integral_constant<int, 8>{}, 128);
          tail(std::integral_constant<int, 4>{}, 64);
          tail(std::integral_constant<int, 1>{}, 0);
        }
        // |sum| <= sum of the row's |w| <= 2^24 (checked when the graph is created)
        const int32_t sum = __reduce_add_sync(0xFFFFFFFFu, t);
        if (lane == 0) {
          const uint32_t side = sum >= 0 ? 1u : 0u;
          if (SIDES == GREEDY_BYTES) sides[cur.x] = (uint8_t)side;
          else if (SIDES == GREEDY_BITS) atomicXor(words + (cur.x >> 4), (2u ^ side) << (2 * (cur.x & 15)));
          else z[(size_t)cur.x * B + b] = (uint8_t)side;
        }
        __syncwarp();   // the next vertices read this side
      }
    }
    __syncthreads();
  }
  if (SIDES != GREEDY_COLUMN) {
    uint8_t* out = reinterpret_cast<uint8_t*>(ord);
    for (int i = threadIdx.x; i < n; i += 64)
      out[i] = SIDES == GREEDY_BYTES ? sides[i] : (uint8_t)((words[i >> 4] >> (2 * (i & 15))) & 3u);
  }
}

// run-major sides (run b at src + 4 n b bytes) to z (n x B bytes) and bits (n x W words): a warp per 32 x 32 tile
__global__ void __launch_bounds__(256) k_sides_out(int32_t n, int32_t B, int32_t W, const uint8_t* __restrict__ src,
                                                   uint8_t* z, uint32_t* bits) {
  __shared__ uint8_t t[8][32][33];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int64_t tiles = (int64_t)((n + 31) / 32) * W, warps = (int64_t)gridDim.x * 8;
  for (int64_t i = (int64_t)blockIdx.x * 8 + wib; i < tiles; i += warps) {
    const int32_t v0 = (int32_t)(i / W) * 32, k = (int32_t)(i % W);
    __syncwarp();
#pragma unroll 8
    for (int c = 0; c < 32; ++c)
      t[wib][c][lane] = 32 * k + c < B && v0 + lane < n ? src[(size_t)(32 * k + c) * 4 * n + v0 + lane] : 0;
    __syncwarp();
    for (int r = 0; r < 32 && v0 + r < n; ++r) {
      const uint8_t x = t[wib][lane][r];
      if (32 * k + lane < B) z[(size_t)(v0 + r) * B + 32 * k + lane] = x;
      const uint32_t word = __ballot_sync(0xFFFFFFFFu, x != 0);
      if (lane == 0) bits[(size_t)(v0 + r) * W + k] = word;
    }
  }
}

// bits (n x W words, bit b % 32 of word b / 32) -> bytes (n x B)
__global__ void k_bits_to_bytes(int32_t n, int32_t B, int32_t W, const uint32_t* bits, uint8_t* z) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)n * B) return;
  const int32_t v = (int32_t)(i / B), b = (int32_t)(i % B);
  z[i] = (uint8_t)((bits[(size_t)v * W + b / 32] >> (b % 32)) & 1u);
}

// gains[v][32k + c] = sum_u w_vu (+1 same side, -1 other side) for column 32k + c
__global__ void k_ls_gain(int32_t n, int32_t W, const int32_t* row_ptr, const int32_t* col_idx, const int32_t* wint,
                          const uint32_t* zb, int32_t* gains, const int32_t* run) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)n * W || !*run) return;
  const int32_t v = (int32_t)(i / W), k = (int32_t)(i % W);
  const uint32_t zv = zb[i];
  int32_t acc[32];
#pragma unroll
  for (int c = 0; c < 32; ++c) acc[c] = 0;
  for (int32_t e = row_ptr[v]; e < row_ptr[v + 1]; ++e) {
    const int32_t u = col_idx[e];
    const int32_t w = wint ? wint[e] : 1;
    const uint32_t x = zb[(size_t)u * W + k] ^ zv;
#pragma unroll
    for (int c = 0; c < 32; ++c) acc[c] += ((x >> c) & 1u) ? -w : w;
  }
  int32_t* out = gains + (size_t)v * 32 * W + 32 * k;
#pragma unroll
  for (int c = 0; c < 32; ++c) out[c] = acc[c];
}

__global__ void k_ls_flip(int32_t n, int32_t W, int32_t B, const int32_t* row_ptr, const int32_t* col_idx,
                          const int32_t* gains, uint32_t* zb, const int32_t* run, int32_t* next) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)n * W || !*run) return;
  const int32_t v = (int32_t)(i / W), k = (int32_t)(i % W);
  const int32_t* gv = gains + (size_t)v * 32 * W + 32 * k;
  int32_t g[32];
  uint32_t pos = 0;
#pragma unroll
  for (int c = 0; c < 32; ++c) {
    g[c] = gv[c];
    if (g[c] > 0 && 32 * k + c < B) pos |= 1u << c;
  }
  if (!pos) return;
  uint32_t beaten = 0;
  for (int32_t e = row_ptr[v]; e < row_ptr[v + 1] && (pos & ~beaten); ++e) {
    const int32_t u = col_idx[e];
    const int32_t* gu = gains + (size_t)u * 32 * W + 32 * k;
#pragma unroll
    for (int c = 0; c < 32; ++c) {
      const int32_t x = gu[c];
      if (((pos >> c) & 1u) && x > 0 && (x > g[c] || (x == g[c] && u < v))) beaten |= 1u << c;
    }
  }
  const uint32_t flip = pos & ~beaten;
  if (flip) {
    zb[i] ^= flip;
    *next = 1;
  }
}

// ---- gains as bit planes.  A word's 32 columns are
// worked on together: the neighbours on the side that a flip would lose are
// counted by ripple-carry adders over bit planes (plane p holds bit p of every
// column's count), positive gains are kept as NP planes, and two nodes' gains
// compare in two operations a plane.  A thread owns a (row, word).  Integral
// weights (GEN) count an entry once for every set bit of |w|, from that bit's
// plane up; the sum of |w| takes the degree's place.
template <int NP>
__device__ __forceinline__ void planes_load(const uint32_t* p, uint32_t* g) {
#pragma unroll
  for (int h = 0; h < NP / 4; ++h) {
    const uint4 q = __ldcg(reinterpret_cast<const uint4*>(p) + h);
    g[4 * h] = q.x; g[4 * h + 1] = q.y; g[4 * h + 2] = q.z; g[4 * h + 3] = q.w;
  }
}

template <int NP>
__device__ __forceinline__ void planes_store(uint32_t* p, const uint32_t* g) {
#pragma unroll
  for (int h = 0; h < NP / 4; ++h)
    __stcg(reinterpret_cast<uint4*>(p) + h, make_uint4(g[4 * h], g[4 * h + 1], g[4 * h + 2], g[4 * h + 3]));
}

// counts: add 1 to the columns of x
template <int NP>
__device__ __forceinline__ void ls_count(uint32_t* c, uint32_t x) {
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    const uint32_t t = c[p] & x;
    c[p] ^= x;
    x = t;
  }
}

// counts: add a to the columns of x
template <int NP>
__device__ __forceinline__ void ls_count_weight(uint32_t* c, uint32_t x, uint32_t a) {
#pragma unroll
  for (int b = 0; b < NP; ++b) {
    if (!(a >> b)) break;
    uint32_t y = (a >> b) & 1u ? x : 0u;
#pragma unroll
    for (int p = b; p < NP; ++p) {
      const uint32_t t = c[p] & y;
      c[p] ^= y;
      y = t;
    }
  }
}

// g = d - 2 c where that is positive (columns `cols`), else 0; returns the columns with a positive gain
template <int NP>
__device__ __forceinline__ uint32_t ls_gain(const uint32_t* c, int32_t d, uint32_t cols, uint32_t* g) {
  uint32_t borrow = 0u, any = 0u;
#pragma unroll
  for (int p = 0; p <= NP; ++p) {
    const uint32_t a = p < NP && ((d >> p) & 1) ? 0xFFFFFFFFu : 0u, b = p ? c[p > 0 ? p - 1 : 0] : 0u;
    if (p < NP) g[p < NP ? p : 0] = a ^ b ^ borrow;
    borrow = (~a & (b | borrow)) | (b & borrow);
  }
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    g[p] &= ~borrow & cols;
    any |= g[p];
  }
  return any;
}

// columns where gu > g, or gu == g and `lower` (the other node has the lower index)
template <int NP>
__device__ __forceinline__ uint32_t ls_beats(const uint32_t* gu, const uint32_t* g, bool lower) {
  uint32_t beats = lower ? 0xFFFFFFFFu : 0u;
#pragma unroll
  for (int p = 0; p < NP; ++p) beats = (gu[p] & ~g[p]) | (~(gu[p] ^ g[p]) & beats);
  return beats;
}

// col: index, or index | sign bit of a +-1 graph; wint: weights (GEN).  zk: the word column, row u at zk[u W].
template <int NP, bool GEN>
__device__ __forceinline__ void ls_gain_row(int32_t v, int32_t W, const int32_t* __restrict__ row_ptr,
                                            const uint32_t* __restrict__ col, const int32_t* __restrict__ wint,
                                            const uint32_t* zk, uint32_t cols, uint32_t* gains) {
  const int32_t e0 = __ldg(row_ptr + v), e1 = __ldg(row_ptr + v + 1);
  const uint32_t zv = zk[(size_t)v * W];
  uint32_t c[NP], g[NP];
  int32_t sum = GEN ? 0 : e1 - e0;
#pragma unroll
  for (int p = 0; p < NP; ++p) c[p] = 0u;
  for (int32_t e = e0; e < e1; e += 8) {
    uint32_t u[8], x[8];
    int32_t w[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      u[q] = __ldg(col + min(e + q, e1 - 1));
      if (GEN) w[q] = e + q < e1 ? __ldg(wint + e + q) : 0;
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = zk[(size_t)(u[q] & 0x7FFFFFFFu) * W];
    // columns where the entry is lost to a flip: the other side of a +1, the same side of a -1
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      if (GEN) {
        sum += abs(w[q]);
        ls_count_weight<NP>(c, x[q] ^ zv ^ (w[q] < 0 ? 0xFFFFFFFFu : 0u), (uint32_t)abs(w[q]));
      } else {
        ls_count<NP>(c, e + q < e1 ? x[q] ^ zv ^ ((u[q] & 0x80000000u) ? 0xFFFFFFFFu : 0u) : 0u);
      }
    }
  }
  ls_gain<NP>(c, sum, cols, g);
  planes_store<NP>(gains + (size_t)v * NP, g);
}

// flips row v's columns whose positive gain no neighbour beats; true if any
template <int NP>
__device__ __forceinline__ bool ls_flip_row(int32_t v, int32_t W, const int32_t* __restrict__ row_ptr,
                                            const uint32_t* __restrict__ col, const uint32_t* gains, uint32_t* zk) {
  uint32_t g[NP], left = 0u;
  planes_load<NP>(gains + (size_t)v * NP, g);
#pragma unroll
  for (int p = 0; p < NP; ++p) left |= g[p];
  if (!left) return false;
  const int32_t e1 = __ldg(row_ptr + v + 1);
  for (int32_t e = __ldg(row_ptr + v); e < e1 && left; e += 4) {
    uint32_t gu[4][NP];
    int32_t u[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) u[q] = (int32_t)(__ldg(col + min(e + q, e1 - 1)) & 0x7FFFFFFFu);
#pragma unroll
    for (int q = 0; q < 4; ++q) planes_load<NP>(gains + (size_t)u[q] * NP, gu[q]);
    // a repeated last entry changes nothing
#pragma unroll
    for (int q = 0; q < 4; ++q) left &= ~ls_beats<NP>(gu[q], g, u[q] < v);
  }
  if (!left) return false;
  zk[(size_t)v * W] ^= left;
  return true;
}

__device__ __forceinline__ uint32_t word_columns(int32_t B, int32_t k) {
  return B - 32 * k >= 32 ? 0xFFFFFFFFu : (1u << (B - 32 * k)) - 1u;
}

// All rounds of one word in one cluster of LS_CLUSTER CTAs (columns are
// independent of one another), so the word stops at its own optimum.  CTA i
// owns a range of rows, holds their entries in shared memory (16-bit index |
// sign, |w| in the upper half of a word with integral weights) and a copy of the word's column of z and of its positive-gain masks,
// which the owners of the rows update in all CTAs through distributed shared
// memory; a cluster barrier ends each half round.  Only gains of neighbours
// that have a positive gain in a column still open are read (L2).  Bound by
// the latency of the half rounds.  Measured, n = 5 000, degree 10, 256 columns,
// rounded vectors: 94 us; with z and all gains read through L2 275, a launch
// per half round of 32 integer gains a word 780.
constexpr int LS_CLUSTER = 8;

struct LsSmem {
  size_t z, pos, rp, ent, total;   // byte offsets
};
__host__ __device__ inline LsSmem ls_smem(int32_t n, int32_t entries, bool gen) {
  LsSmem L;
  const int32_t own = (n + LS_CLUSTER - 1) / LS_CLUSTER;
  L.z = 0;
  L.pos = L.z + (size_t)n * 4;
  L.rp = L.pos + (size_t)n * 4;
  L.ent = L.rp + (size_t)(own + 1) * 4;
  L.total = L.ent + ((size_t)entries * (gen ? 4 : 2) + 15) / 16 * 16;
  return L;
}

template <int NP, bool GEN>
__global__ void __cluster_dims__(LS_CLUSTER, 1, 1) __launch_bounds__(1024)
    k_ls_cluster(int32_t n, int32_t W, int32_t B, const int32_t* __restrict__ row_ptr,
                 const uint32_t* __restrict__ col, const int32_t* __restrict__ wint, uint32_t* zb, uint32_t* gains, int32_t max_rounds,
                 int32_t* changed, int32_t max_entries) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int32_t s_any[2][LS_CLUSTER];
  cg::cluster_group cluster = cg::this_cluster();
  const LsSmem L = ls_smem(n, max_entries, GEN);
  uint32_t* const z = reinterpret_cast<uint32_t*>(smem + L.z);
  uint32_t* const pos = reinterpret_cast<uint32_t*>(smem + L.pos);
  int32_t* const rp = reinterpret_cast<int32_t*>(smem + L.rp);
  using Entry = std::conditional_t<GEN, uint32_t, uint16_t>;
  Entry* const ent = reinterpret_cast<Entry*>(smem + L.ent);
  const int rank = (int)cluster.block_rank(), tid = threadIdx.x, nt = blockDim.x;
  const int32_t k = blockIdx.x / LS_CLUSTER, own = (n + LS_CLUSTER - 1) / LS_CLUSTER;
  const int32_t ra = min(n, rank * own), rows = min(n, ra + own) - ra;
  uint32_t* const gk = gains + (size_t)k * n * NP;
  const uint32_t cols = word_columns(B, k);
  const int32_t ebase = __ldg(row_ptr + ra);
  for (int32_t i = tid; i <= rows; i += nt) rp[i] = __ldg(row_ptr + ra + i) - ebase;
  const int32_t entries = __ldg(row_ptr + ra + rows) - ebase;
  for (int32_t i = tid; i < entries; i += nt) {
    const uint32_t c = __ldg(col + ebase + i);
    if (GEN) {
      const int32_t w = __ldg(wint + ebase + i);
      ent[i] = (Entry)((c & 0x7FFFu) | (w < 0 ? 0x8000u : 0u) | (uint32_t)abs(w) << 16);
    } else {
      ent[i] = (Entry)((c & 0x7FFFu) | (c >> 31 << 15));
    }
  }
  for (int32_t v = tid; v < n; v += nt) z[v] = zb[(size_t)v * W + k];
  // the same word of every CTA of the cluster
  auto put = [&](uint32_t* at, uint32_t x) {
#pragma unroll
    for (int q = 0; q < LS_CLUSTER; ++q) *cluster.map_shared_rank(at, q) = x;
  };
  cluster.sync();
  for (int32_t r = 0; r < max_rounds; ++r) {
    for (int32_t i = tid; i < rows; i += nt) {
      const int32_t e0 = rp[i], d = rp[i + 1] - e0;
      const uint32_t zv = z[ra + i];
      uint32_t c[NP], g[NP];
      int32_t sum = GEN ? 0 : d;
#pragma unroll
      for (int p = 0; p < NP; ++p) c[p] = 0u;
#pragma unroll 4
      for (int32_t e = 0; e < d; ++e) {
        const uint32_t u = ent[e0 + e];
        const uint32_t lost = z[u & 0x7FFFu] ^ zv ^ ((u & 0x8000u) ? 0xFFFFFFFFu : 0u);
        if (GEN) {
          sum += (int32_t)(u >> 16);
          ls_count_weight<NP>(c, lost, u >> 16);
        } else {
          ls_count<NP>(c, lost);
        }
      }
      const uint32_t any = ls_gain<NP>(c, sum, cols, g);
      put(pos + ra + i, any);
      if (any) planes_store<NP>(gk + (size_t)(ra + i) * NP, g);
    }
    cluster.sync();
    bool flipped = false;
    for (int32_t i = tid; i < rows; i += nt) {
      const int32_t v = ra + i;
      uint32_t left = pos[v];
      if (!left) continue;
      uint32_t g[NP];
      planes_load<NP>(gk + (size_t)v * NP, g);
      const int32_t e1 = rp[i + 1];
      for (int32_t e = rp[i]; e < e1 && left; e += 4) {
        uint32_t gu[4][NP];
        int32_t u[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          u[q] = ent[min(e + q, e1 - 1)] & 0x7FFF;
          if (pos[u[q]] & left) {
            planes_load<NP>(gk + (size_t)u[q] * NP, gu[q]);
          } else {
            u[q] = n;   // no open column to compare: a gain of 0, and not the lower index
#pragma unroll
            for (int p = 0; p < NP; ++p) gu[q][p] = 0u;
          }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) left &= ~ls_beats<NP>(gu[q], g, u[q] < v);
      }
      if (!left) continue;
      flipped = true;
      put(z + v, z[v] ^ left);
    }
    const int block_any = __syncthreads_or(flipped ? 1 : 0);
    if (tid < LS_CLUSTER) *cluster.map_shared_rank(&s_any[r & 1][rank], tid) = block_any;
    cluster.sync();
    int32_t sum = 0;
#pragma unroll
    for (int i = 0; i < LS_CLUSTER; ++i) sum |= s_any[r & 1][i];
    if (!sum) break;   // the same in every CTA of the cluster
    if (rank == 0 && tid == 0) changed[r + 1] = 1;
  }
  for (int32_t i = tid; i < rows; i += nt) zb[(size_t)(ra + i) * W + k] = z[ra + i];
}

// one half round of all words per launch (graphs with more rows than a cluster covers well)
template <int NP, bool GEN>
__global__ void __launch_bounds__(128) k_ls_gain_planes(int32_t n, int32_t W, int32_t B,
                                                        const int32_t* __restrict__ row_ptr,
                                                        const uint32_t* __restrict__ col,
                                                        const int32_t* __restrict__ wint, const uint32_t* zb,
                                                        uint32_t* gains, const int32_t* run) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)n * W || !*run) return;
  const int32_t v = (int32_t)(i % n), k = (int32_t)(i / n);
  ls_gain_row<NP, GEN>(v, W, row_ptr, col, wint, zb + k, word_columns(B, k), gains + (size_t)k * n * NP);
}
template <int NP>
__global__ void __launch_bounds__(128) k_ls_flip_planes(int32_t n, int32_t W, const int32_t* __restrict__ row_ptr,
                                                        const uint32_t* __restrict__ col, const uint32_t* gains,
                                                        uint32_t* zb, const int32_t* run, int32_t* next) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)n * W || !*run) return;
  const int32_t v = (int32_t)(i % n), k = (int32_t)(i / n);
  if (ls_flip_row<NP>(v, W, row_ptr, col, gains + (size_t)k * n * NP, zb + k)) *next = 1;
}

unsigned blocks_for(int64_t threads, int per) { return (unsigned)((threads + per - 1) / per); }

}  // namespace

// Bit planes of a positive gain (at most the row's sum of |w|), 0: the sums do
// not allow them and the gains are kept as integers.
static int ls_planes(const deco_graph* g) {
  const int32_t most = g->wmode == W_GENERAL ? g->max_row_abs : g->max_deg;
  if (most < 16) return 4;
  if (most < 256) return 8;
  return most < 65536 ? 16 : 0;
}

size_t local_search_words(const deco_graph* g, int32_t B) {
  const int np = ls_planes(g);
  return (size_t)g->n * ((B + 31) / 32) * (np ? np : 32);
}

template <int NP, bool GEN>
static int run_planes(const deco_graph* g, int32_t B, uint32_t* zbits, int32_t max_rounds, uint32_t* gains,
                      int32_t* changed, int64_t* kernels, cudaStream_t st) {
  const int32_t W = (B + 31) / 32, n = g->n;
  const uint32_t* col = g->wmode == W_SIGN ? g->col_sw : reinterpret_cast<const uint32_t*>(g->col_idx);
  // One cluster per word while its rows fit on chip (n of about 20 000 at degree 10), for any number of columns: the
  // launches of the other form alone cost 2 x 2.2 us a round.  us per call, cluster and launches: 1 000 nodes, 1 column
  // 131 / 426; 20 000 of degree 10, 32 columns 549 / 618, 256 columns 637 / 1 033
  int32_t entries = 0;
  const int32_t own = (n + LS_CLUSTER - 1) / LS_CLUSTER;
  for (int q = 0; q < LS_CLUSTER; ++q)
    entries = std::max(entries, g->h_row_ptr[std::min(n, (q + 1) * own)] - g->h_row_ptr[std::min(n, q * own)]);
  const size_t smem = ls_smem(n, entries, GEN).total;
  if (n <= 32768 && smem + 1024 <= (size_t)slab_max_smem()) {
    const int nt = own <= 256 ? 256 : own <= 512 ? 512 : 1024;
    DECO_CUDA_TRY(allow_smem(k_ls_cluster<NP, GEN>));
    k_ls_cluster<NP, GEN><<<(unsigned)W * LS_CLUSTER, nt, smem, st>>>(n, W, B, g->row_ptr, col, g->wint, zbits, gains, max_rounds,
                                                                 changed, entries);
    DECO_CUDA_TRY(cudaGetLastError());
    if (kernels) *kernels += 1;
    return DECO_OK;
  }
  const int64_t threads = (int64_t)n * W;
  for (int32_t r = 0; r < max_rounds; ++r) {
    k_ls_gain_planes<NP, GEN><<<blocks_for(threads, 128), 128, 0, st>>>(n, W, B, g->row_ptr, col, g->wint, zbits, gains,
                                                                        changed + r);
    k_ls_flip_planes<NP><<<blocks_for(threads, 128), 128, 0, st>>>(n, W, g->row_ptr, col, gains, zbits, changed + r,
                                                                   changed + r + 1);
  }
  DECO_CUDA_TRY(cudaGetLastError());
  if (kernels) *kernels += 2 * (int64_t)max_rounds;
  return DECO_OK;
}

template <int NP>
static int run_weights(const deco_graph* g, int32_t B, uint32_t* zbits, int32_t max_rounds, uint32_t* gains,
                       int32_t* changed, int64_t* kernels, cudaStream_t st) {
  return g->wmode == W_GENERAL ? run_planes<NP, true>(g, B, zbits, max_rounds, gains, changed, kernels, st)
                               : run_planes<NP, false>(g, B, zbits, max_rounds, gains, changed, kernels, st);
}

// The rounds of the local search on bit-packed columns (stream-ordered).
// gains: local_search_words(g, B) words of scratch; changed: max_rounds + 1
// int32 scratch, changed[r] nonzero where round r flipped (r >= 1).
int launch_local_search(const deco_graph* g, int32_t B, uint32_t* zbits, int32_t max_rounds, uint32_t* gains,
                        int32_t* changed, int64_t* kernels, cudaStream_t st) {
  const int32_t W = (B + 31) / 32;
  if (max_rounds <= 0 || g->n == 0) return DECO_OK;
  DECO_CUDA_TRY(cudaMemsetAsync(changed, 0, sizeof(int32_t) * (size_t)(max_rounds + 1), st));
  DECO_CUDA_TRY(cudaMemsetAsync(changed, 1, sizeof(int32_t), st));   // round 0 runs (any nonzero word)
  switch (ls_planes(g)) {
    case 4: return run_weights<4>(g, B, zbits, max_rounds, gains, changed, kernels, st);
    case 8: return run_weights<8>(g, B, zbits, max_rounds, gains, changed, kernels, st);
    case 16: return run_weights<16>(g, B, zbits, max_rounds, gains, changed, kernels, st);
    default: break;
  }
  const int64_t threads = (int64_t)g->n * W;
  int32_t* gi = reinterpret_cast<int32_t*>(gains);
  for (int32_t r = 0; r < max_rounds; ++r) {
    k_ls_gain<<<blocks_for(threads, 128), 128, 0, st>>>(g->n, W, g->row_ptr, g->col_idx, g->wint, zbits, gi,
                                                        changed + r);
    k_ls_flip<<<blocks_for(threads, 128), 128, 0, st>>>(g->n, W, B, g->row_ptr, g->col_idx, gi, zbits, changed + r,
                                                        changed + r + 1);
  }
  DECO_CUDA_TRY(cudaGetLastError());
  if (kernels) *kernels += 2 * (int64_t)max_rounds;
  return DECO_OK;
}

}  // namespace deco

using namespace deco;

namespace {

// Where the runs keep their sides, by the rounds of runs that each form takes
// (some ten runs share an SM before they slow each other down) and its time
// per placement: bytes 1, two bits 1.7 (weights: 1.2), a column of z 4.5 (2.7),
// 7 (4.2) once the n x B bytes leave L2, or 0.0038 (0.0024) a run where the
// memory is the limit.  ms, bytes / two bits / column: n = 20 000, degree 10,
// B = 2 048 5.2 / 5.7 / 9.3; n = 40 000, B = 4 096 31 / 25 / 48; n = 200 000,
// degree 6, B = 64 19 / 33 / 77, B = 1 024 147 / 101 / 130, B = 4 096 572 / 313
// / 299; n = 400 000 (no bytes), B = 64 66 / 155, B = 2 048 469 / 312; weights,
// n = 100 000, B = 256 36 / 22 / 49.  Columns of weighted graphs take windows of
// 8 vertices where those of 16 hold too few runs on an SM (n = 200 000, B =
// 4 096: 461 ms with 16, 346 with 8; n = 400 000, B = 1 024: 310 and 325).
struct GreedyPlan {
  int sides = GREEDY_COLUMN;
  size_t smem = 0;       // dynamic shared memory
  bool narrow = false;   // windows of 8
};

template <bool WT>
GreedyPlan greedy_plan(int32_t n, int32_t B) {
  constexpr size_t windows = 2 * sizeof(GreedyWindow<WT, 16>) + 1024;
  const size_t limit = (size_t)block_smem_limit();
  const int64_t sms = device_sm_count();
  GreedyPlan p;
  p.narrow = WT && B > sms * (int64_t)((limit + 1024) / windows);
  double least = std::max((double)n * B > 1e8 ? (WT ? 4.2 : 7.0) : (WT ? 2.7 : 4.5), (WT ? 0.0024 : 0.0038) * B);
  auto consider = [&](int sides, size_t smem, double placement) {
    if (smem + windows > limit) return;
    const int64_t runs = sms * std::min<int64_t>(10, (int64_t)((limit + 1024) / (smem + windows)));
    const double cost = placement * (double)((B + runs - 1) / runs);
    if (cost < least) { least = cost; p = GreedyPlan{sides, smem, false}; }
  };
  consider(GREEDY_BITS, ((size_t)n + 63) / 64 * 16, WT ? 1.2 : 1.7);
  consider(GREEDY_BYTES, ((size_t)n + 15) / 16 * 16, 1.0);
  return p;
}

// the placement of B runs in the order of `order`: sides in it (run-major), or in z where *columns
template <bool WT>
int launch_greedy(const deco_graph* g, int32_t B, int32_t* order, uint8_t* z, bool* columns, cudaStream_t st) {
  const GreedyPlan p = greedy_plan<WT>(g->n, B);
  auto fn = p.sides == GREEDY_BYTES  ? k_greedy<WT, GREEDY_BYTES, 16>
            : p.sides == GREEDY_BITS ? k_greedy<WT, GREEDY_BITS, 16>
            : WT && p.narrow         ? k_greedy<WT, GREEDY_COLUMN, WT ? 8 : 16>
                                     : k_greedy<WT, GREEDY_COLUMN, 16>;
  *columns = p.sides == GREEDY_COLUMN;
  if (*columns) DECO_CUDA_TRY(cudaMemsetAsync(z, 2, (size_t)g->n * B, st));
  DECO_CUDA_TRY(allow_smem(fn, 2 * sizeof(GreedyWindow<WT, 16>) + 1024));
  fn<<<(unsigned)B, 64, p.smem, st>>>(g->n, B, g->row_ptr, g->col_idx, g->wint, order, z);
  DECO_CUDA_TRY(cudaGetLastError());
  return DECO_OK;
}

}  // namespace

extern "C" int deco_greedy(const deco_graph* g, int32_t B, uint64_t seed, uint8_t* z, int64_t* cuts, void* stream) {
  clear_error();
  int rc = check_graph(g);
  if (rc) return rc;
  if (B < 1 || !z || !cuts) { set_error("need B >= 1 and device z, cuts"); return DECO_ERR_ARG; }
  if (g->n >= (1 << 30)) { set_error("n too large for the greedy orderings"); return DECO_ERR_UNSUPPORTED; }
  cudaStream_t st = as_stream(stream);
  Scratch s(st);
  int32_t* order = nullptr;
  if ((rc = s.alloc(&order, sizeof(int32_t) * (size_t)g->n * B))) return rc;
  Feistel F{};
  F.h = 1;
  while ((1ull << (2 * F.h)) < (uint64_t)g->n) ++F.h;
  F.mask = (uint32_t)((1ull << F.h) - 1);
  F.n = (uint32_t)g->n;
  F.k0 = (uint32_t)(seed & 0xFFFFFFFFu);
  F.k1 = (uint32_t)(seed >> 32);
  const int32_t n = g->n, W = (B + 31) / 32;
  uint32_t* bits = nullptr;
  if ((rc = s.alloc(&bits, sizeof(uint32_t) * (size_t)n * W))) return rc;
  const dim3 ogrid((unsigned)B, (unsigned)std::min((n + 1023) / 1024, device_sm_count()));
  if (F.h <= ORDER_MAX_H) k_orders<true><<<ogrid, 256, sizeof(uint16_t) * (4u << F.h), st>>>(F, B, order);
  else k_orders<false><<<ogrid, 256, 0, st>>>(F, B, order);
  DECO_CUDA_TRY(cudaGetLastError());
  bool columns = false;
  if ((rc = g->wint ? launch_greedy<true>(g, B, order, z, &columns, st) : launch_greedy<false>(g, B, order, z, &columns, st)))
    return rc;
  if (!columns) {
    const int64_t tiles = (int64_t)((n + 31) / 32) * W;
    k_sides_out<<<(unsigned)std::min<int64_t>((tiles + 7) / 8, (int64_t)device_sm_count() * 16), 256, 0, st>>>(
        n, B, W, reinterpret_cast<const uint8_t*>(order), z, bits);
    DECO_CUDA_TRY(cudaGetLastError());
  } else if ((rc = launch_bytes_to_bits(n, B, z, bits, st))) {
    return rc;
  }
  return launch_cut_bits(g, B, bits, cuts, st);
}

extern "C" int deco_local_search(const deco_graph* g, int32_t B, uint8_t* z, int32_t max_rounds, int64_t* cuts,
                                 int32_t* rounds, void* stream) {
  clear_error();
  int rc = check_graph(g);
  if (rc) return rc;
  if (B < 1 || !z || max_rounds < 0) { set_error("need B >= 1, device z and max_rounds >= 0"); return DECO_ERR_ARG; }
  cudaStream_t st = as_stream(stream);
  const int32_t W = (B + 31) / 32;
  Scratch s(st);
  uint32_t* bits = nullptr;
  uint32_t* gains = nullptr;
  int32_t* changed = nullptr;
  if ((rc = s.alloc(&bits, sizeof(uint32_t) * (size_t)g->n * W)) ||
      (rc = s.alloc(&gains, sizeof(uint32_t) * local_search_words(g, B))) ||
      (rc = s.alloc(&changed, sizeof(int32_t) * (size_t)(max_rounds + 1))))
    return rc;
  if (g->n > 0) {
    if ((rc = launch_bytes_to_bits(g->n, B, z, bits, st))) return rc;
    if ((rc = launch_local_search(g, B, bits, max_rounds, gains, changed, nullptr, st))) return rc;
    k_bits_to_bytes<<<blocks_for((int64_t)g->n * B, 256), 256, 0, st>>>(g->n, B, W, bits, z);
    DECO_CUDA_TRY(cudaGetLastError());
  }
  if (cuts && (rc = launch_cut_bits(g, B, bits, cuts, st))) return rc;
  if (rounds) {
    std::vector<int32_t> h((size_t)max_rounds + 1, 0);
    DECO_CUDA_TRY(cudaMemcpyAsync(h.data(), changed, sizeof(int32_t) * h.size(), cudaMemcpyDeviceToHost, st));
    DECO_CUDA_TRY(cudaStreamSynchronize(st));
    int32_t c = 0;
    for (int32_t r = 1; r <= max_rounds; ++r) c += h[r] ? 1 : 0;
    *rounds = g->n > 0 ? c : 0;
  }
  return DECO_OK;
}
