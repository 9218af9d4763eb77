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
#include <algorithm>

#include "api_util.cuh"
#include "deco_internal.cuh"
#include "slab.cuh"

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

// order[b n + k] = pi_b(k).  A thread walks one item after another, so that a
// warp is not held by its longest walk: 5 000 x 256 items 133 us, one item per
// thread 129.
__global__ void k_orders(Feistel F, int32_t B, int32_t* order) {
  const int64_t total = (int64_t)F.n * B, step = (int64_t)gridDim.x * blockDim.x;
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) return;
  uint32_t b = (uint32_t)(i / F.n), x = (uint32_t)(i % F.n);
  for (;;) {
    // a cycle of the bijection on [0, 4^h) passes through [0, n): every walk ends
    x = F.net(x, b);
    if (x >= F.n) continue;
    order[i] = (int32_t)x;
    i += step;
    if (i >= total) return;
    b = (uint32_t)(i / F.n);
    x = (uint32_t)(i % F.n);
  }
}

// One run (one warp, one block) places its vertices in order.  Bound by the
// chain of n dependent placements; everything that does not depend on the
// sides is loaded ahead of it: the orders and row bounds a window of 32
// vertices ahead (one per lane), the first 64 neighbours GREEDY_AHEAD
// vertices ahead.  SMEM: the sides (2: not placed) live in shared memory, a
// byte per vertex, and a placement is a shared load, a warp reduction and a
// shared store; at the end they go to the run's part of `order`, which it has
// consumed (4 n bytes of stride).  Else (a graph whose sides do not fit) the
// sides are column b of z, in global memory.  Measured, n = 5 000, degree 10,
// 256 runs: 1.07 ms; with the whole chain of loads in each placement 4.28.
constexpr int GREEDY_AHEAD = 8;

template <bool WT, bool SMEM>
__global__ void __launch_bounds__(32) k_greedy(int32_t n, int32_t B, const int32_t* __restrict__ row_ptr,
                                               const int32_t* __restrict__ col_idx, const int32_t* __restrict__ wint,
                                               int32_t* order, uint8_t* z) {
  extern __shared__ __align__(16) uint8_t sides[];
  const int lane = threadIdx.x;
  const int32_t b = blockIdx.x;
  int32_t* const ord = order + (size_t)b * n;
  if (SMEM) {
    for (int i = lane; i < (n + 3) / 4; i += 32) reinterpret_cast<uint32_t*>(sides)[i] = 0x02020202u;
    __syncwarp();
  }
  auto side = [&](int32_t u) -> int { return SMEM ? sides[u] : z[(size_t)u * B + b]; };
  // w of the entry if its vertex is in S-bar (placing v in S cuts it), -w if in S, 0 if not placed
  auto vote = [&](int32_t u, int32_t w) -> int32_t {
    const int s = u >= 0 ? side(u) : 2;
    return s == 0 ? w : s == 1 ? -w : 0;
  };
  struct Ahead { int32_t u[2], w[2]; };
  Ahead q[GREEDY_AHEAD];
  auto fetch = [&](int32_t e0, int32_t d, Ahead& a) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      a.u[h] = -1;
      a.w[h] = 1;
      if (32 * h + lane < d) {
        a.u[h] = __ldg(col_idx + e0 + 32 * h + lane);
        if (WT) a.w[h] = __ldg(wint + e0 + 32 * h + lane);
      }
    }
  };
  // window of 32 vertices, one per lane: vertex, first entry, entries (0 past n)
  int32_t v = lane < n ? ord[lane] : -1, vn = -1;
  int32_t e0 = v >= 0 ? __ldg(row_ptr + v) : 0, d = v >= 0 ? __ldg(row_ptr + v + 1) - e0 : 0, e0n = 0, dn = 0;
#pragma unroll
  for (int i = 0; i < GREEDY_AHEAD; ++i)
    fetch(__shfl_sync(0xFFFFFFFFu, e0, i), __shfl_sync(0xFFFFFFFFu, d, i), q[i]);
  for (int32_t k0 = 0; k0 < n; k0 += 32) {
    vn = k0 + 32 + lane < n ? ord[k0 + 32 + lane] : -1;
#pragma unroll 1
    for (int j0 = 0; j0 < 32; j0 += GREEDY_AHEAD) {
      if (k0 + j0 >= n) break;
      if (j0 == GREEDY_AHEAD) {
        e0n = vn >= 0 ? __ldg(row_ptr + vn) : 0;
        dn = vn >= 0 ? __ldg(row_ptr + vn + 1) - e0n : 0;
      }
#pragma unroll
      for (int i = 0; i < GREEDY_AHEAD; ++i) {
        const int j = j0 + i;
        if (k0 + j < n) {
          const int32_t vv = __shfl_sync(0xFFFFFFFFu, v, j), dd = __shfl_sync(0xFFFFFFFFu, d, j);
          int32_t t = vote(q[i].u[0], q[i].w[0]);
          if (dd > 32) t += vote(q[i].u[1], q[i].w[1]);
          if (dd > 64) {
            const int32_t ee = __shfl_sync(0xFFFFFFFFu, e0, j);
            for (int32_t x = 64 + lane; x < dd; x += 32)
              t += vote(__ldg(col_idx + ee + x), WT ? __ldg(wint + ee + x) : 1);
          }
          // |sum| <= sum of the row's |w| <= 2^24 (checked when the graph is created)
          const int32_t sum = __reduce_add_sync(0xFFFFFFFFu, t);
          if (lane == 0) {
            if (SMEM) sides[vv] = sum >= 0 ? 1 : 0;
            else z[(size_t)vv * B + b] = sum >= 0 ? 1 : 0;
          }
          __syncwarp();   // the next vertices read this side
        }
        // vertex j + GREEDY_AHEAD: of this window, or of the next
        const int ja = j + GREEDY_AHEAD;
        if (ja < 32) fetch(__shfl_sync(0xFFFFFFFFu, e0, ja), __shfl_sync(0xFFFFFFFFu, d, ja), q[i]);
        else fetch(__shfl_sync(0xFFFFFFFFu, e0n, ja - 32), __shfl_sync(0xFFFFFFFFu, dn, ja - 32), q[i]);
      }
    }
    v = vn;
    e0 = e0n;
    d = dn;
  }
  if (SMEM) {
    uint8_t* out = reinterpret_cast<uint8_t*>(ord);
    for (int i = lane; i < n; i += 32) out[i] = sides[i];
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

unsigned blocks_for(int64_t threads, int per) { return (unsigned)((threads + per - 1) / per); }

}  // namespace

// The rounds of the local search on bit-packed columns (stream-ordered).
// gains: n x 32W int32 scratch; changed: max_rounds + 1 int32 scratch.
int launch_local_search(const deco_graph* g, int32_t B, uint32_t* zbits, int32_t max_rounds, int32_t* gains,
                        int32_t* changed, cudaStream_t st) {
  const int32_t W = (B + 31) / 32;
  if (max_rounds <= 0 || g->n == 0) return DECO_OK;
  DECO_CUDA_TRY(cudaMemsetAsync(changed, 0, sizeof(int32_t) * (size_t)(max_rounds + 1), st));
  DECO_CUDA_TRY(cudaMemsetAsync(changed, 1, sizeof(int32_t), st));   // round 0 runs (any nonzero word)
  const int64_t threads = (int64_t)g->n * W;
  for (int32_t r = 0; r < max_rounds; ++r) {
    k_ls_gain<<<blocks_for(threads, 128), 128, 0, st>>>(g->n, W, g->row_ptr, g->col_idx, g->wint, zbits, gains,
                                                        changed + r);
    k_ls_flip<<<blocks_for(threads, 128), 128, 0, st>>>(g->n, W, B, g->row_ptr, g->col_idx, gains, zbits,
                                                        changed + r, changed + r + 1);
  }
  DECO_CUDA_TRY(cudaGetLastError());
  return DECO_OK;
}

}  // namespace deco

using namespace deco;

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
  const int64_t items = (int64_t)n * B;
  k_orders<<<(unsigned)std::min<int64_t>((items + 255) / 256, (int64_t)device_sm_count() * 8), 256, 0, st>>>(F, B,
                                                                                                            order);
  DECO_CUDA_TRY(cudaGetLastError());
  const size_t smem = ((size_t)n + 15) / 16 * 16;
  const bool fits = smem <= (size_t)slab_max_smem();
  auto fn = g->wint ? (fits ? k_greedy<true, true> : k_greedy<true, false>)
                    : (fits ? k_greedy<false, true> : k_greedy<false, false>);
  if (fits) {
    if (smem > 48 * 1024)
      DECO_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  } else {
    DECO_CUDA_TRY(cudaMemsetAsync(z, 2, (size_t)n * B, st));
  }
  fn<<<(unsigned)B, 32, fits ? smem : 0, st>>>(n, B, g->row_ptr, g->col_idx, g->wint, order, z);
  DECO_CUDA_TRY(cudaGetLastError());
  if (fits) {
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
  int32_t* gains = nullptr;
  int32_t* changed = nullptr;
  if ((rc = s.alloc(&bits, sizeof(uint32_t) * (size_t)g->n * W)) ||
      (rc = s.alloc(&gains, sizeof(int32_t) * (size_t)g->n * 32 * W)) ||
      (rc = s.alloc(&changed, sizeof(int32_t) * (size_t)(max_rounds + 1))))
    return rc;
  if (g->n > 0) {
    if ((rc = launch_bytes_to_bits(g->n, B, z, bits, st))) return rc;
    if ((rc = launch_local_search(g, B, bits, max_rounds, gains, changed, st))) return rc;
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
