// Rounding, integer cut evaluation and argmax over starting points
// (the rounding and selection steps of Alg. 1 / Alg. 2; Eq. 5, Eq. 11, Eq. 1).
//
//  pack:   one thread per (row, 8 starting points) reads their columns as
//          16-byte vectors and writes 8 bits; blocks whose rows are not
//          16-byte aligned, and lifts above 4, take one warp per (row, 32
//          starting points) and a ballot.
//  cut:    warps take equal ranges of the stored entries, a lane per entry.
//          Without weights a lane counts its entries' words z_v xor z_u in bit
//          planes (carry-save adders); now and then the warp transposes the
//          planes, 32 x 32 bits each, and lane b adds starting point b's bits
//          with one popc a plane.  With weights the words of 32 entries are
//          transposed themselves, and lane b takes one popc per bit of |w| and
//          sign.  Entries with u > v count (each unordered edge once), in
//          integers; the block reduces and issues one 64-bit atomic per
//          starting point.  Integer sums are exact in any order.  Vectors
//          given as bytes are packed first, or read where they are (k_cut_bytes).
//  argmax: one block; lowest index among the maximal cuts.
#include <algorithm>

#include "api_util.cuh"
#include "deco_internal.cuh"

namespace deco {

int device_sm_count();

namespace {

template <int PREC>
__device__ __forceinline__ float load_y(const void* y, size_t i) {
  if (PREC == DECO_PREC_FP32) return __ldg(static_cast<const float*>(y) + i);
  return __bfloat162float(static_cast<const __nv_bfloat16*>(y)[i]);
}

template <int PREC>
__global__ void k_pack(int32_t n, int32_t B, int32_t lift, int32_t ld, int32_t W, const void* y,
                       uint32_t* zbits) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (warp >= (int64_t)n * W) return;
  const int32_t v = (int32_t)(warp / W);
  const int32_t k = (int32_t)(warp % W);
  const int32_t b = k * 32 + lane;
  bool bit = false;
  if (b < B) {
    const size_t base = (size_t)v * ld + (size_t)b * lift;
    if (lift == 1) {
      bit = load_y<PREC>(y, base) > 0.0f;               // Eq. 5: strict
    } else {
      float s = 0.0f;
      for (int i = 0; i < lift; ++i) s += load_y<PREC>(y, base + i);
      bit = s >= 0.0f;                                   // Eq. 11: non-strict
    }
  }
  const uint32_t word = __ballot_sync(0xFFFFFFFFu, bit);
  if (lane == 0) zbits[(size_t)v * W + k] = word;
}

// Byte q of row v: starting points 8q ... 8q + 7, i.e. columns 8 q LIFT ... of
// the row, 16-byte aligned (ld % 8 == 0).  A vector may reach past column C
// but not past ld; points >= B give 0.  Bound by HBM: 10^6 rows of 128 BF16
// columns in 56 us (4.8 TB/s; 64 with 64-bit divisions); a warp per word, 2
// bytes a lane, took 456.
template <int PREC, int LIFT>
__global__ void __launch_bounds__(256) k_pack_vec(int32_t n, int32_t B, int32_t ld, int32_t W, const void* y,
                                                  uint8_t* zbytes) {
  constexpr int VN = PREC == DECO_PREC_BF16 ? 8 : 4;    // values of a vector
  constexpr int NV = 8 * LIFT / VN;                     // vectors of 8 points
  const int64_t total = (int64_t)n * W * 4, step = (int64_t)gridDim.x * blockDim.x;
  const uint32_t W4 = (uint32_t)W * 4u;
  const bool small = total < (int64_t)1 << 31;          // 32-bit divisions: a 64-bit one costs more than the rounding
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += step) {
    const int32_t v = small ? (int32_t)((uint32_t)i / W4) : (int32_t)(i / W4);
    const int32_t q = (int32_t)(i - (int64_t)v * W4);
    uint32_t bits = 0;
    const int32_t c0 = 8 * q * LIFT;
    const uint4* src = reinterpret_cast<const uint4*>(static_cast<const char*>(y) +
                                                      ((size_t)v * ld + c0) * (PREC == DECO_PREC_BF16 ? 2 : 4));
    uint4 raw[NV];
#pragma unroll
    for (int h = 0; h < NV; ++h) {
      raw[h] = make_uint4(0u, 0u, 0u, 0u);
      if (c0 + h * VN < B * LIFT) raw[h] = __ldg(src + h);
    }
    float val[8 * LIFT];
#pragma unroll
    for (int h = 0; h < NV; ++h) {
      const uint32_t u[4] = {raw[h].x, raw[h].y, raw[h].z, raw[h].w};
#pragma unroll
      for (int k = 0; k < VN; ++k) {
        if (PREC == DECO_PREC_FP32) val[h * VN + k] = __uint_as_float(u[k % 4]);
        else val[h * VN + k] = (k & 1) ? bf16hi(u[k / 2]) : bf16lo(u[k / 2]);
      }
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      bool bit;
      if (LIFT == 1) {
        bit = val[k] > 0.0f;                             // Eq. 5: strict
      } else {
        float s = 0.0f;
#pragma unroll
        for (int l = 0; l < LIFT; ++l) s += val[k * LIFT + l];
        bit = s >= 0.0f;                                 // Eq. 11: non-strict
      }
      if (bit) bits |= 1u << k;
    }
    if (8 * q + 8 > B) bits &= 8 * q < B ? (1u << (B - 8 * q)) - 1u : 0u;   // points below B
    zbytes[i] = (uint8_t)bits;
  }
}

// 0/1 bytes (n x B, any nonzero byte counts as 1) to bits: a warp per (row, word)
__global__ void k_bytes_to_bits(int32_t n, int32_t B, int32_t W, const uint8_t* z, uint32_t* bits) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < (int64_t)n * W; i += warps) {
    const int32_t v = (int32_t)(i / W), b = (int32_t)(i % W) * 32 + lane;
    const uint32_t word = __ballot_sync(0xFFFFFFFFu, b < B && z[(size_t)v * B + b] != 0);
    if (lane == 0) bits[i] = word;
  }
}

// lane b of the result holds, at bit e, bit b of lane e's x
__device__ __forceinline__ uint32_t transpose32(uint32_t x, int lane) {
#pragma unroll
  for (int s = 16; s >= 1; s >>= 1) {
    const uint32_t m = s == 16 ? 0x0000FFFFu : s == 8 ? 0x00FF00FFu : s == 4 ? 0x0F0F0F0Fu : s == 2 ? 0x33333333u
                                                                                                   : 0x55555555u;
    const uint32_t y = __shfl_xor_sync(0xFFFFFFFFu, x, s);
    x = (lane & s) ? ((x & ~m) | ((y >> s) & m)) : ((x & m) | ((y & m) << s));
  }
  return x;
}

constexpr int CUT_BLOCK = 256;
constexpr int cut_batches(bool wt) { return wt ? 2 : 4; }   // batches of 32 entries in flight per warp
constexpr int CUT_PLANES = 5;                               // a lane's counts below 32

// Cuts of the starting points of V words (word group blockIdx.y) over the
// rows of graph blockIdx.z (goff: first rows; null: all n rows), added to
// cuts[graph B + b].  Bound by the latency of the gathered words and by issue
// slots: 10^6 nodes, degree 10, 128 starting points in 69 us; every entry's
// words transposed 109, a warp per row that walked its neighbours 1 059.
template <int V, bool WT>
__global__ void __launch_bounds__(CUT_BLOCK, 4) k_cut(int32_t n, int32_t B, int32_t W, const int32_t* __restrict__ row_ptr,
                                                   const int32_t* __restrict__ col_idx, const int32_t* __restrict__ wint,
                                                   int wbits, const uint32_t* __restrict__ zbits,
                                                   const int32_t* __restrict__ goff, int64_t* cuts) {
  __shared__ long long part[CUT_BLOCK / 32][32 * V];
  constexpr int CUT_U = cut_batches(WT);
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int32_t k0 = blockIdx.y * V, g = blockIdx.z;
  const int32_t ra = goff ? __ldg(goff + g) : 0, rb = goff ? __ldg(goff + g + 1) : n;
  const int64_t Ea = __ldg(row_ptr + ra), Eb = __ldg(row_ptr + rb);
  const int64_t warps = (int64_t)gridDim.x * (CUT_BLOCK / 32);
  const int64_t per = ((Eb - Ea + warps - 1) / warps + 31) / 32 * 32;
  int64_t e = Ea + ((int64_t)blockIdx.x * (CUT_BLOCK / 32) + wib) * per;
  const int64_t E1 = min(Eb, e + per);
  long long acc[V];
#pragma unroll
  for (int j = 0; j < V; ++j) acc[j] = 0;
  uint32_t plane[V][CUT_PLANES] = {};
  int held = 0;            // entries a lane may have counted since the planes were last emptied
  auto empty_planes = [&]() {
#pragma unroll
    for (int j = 0; j < V; ++j)
#pragma unroll
      for (int p = 0; p < CUT_PLANES; ++p) {
        acc[j] += (long long)__popc(transpose32(plane[j][p], lane)) << p;
        plane[j][p] = 0u;
      }
    held = 0;
  };
  if (e < E1) {
    // the row that holds entry e: row_ptr[r] <= e < row_ptr[r + 1]
    int32_t lo = ra, hi = rb;
    while (hi - lo > 1) {
      const int32_t step = (hi - lo + 31) / 32;
      const int64_t p = lo + (int64_t)(lane + 1) * step;
      const int cnt = __popc(__ballot_sync(0xFFFFFFFFu, p < hi && __ldg(row_ptr + p) <= e));
      lo += cnt * step;
      hi = min(hi, lo + step);
    }
    // window of 32 rows: lane i holds the end of row r + i
    int32_t r = lo;
    int32_t end = __ldg(row_ptr + min(r + lane + 1, rb));
    while (e < E1) {
      const int32_t last = __shfl_sync(0xFFFFFFFFu, end, 31);
      if (last <= e) {
        r += 32;
        end = __ldg(row_ptr + min(r + lane + 1, rb));
        continue;
      }
      const int64_t lim = min(E1, (int64_t)last);
      for (; e < lim; e += 32 * CUT_U) {
        int32_t row[CUT_U], u[CUT_U], w[CUT_U];
#pragma unroll
        for (int q = 0; q < CUT_U; ++q) {
          const int64_t x = e + 32 * q + lane;
          u[q] = -1;
          w[q] = 1;
          if (x < lim) {
            u[q] = __ldg(col_idx + x);
            if (WT) w[q] = __ldg(wint + x);
          }
        }
#pragma unroll
        for (int q = 0; q < CUT_U; ++q) {
          const int64_t x = e + 32 * q + lane;
          int pos = 0;   // rows of the window that end at or before entry x
#pragma unroll
          for (int s = 16; s >= 1; s >>= 1)
            if (__shfl_sync(0xFFFFFFFFu, end, pos + s - 1) <= x) pos += s;
          row[q] = r + pos;
        }
        uint32_t d[CUT_U][V];
#pragma unroll
        for (int q = 0; q < CUT_U; ++q) {
#pragma unroll
          for (int j = 0; j < V; ++j) d[q][j] = 0u;
          if (u[q] > row[q]) {
            const uint32_t* zu = zbits + (size_t)u[q] * W + k0;
            const uint32_t* zv = zbits + (size_t)row[q] * W + k0;
            if (V == 4) {
              const uint4 a = __ldg(reinterpret_cast<const uint4*>(zu)), b = __ldg(reinterpret_cast<const uint4*>(zv));
              d[q][0] = a.x ^ b.x; d[q][1 % V] = a.y ^ b.y; d[q][2 % V] = a.z ^ b.z; d[q][3 % V] = a.w ^ b.w;
            } else if (V == 2) {
              const uint2 a = __ldg(reinterpret_cast<const uint2*>(zu)), b = __ldg(reinterpret_cast<const uint2*>(zv));
              d[q][0] = a.x ^ b.x; d[q][1 % V] = a.y ^ b.y;
            } else {
              d[q][0] = __ldg(zu) ^ __ldg(zv);
            }
          }
        }
        if constexpr (!WT) {
#pragma unroll
          for (int j = 0; j < V; ++j) {
            uint32_t* const c = plane[j];
            const uint32_t d0 = d[0][j], d1 = d[1][j], d2 = d[2 % CUT_U][j], d3 = d[3 % CUT_U][j];
            const uint32_t t0 = (c[0] & d0) | (c[0] & d1) | (d0 & d1);
            c[0] ^= d0 ^ d1;
            const uint32_t t1 = (c[0] & d2) | (c[0] & d3) | (d2 & d3);
            c[0] ^= d2 ^ d3;
            uint32_t carry = (c[1] & t0) | (c[1] & t1) | (t0 & t1);
            c[1] ^= t0 ^ t1;
#pragma unroll
            for (int p = 2; p < CUT_PLANES; ++p) {
              const uint32_t t = c[p] & carry;
              c[p] ^= carry;
              carry = t;
            }
          }
          held += CUT_U;
          if (held + CUT_U >= 1 << CUT_PLANES) empty_planes();
        } else {
#pragma unroll
          for (int q = 0; q < CUT_U; ++q) {
#pragma unroll
            for (int j = 0; j < V; ++j) d[q][j] = transpose32(d[q][j], lane);
            for (int h = 0; h < wbits; ++h) {
              const uint32_t pos = __ballot_sync(0xFFFFFFFFu, w[q] > 0 && ((w[q] >> h) & 1));
              const uint32_t neg = __ballot_sync(0xFFFFFFFFu, w[q] < 0 && ((-w[q] >> h) & 1));
#pragma unroll
              for (int j = 0; j < V; ++j)
                acc[j] += (long long)(__popc(d[q][j] & pos) - __popc(d[q][j] & neg)) << h;
            }
          }
        }
      }
      e = lim;
    }
    if (!WT && held) empty_planes();
  }
#pragma unroll
  for (int j = 0; j < V; ++j) part[wib][32 * j + lane] = acc[j];
  __syncthreads();
  for (int x = threadIdx.x; x < 32 * V; x += CUT_BLOCK) {
    long long s = 0;
    for (int i = 0; i < CUT_BLOCK / 32; ++i) s += part[i][x];
    const int32_t b = 32 * k0 + x;
    if (b < B && s != 0)
      atomicAdd(reinterpret_cast<unsigned long long*>(cuts + (size_t)g * B + b), (unsigned long long)s);
  }
}

// Cuts of byte columns read where they are: a warp per row, 2^lb lanes over the
// columns of group k0 + blockIdx.y (of 32) times 32 / 2^lb over the row's entries.
// No scratch memory: for few vectors or small graphs, where packing them first
// (an allocation, a launch) costs more than it saves, and where none is to be had.
template <bool WT>
__global__ void __launch_bounds__(CUT_BLOCK) k_cut_bytes(int32_t n, int32_t B, int lb, int32_t k0, const int32_t* __restrict__ row_ptr,
                                                         const int32_t* __restrict__ col_idx,
                                                         const int32_t* __restrict__ wint, const uint8_t* __restrict__ z,
                                                         int64_t* cuts) {
  __shared__ long long part[CUT_BLOCK / 32][32];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int32_t b = 32 * (k0 + (int32_t)blockIdx.y) + (lane & ((1 << lb) - 1));
  const int slots = 32 >> lb;
  const int64_t warps = (int64_t)gridDim.x * (CUT_BLOCK / 32);
  long long acc = 0;
  if (b < B) {
    for (int64_t v = (int64_t)blockIdx.x * (CUT_BLOCK / 32) + wib; v < n; v += warps) {
      const int32_t e1 = __ldg(row_ptr + v + 1);
      const bool zv = __ldg(z + (size_t)v * B + b) != 0;
      int32_t sum = 0;   // |sum| <= the row's sum of |w| <= 2^24
#pragma unroll 4
      for (int32_t e = __ldg(row_ptr + v) + (lane >> lb); e < e1; e += slots) {
        const int32_t u = __ldg(col_idx + e);
        if (u > v && (__ldg(z + (size_t)u * B + b) != 0) != zv) sum += WT ? __ldg(wint + e) : 1;
      }
      acc += sum;
    }
  }
  for (int s = 16; s >= 1 << lb; s >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, s);
  part[wib][lane] = acc;
  __syncthreads();
  if (threadIdx.x < (1 << lb) && b < B) {
    long long s = 0;
    for (int i = 0; i < CUT_BLOCK / 32; ++i) s += part[i][threadIdx.x];
    if (s != 0) atomicAdd(reinterpret_cast<unsigned long long*>(cuts + b), (unsigned long long)s);
  }
}

__global__ void k_argmax(int32_t B, const int64_t* cuts, int32_t* best) {
  __shared__ long long sv[1024];
  __shared__ int32_t si[1024];
  long long bv = LLONG_MIN;
  int32_t bi = INT32_MAX;
  for (int32_t b = threadIdx.x; b < B; b += blockDim.x) {
    long long c = cuts[b];
    if (c > bv) { bv = c; bi = b; }   // ascending b per thread: first max kept
  }
  sv[threadIdx.x] = bv;
  si[threadIdx.x] = bi;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      long long ov = sv[threadIdx.x + s];
      int32_t oi = si[threadIdx.x + s];
      if (ov > sv[threadIdx.x] || (ov == sv[threadIdx.x] && oi < si[threadIdx.x])) {
        sv[threadIdx.x] = ov;
        si[threadIdx.x] = oi;
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) *best = si[0];
}

// Record update: the evaluation's best becomes the global best if it is the
// first evaluation of the solve or strictly larger.
__global__ void k_record(int32_t phase, int32_t first, const int64_t* cuts, const int32_t* best_idx,
                         BestRecord* rec) {
  const int32_t b = *best_idx;
  const long long c = cuts[b];
  if (first || c > rec->cut) {
    rec->cut = c;
    rec->init = b;
    rec->phase = phase;
    rec->improved = 1;
  } else {
    rec->improved = 0;
  }
}

__global__ void k_extract(int32_t n, int32_t W, const uint32_t* zbits, const int32_t* best_idx,
                          const BestRecord* rec, uint8_t* phase_best_z, uint8_t* best_z) {
  const int32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  const int32_t b = *best_idx;
  const uint8_t z = (uint8_t)((zbits[(size_t)v * W + (b >> 5)] >> (b & 31)) & 1u);
  if (phase_best_z) phase_best_z[v] = z;
  if (rec->improved && best_z) best_z[v] = z;
}

template <int V>
void launch_cut_v(const deco_graph* g, int32_t B, int32_t W, const uint32_t* zbits, const int32_t* goff, int32_t graphs,
                  int64_t* cuts, cudaStream_t st) {
  // enough warps to keep every SM's slots filled, at least 64 entries each
  const int groups = W / V;
  const int64_t want = (g->nnz / graphs + CUT_BLOCK * 2 - 1) / (CUT_BLOCK * 2);
  const int64_t cap = std::max<int64_t>(1, (int64_t)device_sm_count() * 8 / ((int64_t)groups * graphs));
  const dim3 grid((unsigned)std::max<int64_t>(1, std::min(want, cap)), (unsigned)groups, (unsigned)graphs);
  int wbits = 1;
  while (wbits < 31 && (g->max_abs_w >> wbits)) ++wbits;
  if (g->wint)
    k_cut<V, true><<<grid, CUT_BLOCK, 0, st>>>(g->n, B, W, g->row_ptr, g->col_idx, g->wint, wbits, zbits, goff, cuts);
  else
    k_cut<V, false><<<grid, CUT_BLOCK, 0, st>>>(g->n, B, W, g->row_ptr, g->col_idx, nullptr, 1, zbits, goff, cuts);
}

template <int PREC, int LIFT>
void launch_pack_vec(const deco_graph* g, int32_t B, int32_t ld, int32_t W, const void* y, uint32_t* zbits,
                     cudaStream_t st) {
  const int64_t blocks = ((int64_t)g->n * W * 4 + 255) / 256;
  k_pack_vec<PREC, LIFT><<<(unsigned)std::min<int64_t>(blocks, (int64_t)device_sm_count() * 64), 256, 0, st>>>(
      g->n, B, ld, W, y, reinterpret_cast<uint8_t*>(zbits));
}

}  // namespace

int launch_pack(const deco_graph* g, int32_t B, int32_t lift, int32_t ld, int precision,
                const void* y, uint32_t* zbits, cudaStream_t st) {
  const int32_t W = (B + 31) / 32;
  if (lift <= 4 && ld % 8 == 0 && reinterpret_cast<uintptr_t>(y) % 16 == 0) {
    if (precision == DECO_PREC_BF16) {
      if (lift == 1) launch_pack_vec<DECO_PREC_BF16, 1>(g, B, ld, W, y, zbits, st);
      else if (lift == 2) launch_pack_vec<DECO_PREC_BF16, 2>(g, B, ld, W, y, zbits, st);
      else if (lift == 3) launch_pack_vec<DECO_PREC_BF16, 3>(g, B, ld, W, y, zbits, st);
      else launch_pack_vec<DECO_PREC_BF16, 4>(g, B, ld, W, y, zbits, st);
    } else {
      if (lift == 1) launch_pack_vec<DECO_PREC_FP32, 1>(g, B, ld, W, y, zbits, st);
      else if (lift == 2) launch_pack_vec<DECO_PREC_FP32, 2>(g, B, ld, W, y, zbits, st);
      else if (lift == 3) launch_pack_vec<DECO_PREC_FP32, 3>(g, B, ld, W, y, zbits, st);
      else launch_pack_vec<DECO_PREC_FP32, 4>(g, B, ld, W, y, zbits, st);
    }
    DECO_CUDA_TRY(cudaGetLastError());
    return DECO_OK;
  }
  const int64_t threads = (int64_t)g->n * W * 32;
  const int block = 256;
  const unsigned grid = (unsigned)((threads + block - 1) / block);
  if (precision == DECO_PREC_BF16) k_pack<DECO_PREC_BF16><<<grid, block, 0, st>>>(g->n, B, lift, ld, W, y, zbits);
  else k_pack<DECO_PREC_FP32><<<grid, block, 0, st>>>(g->n, B, lift, ld, W, y, zbits);
  DECO_CUDA_TRY(cudaGetLastError());
  return DECO_OK;
}

int launch_cut_graphs(const deco_graph* g, int32_t B, const uint32_t* zbits, const int32_t* goff, int32_t graphs,
                      int64_t* cuts, cudaStream_t st) {
  const int32_t W = (B + 31) / 32;
  DECO_CUDA_TRY(cudaMemsetAsync(cuts, 0, sizeof(int64_t) * (size_t)B * graphs, st));
  // the widest vector of words that every row's words are aligned to
  const uintptr_t at = reinterpret_cast<uintptr_t>(zbits);
  for (int32_t g0 = 0; g0 < graphs; g0 += 65535) {   // grid limit
    const int32_t gc = std::min(graphs - g0, 65535);
    const int32_t* go = goff ? goff + g0 : nullptr;
    int64_t* c = cuts + (size_t)g0 * B;
    if (W % 4 == 0 && at % 16 == 0) launch_cut_v<4>(g, B, W, zbits, go, gc, c, st);
    else if (W % 2 == 0 && at % 8 == 0) launch_cut_v<2>(g, B, W, zbits, go, gc, c, st);
    else launch_cut_v<1>(g, B, W, zbits, go, gc, c, st);
    DECO_CUDA_TRY(cudaGetLastError());
  }
  return DECO_OK;
}

int launch_cut_bits(const deco_graph* g, int32_t B, const uint32_t* zbits, int64_t* cuts,
                    cudaStream_t st) {
  return launch_cut_graphs(g, B, zbits, nullptr, 1, cuts, st);
}

int launch_bytes_to_bits(int32_t n, int32_t B, const uint8_t* z, uint32_t* bits, cudaStream_t st) {
  const int32_t W = (B + 31) / 32;
  const int64_t blocks = ((int64_t)n * W + 7) / 8;
  k_bytes_to_bits<<<(unsigned)std::min<int64_t>(blocks, (int64_t)device_sm_count() * 64), 256, 0, st>>>(n, B, W, z,
                                                                                                       bits);
  DECO_CUDA_TRY(cudaGetLastError());
  return DECO_OK;
}

static int launch_cut_bytes(const deco_graph* g, int32_t B, const uint8_t* z, int64_t* cuts, cudaStream_t st) {
  const int32_t W = (B + 31) / 32;
  int lb = 0;
  while ((1 << lb) < std::min(B, 32)) ++lb;
  DECO_CUDA_TRY(cudaMemsetAsync(cuts, 0, sizeof(int64_t) * (size_t)B, st));
  const int64_t rows = ((int64_t)g->n + CUT_BLOCK / 32 - 1) / (CUT_BLOCK / 32), sms = device_sm_count();
  for (int32_t k0 = 0; k0 < W; k0 += 65535) {   // grid limit
    const dim3 grid((unsigned)std::min(rows, std::max(sms, sms * 8 / W)), (unsigned)std::min(W - k0, 65535));
    if (g->wint) k_cut_bytes<true><<<grid, CUT_BLOCK, 0, st>>>(g->n, B, lb, k0, g->row_ptr, g->col_idx, g->wint, z, cuts);
    else k_cut_bytes<false><<<grid, CUT_BLOCK, 0, st>>>(g->n, B, lb, k0, g->row_ptr, g->col_idx, nullptr, z, cuts);
    DECO_CUDA_TRY(cudaGetLastError());
  }
  return DECO_OK;
}

// Packed where that is faster, the scratch for it is there and the stream is
// not capturing (the caller's graph then holds no memory of ours).  us a call,
// packed and as they are: n = 100, degree 10, B = 1 31 / 19, B = 256 31 / 21;
// n = 5 000, degree 10, B = 16 31 / 21, B = 256 40 / 34; n = 3 000, degree 300,
// B = 4 37 / 30, B = 16 37 / 46; n = 20 000, degree 60, B = 4 39 / 27, B = 33
// 45 / 87; n = 10^6, degree 8, B = 1 122 / 97, B = 8 121 / 139.
int cut_bytes(const deco_graph* g, int32_t B, const uint8_t* z, int64_t* cuts, cudaStream_t st) {
  if (g->nnz * B <= (B <= 16 ? 6000000 : 1000000)) return launch_cut_bytes(g, B, z, cuts, st);
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  DECO_CUDA_TRY(cudaStreamIsCapturing(st, &capture));
  if (capture != cudaStreamCaptureStatusNone) return launch_cut_bytes(g, B, z, cuts, st);
  Scratch s(st);
  uint32_t* bits = nullptr;
  int rc = s.alloc(&bits, sizeof(uint32_t) * (size_t)g->n * ((B + 31) / 32));
  if (rc == DECO_ERR_OOM) {
    clear_error();
    return launch_cut_bytes(g, B, z, cuts, st);
  }
  if (rc || (rc = launch_bytes_to_bits(g->n, B, z, bits, st))) return rc;
  return launch_cut_bits(g, B, bits, cuts, st);
}

int launch_argmax(int32_t B, const int64_t* cuts, int32_t* best, cudaStream_t st) {
  k_argmax<<<1, 1024, 0, st>>>(B, cuts, best);
  DECO_CUDA_TRY(cudaGetLastError());
  return DECO_OK;
}

int launch_phase_finish(const deco_graph* g, int32_t B, int32_t phase, bool first, const int64_t* cuts,
                        const uint32_t* zbits, int32_t* best_idx, BestRecord* rec,
                        uint8_t* phase_best_z, uint8_t* best_z, cudaStream_t st) {
  int rc = launch_argmax(B, cuts, best_idx, st);
  if (rc) return rc;
  k_record<<<1, 1, 0, st>>>(phase, first ? 1 : 0, cuts, best_idx, rec);
  DECO_CUDA_TRY(cudaGetLastError());
  const int32_t W = (B + 31) / 32;
  k_extract<<<(g->n + 255) / 256, 256, 0, st>>>(g->n, W, zbits, best_idx, rec, phase_best_z, best_z);
  DECO_CUDA_TRY(cudaGetLastError());
  return DECO_OK;
}

}  // namespace deco
