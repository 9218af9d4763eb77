// Persistent on-chip PGA kernel, row-vector form: all T steps of a phase in
// one launch, one CTA per (graph, narrow column slab), nothing exchanged
// between CTAs.
//
// A slab is LPR 16-byte vectors of every row (LPR = 1, 2, 4 or 8: 4 ... 32
// FP32 or 8 ... 64 BF16 columns).  The CTA keeps two replicas of it in shared
// memory and reads one while it writes the other, so a step is one pass and
// one __syncthreads: no staging area, no cluster, no trip through L2 (k_slab,
// slab.cu, whose 128-byte slabs read without bank conflicts but hold a graph
// only across a cluster of CTAs and exchange every new row).  A group of LPR
// lanes owns a row, so a warp advances 32 / LPR rows at once and one 16-byte
// shared load serves an entry of each.  Rows are sorted by their entry counts,
// which makes the rows of a warp equally long; entries past a row's count read
// a row of zeros, which leaves the sum as it is (a sum that starts at +0 never
// becomes -0).  Per column the operations and their order are k_slab's and
// k_step_global's: the iterates are bit-identical.
//
// Bound by shared-memory wavefronts: rows of 128 / 64 / 32 / 16 bytes at
// random positions cost about 1 / 1.5 / 2.1 / 2.6 times the bytes' wavefronts
// in bank conflicts.  So it is the better form where a graph's rows are short
// or its starts few (latency and exchange dominate k_slab there); plan_phase
// compares both estimates.  Measured per step:
//   graph                       C     precision   k_slab   here (LPR)
//   ER(100, 0.1)                64    FP32        1.58     0.59 (1)
//   ER(500), degree 12          1024  FP32        7.7      2.3 (2)
//   40 x 20 torus, +-1          1024  BF16        6.7      1.57 (1)
//   ER(800, 0.06)               1024  FP32        9.2      11.1 (2): k_slab stays
//   ER(800, 0.06)               1024  BF16        15.0     7.7 (1)
#include <algorithm>
#include <cstring>
#include <numeric>
#include <vector>

#include "rows.cuh"
#include "slab.cuh"

namespace deco {
namespace {

__host__ __device__ inline size_t up16(size_t x) { return (x + 15) & ~(size_t)15; }

__device__ __forceinline__ uint32_t lds_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint4 lds128(uint32_t a) {
  uint4 q;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(q.x), "=r"(q.y), "=r"(q.z), "=r"(q.w) : "r"(a));
  return q;
}

template <int N>
__device__ __forceinline__ void load_f32(float (&v)[N], const float* p) {
#pragma unroll
  for (int h = 0; h < N; h += 4) {
    const float4 q = *reinterpret_cast<const float4*>(p + h);
    v[h] = q.x; v[h + 1] = q.y; v[h + 2] = q.z; v[h + 3] = q.w;
  }
}
template <int N>
__device__ __forceinline__ void store_f32(float* p, const float (&v)[N]) {
#pragma unroll
  for (int h = 0; h < N; h += 4) *reinterpret_cast<float4*>(p + h) = make_float4(v[h], v[h + 1], v[h + 2], v[h + 3]);
}

// acc += +-y or w y for the values of one 16-byte vector
template <int PREC, int SIGN, bool GEN>
__device__ __forceinline__ void add_vec(float* acc, uint4 q, float w) {
  if (PREC == DECO_PREC_FP32) {
    const float y[4] = {__uint_as_float(q.x), __uint_as_float(q.y), __uint_as_float(q.z), __uint_as_float(q.w)};
#pragma unroll
    for (int h = 0; h < 4; ++h) acc[h] = GEN ? fmaf(w, y[h], acc[h]) : SIGN > 0 ? acc[h] + y[h] : acc[h] - y[h];
  } else {
    const uint32_t flip = !GEN && SIGN < 0 ? 0x80008000u : 0u;
    const uint32_t u[4] = {q.x ^ flip, q.y ^ flip, q.z ^ flip, q.w ^ flip};
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      if (GEN) {
        acc[2 * h] = fmaf(w, bf16lo(u[h]), acc[2 * h]);
        acc[2 * h + 1] = fmaf(w, bf16hi(u[h]), acc[2 * h + 1]);
      } else {
        // the mixed-precision add: the 16-bit value widened exactly, one rounding
        asm("{\n .reg .b16 lo, hi;\n mov.b32 {lo, hi}, %2;\n add.rn.f32.bf16 %0, lo, %0;\n add.rn.f32.bf16 %1, hi, %1;\n}"
            : "+f"(acc[2 * h]), "+f"(acc[2 * h + 1])
            : "r"(u[h]));
      }
    }
  }
}

// The sums of `count` entries (the same for every lane of the warp) whose
// 16-bit offsets start at `list`, chunks `stride` bytes apart.
template <int PREC, int SIGN, bool GEN>
__device__ __forceinline__ void gather_rows(float* acc, uint32_t rep, uint32_t list, uint32_t wlist, uint32_t stride,
                                            int count) {
#define DECO_LO(u) (rep + ((u) & 0xFFFFu) * 16u)
#define DECO_HI(u) (rep + ((u) >> 16) * 16u)
#pragma unroll 1
  for (; count >= 8; count -= 8, list += stride, wlist += 2 * stride) {
    const uint4 q = lds128(list);
    const uint32_t o[4] = {q.x, q.y, q.z, q.w};
    float w[8] = {};
    if (GEN) {
      const uint4 a = lds128(wlist), b = lds128(wlist + 16);
      w[0] = __uint_as_float(a.x); w[1] = __uint_as_float(a.y); w[2] = __uint_as_float(a.z); w[3] = __uint_as_float(a.w);
      w[4] = __uint_as_float(b.x); w[5] = __uint_as_float(b.y); w[6] = __uint_as_float(b.z); w[7] = __uint_as_float(b.w);
    }
    uint4 x[8];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      x[2 * h] = lds128(DECO_LO(o[h]));
      x[2 * h + 1] = lds128(DECO_HI(o[h]));
    }
#pragma unroll
    for (int h = 0; h < 8; ++h) add_vec<PREC, SIGN, GEN>(acc, x[h], w[h]);
  }
  if (count > 0) {
    uint4 q = lds128(list);
    uint4 wa = make_uint4(0u, 0u, 0u, 0u), wb = wa;
    if (GEN) { wa = lds128(wlist); wb = lds128(wlist + 16); }
    if (count & 4) {
      const uint4 x0 = lds128(DECO_LO(q.x)), x1 = lds128(DECO_HI(q.x)), x2 = lds128(DECO_LO(q.y)),
                  x3 = lds128(DECO_HI(q.y));
      add_vec<PREC, SIGN, GEN>(acc, x0, __uint_as_float(wa.x));
      add_vec<PREC, SIGN, GEN>(acc, x1, __uint_as_float(wa.y));
      add_vec<PREC, SIGN, GEN>(acc, x2, __uint_as_float(wa.z));
      add_vec<PREC, SIGN, GEN>(acc, x3, __uint_as_float(wa.w));
      q.x = q.z; q.y = q.w;
      wa = wb;
    }
    if (count & 2) {
      const uint4 x0 = lds128(DECO_LO(q.x)), x1 = lds128(DECO_HI(q.x));
      add_vec<PREC, SIGN, GEN>(acc, x0, __uint_as_float(wa.x));
      add_vec<PREC, SIGN, GEN>(acc, x1, __uint_as_float(wa.y));
      q.x = q.y;
      wa.x = wa.z;
    }
    if (count & 1) add_vec<PREC, SIGN, GEN>(acc, lds128(DECO_LO(q.x)), __uint_as_float(wa.x));
  }
#undef DECO_LO
#undef DECO_HI
}

// PERCOL: step sizes and budgets per column (else one step size, every column below C active)
// BATCH: the form of a batch's launch.  Its momentum stays in global memory (this launch's scratch, in L2), which
// leaves room for a second CTA on the SM or for wider slabs, and its warps take the next slice from a counter, longest
// first: scale-free graphs have hubs whose slices cost ten times the others'.  48 BA graphs of 200 - 1 200 rows, 256
// starts, FP32, two rounds: k_slab 40.3 ms; slabs of 2 vectors, momentum in shared memory, slices by turns 28.4; here
// 20.1 with 4 vectors (2: 22.3; slices by turns 21.5).  One graph's phase keeps turns (torus 0.61 ms, 0.70 by counter).
template <int PREC, int WMODE, bool PERCOL, int LPR, bool BATCH, int NT>
__global__ void __launch_bounds__(NT) k_rows(const __grid_constant__ RowsParams P) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ int s_next[2];                              // BATCH: next slice of an even / odd step
  constexpr int VN = PREC == DECO_PREC_BF16 ? 8 : 4;     // columns of a vector
  constexpr size_t ESZ = PREC == DECO_PREC_BF16 ? 2 : 4;
  constexpr int SR = 32 / LPR;                           // rows of a slice
  constexpr int W = 16 * LPR;                            // bytes of a slab row
  constexpr bool GEN = WMODE == W_GENERAL;
  int gi = 0, col0 = blockIdx.x * LPR * VN;
  if (P.items) { const int2 it = P.items[blockIdx.x]; gi = it.x; col0 = it.y; }
  const RowsGraph& G = P.graphs ? P.graphs[gi] : P.g0;
  const int n = G.n, ld = G.ld, C = G.C;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x, nw = nt >> 5;
  const int sub = lane % LPR, ri = lane / LPR;           // vector of the row, row of the slice
  const bool lap = P.objective == DECO_OBJ_LAPLACIAN, mom = P.mu != 0.0f;

  // ---- shared memory: two replicas (rows 0 ... n - 1 in sorted order, row n zero), slice table, lists, weights,
  // net degrees, momentum
  const uint32_t rep_bytes = (uint32_t)(n + 1) * W;
  const uint32_t img16 = (uint32_t)G.nslices + (uint32_t)G.list16 + (uint32_t)G.wts16;
  unsigned char* const img = smem + 2 * (size_t)rep_bytes;
  float* const dn = reinterpret_cast<float*>(img + 16 * (size_t)img16);
  // momentum by position: in shared memory, or (BATCH) this slab's part of G.v, n x (LPR x VN) floats from G.v + col0 n
  float* const vsm = BATCH ? G.v + (size_t)col0 * n
                             : reinterpret_cast<float*>(img + 16 * (size_t)img16 + (lap ? up16((size_t)n * 4) : 0));
  for (uint32_t i = tid; i < img16; i += nt) reinterpret_cast<uint4*>(img)[i] = __ldg(G.image + i);
  const int c0 = col0 + sub * VN;                        // this lane's first column
  const bool in = c0 < ld;                               // ld % 8 == 0: a vector lies inside a row or past it
  unsigned char* const yg = static_cast<unsigned char*>(G.y) + (size_t)c0 * ESZ;
  for (int i = tid; i < n * LPR; i += nt) {
    // nt is a multiple of LPR: i % LPR == sub
    const int p = i / LPR, r = __ldg(G.order + p);
    uint4 q = make_uint4(0u, 0u, 0u, 0u);
    if (in) q = *reinterpret_cast<const uint4*>(yg + (size_t)r * ld * ESZ);
    reinterpret_cast<uint4*>(smem)[i] = q;
    if (lap && sub == 0) dn[p] = __ldg(G.dnet + r);
    if (mom) {
#pragma unroll
      for (int h = 0; h < VN; h += 4) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (!BATCH && P.load_v && in) v = *reinterpret_cast<const float4*>(G.v + (size_t)r * ld + c0 + h);
        *reinterpret_cast<float4*>(vsm + (size_t)i * VN + h) = v;
      }
    }
  }
  if (BATCH && tid < 2) s_next[tid] = nw;
  if (tid < 2 * LPR)
    *reinterpret_cast<uint4*>(smem + (tid / LPR) * (size_t)rep_bytes + (size_t)n * W + (tid % LPR) * 16) =
        make_uint4(0u, 0u, 0u, 0u);

  // ---- this lane's columns
  float alpha[PERCOL ? VN : 1];
  int32_t tmax[PERCOL ? VN : 1];
  uint32_t live = 0u;                                    // columns below C
#pragma unroll
  for (int h = 0; h < VN; ++h) {
    if (c0 + h < C) live |= 1u << h;
    if (PERCOL) {
      alpha[h] = c0 + h < C ? (G.alpha_cols ? P.afac * __ldg(G.alpha_cols + c0 + h) : P.alpha) : 0.0f;
      tmax[h] = c0 + h < C ? (G.steps_cols ? __ldg(G.steps_cols + c0 + h) : P.steps) : 0;
    }
  }
  if (!PERCOL) { alpha[0] = P.alpha; tmax[0] = 0; }
  __syncthreads();

  const uint32_t base = lds_addr(smem), table = base + 2 * rep_bytes, lists = table + 16u * G.nslices,
                 wts = lists + 16u * G.list16;
  int nsteps = P.steps_dev ? min(P.steps, __ldg(P.steps_dev)) : P.steps;
  if (PERCOL) {
    // past its longest budget nothing of the slab changes; every warp's lanes hold all of its columns
    int longest = 0;
#pragma unroll
    for (int h = 0; h < VN; ++h) longest = max(longest, tmax[PERCOL ? h : 0]);
    nsteps = min(nsteps, __reduce_max_sync(0xFFFFFFFFu, longest));
  }
  uint32_t cur = 0;
  bool bad = false;
  for (int t = 0; t < nsteps; ++t) {
    const uint32_t rep = base + cur * rep_bytes + sub * 16u;
    unsigned char* const next = smem + (size_t)(cur ^ 1u) * rep_bytes;
    if (BATCH && tid == 0) s_next[(t + 1) & 1] = nw;     // last read in step t - 1
    // slices by turns, forth and back, so that every warp gets long and short ones (BATCH: from the counter)
    for (int i = 0, s = warp, ahead = 0; s < G.nslices;
         ++i, s = BATCH ? __shfl_sync(0xFFFFFFFFu, ahead, 0) : i * nw + ((i & 1) ? nw - 1 - warp : warp)) {
      const int p = s * SR + ri;
      const bool row = p < n;
      const size_t vs = ((size_t)p * LPR + sub) * VN;
      float v[VN] = {};
      if (BATCH && mom && row) load_f32(v, vsm + vs);   // ahead of the gathers, which hide its latency
      const uint4 si = lds128(table + 16u * s);
      float acc[VN];
#pragma unroll
      for (int h = 0; h < VN; ++h) acc[h] = 0.0f;
      const uint32_t l0 = lists + 16u * (si.x + ri), w0 = wts + 16u * (si.w + 2 * ri);
      gather_rows<PREC, +1, GEN>(acc, rep, l0, w0, 16u * SR, (int)si.y);
      if (WMODE == W_SIGN) gather_rows<PREC, -1, false>(acc, rep, l0 + 16u * SR * ((si.y + 7) / 8), 0, 16u * SR, (int)si.z);
      if (BATCH && lane == 0) ahead = atomicAdd(&s_next[t & 1], 1);
      if (!row) continue;
      // fused epilogue: gradient, momentum, step, projection
      const uint4 old = lds128(rep + (uint32_t)p * W);
      float y[VN];
      if (PREC == DECO_PREC_FP32) {
        y[0] = __uint_as_float(old.x); y[1] = __uint_as_float(old.y); y[2] = __uint_as_float(old.z); y[3] = __uint_as_float(old.w);
      } else {
        const uint32_t u[4] = {old.x, old.y, old.z, old.w};
#pragma unroll
        for (int h = 0; h < 4; ++h) { y[(2 * h) % VN] = bf16lo(u[h]); y[(2 * h + 1) % VN] = bf16hi(u[h]); }
      }
      if (!BATCH && mom) load_f32(v, vsm + vs);
      const float dr = lap ? dn[p] : 0.0f;
      float out[VN];
#pragma unroll
      for (int h = 0; h < VN; ++h) {
        const float grad = lap ? fmaf(dr, y[h], -acc[h]) : -acc[h];
        const float step = mom ? fmaf(P.mu, v[h], grad) : grad;
        const bool active = PERCOL ? t < tmax[PERCOL ? h : 0] : ((live >> h) & 1u) != 0;
        float yn = fmaf(alpha[PERCOL ? h : 0], step, y[h]);
        if (active && !isfinite(yn)) bad = true;
        yn = fminf(fmaxf(yn, -1.0f), 1.0f);
        out[h] = active ? yn : y[h];
        if (mom && active) v[h] = step;
      }
      uint4 q;
      if (PREC == DECO_PREC_FP32)
        q = make_uint4(__float_as_uint(out[0]), __float_as_uint(out[1]), __float_as_uint(out[2]), __float_as_uint(out[3]));
      else
        q = make_uint4(pack_bf16x2(out[0], out[1]), pack_bf16x2(out[2], out[3]), pack_bf16x2(out[4 % VN], out[5 % VN]),
                       pack_bf16x2(out[6 % VN], out[7 % VN]));
      *reinterpret_cast<uint4*>(next + (size_t)p * W + sub * 16) = q;
      if (mom) store_f32(vsm + vs, v);
    }
    __syncthreads();
    cur ^= 1u;
  }

  // ---- the rows (and momentum) back to global memory
  const uint4* const fin = reinterpret_cast<const uint4*>(smem + (size_t)cur * rep_bytes);
  if (in) {
    for (int i = tid; i < n * LPR; i += nt) {
      const int r = __ldg(G.order + i / LPR);
      *reinterpret_cast<uint4*>(yg + (size_t)r * ld * ESZ) = fin[i];
      if (!BATCH && mom && P.store_v) {
#pragma unroll
        for (int h = 0; h < VN; h += 4)
          *reinterpret_cast<float4*>(G.v + (size_t)r * ld + c0 + h) = *reinterpret_cast<const float4*>(vsm + (size_t)i * VN + h);
      }
    }
  }
  if (bad && P.flag) atomicOr(P.flag, 1);
}

template <int PREC, int WMODE, bool PERCOL, int LPR, bool BATCH>
cudaError_t launch_l(const RowsParams& p, int n_items, cudaStream_t st) {
  constexpr int NT = rows_max_threads(PREC, PERCOL);
  auto fn = k_rows<PREC, WMODE, PERCOL, LPR, BATCH, NT>;
  const cudaError_t e = allow_smem(fn);
  if (e != cudaSuccess) return e;
  fn<<<(unsigned)n_items, std::min(p.threads, NT), p.smem, st>>>(p);
  return cudaGetLastError();
}

template <int PREC, int WMODE, bool PERCOL, bool BATCH>
cudaError_t launch_c(const RowsParams& p, int n_items, cudaStream_t st) {
  switch (p.lpr) {
    case 1: return launch_l<PREC, WMODE, PERCOL, 1, BATCH>(p, n_items, st);
    case 2: return launch_l<PREC, WMODE, PERCOL, 2, BATCH>(p, n_items, st);
    case 4: return launch_l<PREC, WMODE, PERCOL, 4, BATCH>(p, n_items, st);
    default: return launch_l<PREC, WMODE, PERCOL, 8, BATCH>(p, n_items, st);
  }
}

template <int PREC, int WMODE>
cudaError_t launch_w(const RowsParams& p, bool percol, int n_items, cudaStream_t st) {
  if (p.graphs) return launch_c<PREC, WMODE, true, true>(p, n_items, st);
  return percol ? launch_c<PREC, WMODE, true, false>(p, n_items, st) : launch_c<PREC, WMODE, false, false>(p, n_items, st);
}

template <int PREC>
cudaError_t launch_p(const RowsParams& p, int wmode, bool percol, int n_items, cudaStream_t st) {
  if (wmode == W_UNIT) return launch_w<PREC, W_UNIT>(p, percol, n_items, st);
  if (wmode == W_SIGN) return launch_w<PREC, W_SIGN>(p, percol, n_items, st);
  return launch_w<PREC, W_GENERAL>(p, percol, n_items, st);
}

// rows by entries (largest first), then + entries, then index; np: + entries of every row
void sort_rows(const int32_t* row_ptr, const float* w, int wmode, int32_t row0, int32_t n, std::vector<int32_t>* order,
               std::vector<int32_t>* np) {
  np->resize((size_t)n);
  for (int32_t r = 0; r < n; ++r) {
    const int32_t e0 = row_ptr[row0 + r], e1 = row_ptr[row0 + r + 1];
    int32_t neg = 0;
    if (wmode == W_SIGN)
      for (int32_t e = e0; e < e1; ++e) neg += w[e] < 0.0f;
    (*np)[(size_t)r] = e1 - e0 - neg;
  }
  order->resize((size_t)n);
  std::iota(order->begin(), order->end(), 0);
  // counting sorts, the second key first: each keeps the order of equal keys
  std::vector<int32_t> from, at;
  auto by = [&](auto&& key) {
    int32_t most = 0;
    for (int32_t r = 0; r < n; ++r) most = std::max(most, key(r));
    at.assign((size_t)most + 2, 0);
    for (int32_t r = 0; r < n; ++r) ++at[(size_t)(most - key(r)) + 1];
    for (int32_t k = 0; k <= most; ++k) at[(size_t)k + 1] += at[(size_t)k];
    from = *order;
    for (int32_t r : from) (*order)[(size_t)at[(size_t)(most - key(r))]++] = r;
  };
  if (wmode == W_SIGN) by([&](int32_t r) { return (*np)[(size_t)r]; });
  by([&](int32_t r) { return row_ptr[row0 + r + 1] - row_ptr[row0 + r]; });
}

// slice table (4 words a slice) and the sizes of *im
void slice_table(const int32_t* row_ptr, int wmode, int32_t row0, const std::vector<int32_t>& order,
                 const std::vector<int32_t>& np, RowsImage* im, std::vector<int32_t>* table) {
  const int SR = 32 / im->lpr;
  im->nslices = (im->n + SR - 1) / SR;
  int64_t l16 = 0, w16 = 0;
  im->padded = 0;
  im->longest = 0;
  table->clear();
  for (int32_t s = 0; s < im->nslices; ++s) {
    int32_t kp = 0, kn = 0;
    for (int32_t p = s * SR; p < std::min(im->n, (s + 1) * SR); ++p) {
      const int32_t r = order[(size_t)p], d = row_ptr[row0 + r + 1] - row_ptr[row0 + r];
      kp = std::max(kp, np[(size_t)r]);
      kn = std::max(kn, d - np[(size_t)r]);
    }
    table->insert(table->end(), {(int32_t)l16, kp, kn, (int32_t)w16});
    const int64_t chunks = (kp + 7) / 8 + (kn + 7) / 8;
    l16 += chunks * SR;
    if (wmode == W_GENERAL) w16 += chunks * SR * 2;
    im->padded += (int64_t)(kp + kn) * SR;
    im->longest = std::max(im->longest, kp + kn);
  }
  im->list16 = (int32_t)std::min<int64_t>(l16, INT32_MAX / 32);
  im->wts16 = (int32_t)std::min<int64_t>(w16, INT32_MAX / 32);
}

}  // namespace

size_t rows_smem_least(int32_t n, int64_t nnz, int prec, int wmode) {
  return 2 * ((size_t)n + 1) * 16 + (size_t)nnz * (wmode == W_GENERAL ? 6 : 2) + (size_t)n * (4 + (prec == DECO_PREC_BF16 ? 32 : 16));
}

size_t rows_smem_bytes(const RowsImage& im, int prec, bool lap, bool mom) {   // mom: in shared memory
  const size_t rep = (size_t)(im.n + 1) * 16 * im.lpr;
  return 2 * rep + 16 * ((size_t)im.nslices + im.list16 + im.wts16) + (lap ? up16((size_t)im.n * 4) : 0) +
         (mom ? (size_t)im.n * im.lpr * (prec == DECO_PREC_BF16 ? 32 : 16) : 0);
}

int rows_threads(int32_t n, int lpr) { return std::min(1024, (int)(((int64_t)n * lpr + 31) / 32 * 32)); }

void rows_measure(const int32_t* row_ptr, const float* w, int wmode, int32_t row0, int32_t n,
                  std::vector<RowsImage>* out) {
  std::vector<int32_t> order, np, table;
  sort_rows(row_ptr, w, wmode, row0, n, &order, &np);
  for (int lpr = 1; lpr <= ROWS_MAX_LPR; lpr *= 2) {
    RowsImage im;
    im.lpr = lpr;
    im.n = n;
    slice_table(row_ptr, wmode, row0, order, np, &im, &table);
    out->push_back(im);
  }
}

void rows_build(const int32_t* row_ptr, const int32_t* col, const float* w, int wmode, int32_t row0, int32_t n,
                int lpr, RowsImage* out, std::vector<uint32_t>* words_out) {
  RowsImage im;
  im.lpr = lpr;
  im.n = n;
  std::vector<int32_t> order, np, table;
  sort_rows(row_ptr, w, wmode, row0, n, &order, &np);
  slice_table(row_ptr, wmode, row0, order, np, &im, &table);
  const int SR = 32 / lpr;
  std::vector<int32_t> pos((size_t)n);
  for (int32_t p = 0; p < n; ++p) pos[(size_t)order[(size_t)p]] = p;
  const uint16_t zero = (uint16_t)(n * lpr);
  std::vector<uint16_t> lists((size_t)im.list16 * 8, zero);
  std::vector<float> wts((size_t)im.wts16 * 4, 0.0f);
  for (int32_t p = 0; p < n; ++p) {
    const int32_t s = p / SR, i = p % SR, r = order[(size_t)p];
    const int32_t e0 = row_ptr[row0 + r], e1 = row_ptr[row0 + r + 1];
    const int32_t l0 = table[4 * (size_t)s], kp = table[4 * (size_t)s + 1], w0 = table[4 * (size_t)s + 3];
    for (int32_t e = e0; e < e1; ++e) {
      // positive (or all) entries, then negative ones: the device edge order
      const int32_t q = e - e0 < np[(size_t)r] ? e - e0 : (kp + 7) / 8 * 8 + (e - e0 - np[(size_t)r]);
      const size_t at = (size_t)(l0 + (q / 8) * SR + i) * 8 + q % 8;
      lists[at] = (uint16_t)(pos[(size_t)(col[e] - row0)] * lpr);
      if (wmode == W_GENERAL) wts[(size_t)(w0 + (q / 8) * SR * 2 + 2 * i) * 4 + q % 8] = w[e];
    }
  }
  const size_t words = 4 * ((size_t)im.nslices + im.list16 + im.wts16) + (size_t)n;
  std::vector<uint32_t>& host = *words_out;
  host.assign(words, 0u);
  uint32_t* at = host.data();
  auto put = [&](const void* src, size_t bytes) {
    if (bytes) memcpy(at, src, bytes);
    at += bytes / 4;
  };
  put(table.data(), 16 * (size_t)im.nslices);
  put(lists.data(), 16 * (size_t)im.list16);
  put(wts.data(), 16 * (size_t)im.wts16);
  put(order.data(), 4 * (size_t)n);
  *out = im;
}

int rows_image(deco_graph* g, int lpr, const RowsImage** out) {
  for (auto& im : g->rows)
    if (im.lpr == lpr) { *out = &im; return DECO_OK; }
  RowsImage im;
  std::vector<uint32_t> host;
  rows_build(g->h_row_ptr.data(), g->h_col.data(), g->h_w.empty() ? nullptr : g->h_w.data(), g->wmode, 0, g->n, lpr,
             &im, &host);
  cudaError_t e = cudaMalloc((void**)&im.data, host.size() * 4);
  if (e != cudaSuccess) return cuda_fail(e, "cudaMalloc(row image)");
  e = upload(im.data, host.data(), host.size() * 4);
  if (e != cudaSuccess) {
    cudaFree(im.data);
    return cuda_fail(e, "cudaMemcpy(row image)");
  }
  g->rows.push_back(im);
  *out = &g->rows.back();
  return DECO_OK;
}

RowsGraph rows_graph(const RowsImage& im) {
  RowsGraph r{};
  r.n = im.n;
  r.nslices = im.nslices;
  r.list16 = im.list16;
  r.wts16 = im.wts16;
  r.image = reinterpret_cast<const uint4*>(im.data);
  r.order = reinterpret_cast<const int32_t*>(im.data + 4 * ((size_t)im.nslices + im.list16 + im.wts16));
  return r;
}

// Fitted to the measured steps of ER(800, 0.06), degree 48 (FP32: 14 500 / 22 600 / 33 000 cycles for LPR 1 / 2 / 4)
// and of graphs of degree 4 ... 20; the shared-memory part is within 10 % of them.
// In registers only the entries' vectors and the new row are left (graphs of 60 - 1 000 rows, degree 5 - 16: within 12 %).
double rows_cycles(const RowsImage& im, bool registers, double* pipe) {
  const double conflict = im.lpr == 8 ? 1.0 : im.lpr == 4 ? 1.5 : im.lpr == 2 ? 2.1 : 2.8;
  // wavefronts: the entries' vectors, the lists (16 bytes per 8 entries), the row's own loads and stores
  const double wave = (double)im.padded * im.lpr / 8.0 * conflict +
                      (double)(im.list16 + im.wts16) / 8.0 + 4.0 * im.n * im.lpr / 8.0;
  if (registers) {
    *pipe = (double)im.padded * im.lpr / 8.0 * conflict + im.n * im.lpr / 8.0;
    return *pipe + 400.0;
  }
  // the longest slice is one warp's chain: about 9 cycles an entry
  const double chain = 9.0 * im.longest + 60.0;
  *pipe = wave;
  return std::max(wave, chain) + 350.0;
}

int launch_rows(const RowsParams& p, int n_items, int prec, int wmode, cudaStream_t st) {
  if (n_items < 1) return DECO_OK;
  const bool percol = p.graphs != nullptr || p.g0.alpha_cols || p.g0.steps_cols;
  const cudaError_t e = prec == DECO_PREC_BF16 ? launch_p<DECO_PREC_BF16>(p, wmode, percol, n_items, st)
                                               : launch_p<DECO_PREC_FP32>(p, wmode, percol, n_items, st);
  if (e != cudaSuccess) return cuda_fail(e, "k_rows launch");
  return DECO_OK;
}

}  // namespace deco
