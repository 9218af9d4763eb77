// Fused PGA step, one launch per step, iterate in global memory.
//
//   G = A Y                                  (CSR gather, FP32 accumulation)
//   grad = d (.) y - G   (Laplacian, Eq. 6 / 9)     or  -G   (multilinear)
//   V <- mu V + grad     (heavy-ball momentum, Sec. 4.2), else V = grad
//   y <- Proj[-1,1](y + alpha_eff V)         (Eq. 7 / 10)
//
// Layout: a group of G lanes owns one (row, column chunk); each lane owns one
// 16-byte vector of the row (4 FP32 or 8 BF16 columns).  Every gathered
// neighbour row segment is therefore read as G x 16 contiguous bytes.  The
// column chunks are the grid's second dimension: all rows of one before the
// next, so that a gathered chunk keeps L2 to itself.  Used for graphs whose
// iterate does not fit on chip and as the reference launch shape for the
// persistent kernels.
//
// Bound by the latency of a row's chain (row bounds, indices, gathers) over
// the warps that the registers allow, and by instruction issue (78 % with
// 16-bit blocks before the mixed-precision adds).  So: few registers and many
// warps; four gathers at once and the last one to three together, not one by
// one; the own row loaded ahead of the gathers, the momentum after them (held
// through them it costs registers, and spills on +-1 graphs; read past L2,
// evict-first, it left L2 where the whole block fits there); the sums of +-1
// and unit graphs in 16 bits by mixed-precision adds; blocks of two warps.  us
// per step, with eight gathers, a serial tail and the own row last, and here:
//   n        degree  C    precision  weights   momentum
//   200 003  12      100  FP32       general   0.9       189 -> 160
//   200 003  12      128  BF16       unit      0          91 ->  61
//   200 003  12      128  BF16       unit      0.9       121 ->  85
//   200 003  12       60  FP32       unit      0          75 ->  51
//   10^6      8      128  BF16       unit      0         522 -> 335
//   10^6     10       64  FP32       unit      0.9       525 -> 437
//   10^6      8       20  FP32       unit      0         239 -> 166
//   700 000   5       40  FP32       +-1       0.9       236 -> 209 (momentum ahead and evict-first 271)
//   700 000   5        3  BF16       general   0.9        91 ->  84 (99)
// Eight gathers in flight without momentum cost 5 % on the second and fifth; a
// loop over rows with the next row's indices prefetched took 136 and 649 us
// (24 warps an SM); indices held a chunk ahead spill.
#include <algorithm>

#include "deco_internal.cuh"
#include "spmm.cuh"

namespace deco {

int device_sm_count();

namespace {

struct KArgs {
  int32_t n, C, ld, G, lg;   // G = 2^lg lanes per row
  int32_t lr;                // 2^lr rows per block
  int32_t ch0;               // first column chunk of the launch
  const int32_t* row_ptr;
  const int32_t* col_idx;
  const uint32_t* col_sw;
  const float* w;
  const float* dnet;
  const void* yin;
  void* yout;
  float* v;
  float alpha_eff;      // alpha * objective factor
  float afac;           // objective factor applied to alpha_cols (1 or 2)
  float mu;
  const float* alpha_cols;
  const int32_t* steps_cols;
  int32_t t;
  int32_t* flag;
};

// Gathers in flight per lane, and blocks of 256 threads per SM (registers): more of both at once does not fit.  With
// momentum more gathers win over more warps (206 319 nodes, 9 columns, 16-bit 31 against 26 us), and without it on long
// rows and small grids (4 / 8 gathers: 4 096 nodes of degree 300 45 / 29 us, 8 000 of degree 20 9.2 / 8.1; 200 000 of
// degree 24, 16-bit 88 / 96).
template <bool EIGHT>
struct Shape {
  static constexpr int U = EIGHT ? 8 : 4;
  static constexpr int BLOCKS = EIGHT ? 4 : 6;
};

__device__ __forceinline__ void unpack(const uint4 q, float (&v)[4]) {
  v[0] = __uint_as_float(q.x); v[1] = __uint_as_float(q.y); v[2] = __uint_as_float(q.z); v[3] = __uint_as_float(q.w);
}
__device__ __forceinline__ void unpack(const uint4 q, float (&v)[8]) {
  v[0] = bf16lo(q.x); v[1] = bf16hi(q.x); v[2] = bf16lo(q.y); v[3] = bf16hi(q.y);
  v[4] = bf16lo(q.z); v[5] = bf16hi(q.z); v[6] = bf16lo(q.w); v[7] = bf16hi(q.w);
}

// acc += the vector q of entry x (column index, or index | sign bit), weight w (W_GENERAL)
template <int PREC, int WMODE, int VN>
__device__ __forceinline__ void add_entry(float (&acc)[VN], uint4 q, uint32_t x, float w) {
  if constexpr (PREC == DECO_PREC_BF16 && WMODE != W_GENERAL) {
    // +-1: the sign bits of both halves, then the mixed-precision add (bf16 widened exactly, one rounding)
    const uint32_t flip = WMODE == W_SIGN && (x & 0x80000000u) ? 0x80008000u : 0u;
    const uint32_t u[4] = {q.x ^ flip, q.y ^ flip, q.z ^ flip, q.w ^ flip};
#pragma unroll
    for (int h = 0; h < 4; ++h)
      asm("{\n .reg .b16 lo, hi;\n mov.b32 {lo, hi}, %2;\n add.rn.f32.bf16 %0, lo, %0;\n add.rn.f32.bf16 %1, hi, %1;\n}"
          : "+f"(acc[2 * h]), "+f"(acc[2 * h + 1])
          : "r"(u[h]));
  } else {
    float v[VN];
    unpack(q, v);
    if (WMODE == W_SIGN) w = (x & 0x80000000u) ? -1.0f : 1.0f;
#pragma unroll
    for (int k = 0; k < VN; ++k) acc[k] = WMODE == W_UNIT ? acc[k] + v[k] : fmaf(w, v[k], acc[k]);
  }
}

// OVERLAP: launched to start while the step before it still runs (programmatic dependent launch).  It then reads the
// graph ahead of waiting for that step, and the block by plain loads, since others still write it when this kernel
// starts.  Saves the launch gap of the smaller steps; on large ones the wait ahead of the own row's loads costs 1 - 5 %.
template <int PREC, int WMODE, bool MOM, bool LAP, bool EIGHT, bool OVERLAP>
__global__ void __launch_bounds__(256, Shape<EIGHT>::BLOCKS) k_step_global(const __grid_constant__ KArgs a) {
  using V = VecT<PREC>;
  constexpr int VN = V::N, U = Shape<EIGHT>::U;
  if (OVERLAP) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the next step's blocks may be placed
  const int gl = threadIdx.x & (a.G - 1);         // lane within the group
  const int64_t row = ((int64_t)blockIdx.x << a.lr) + (threadIdx.x >> a.lg);
  const int32_t c0 = ((a.ch0 + (int32_t)blockIdx.y) * a.G + gl) * VN;   // first column of this lane
  if (row >= a.n || c0 >= a.C) return;
  const int32_t r = (int32_t)row;

  const uint32_t* const col = WMODE == W_SIGN ? a.col_sw : reinterpret_cast<const uint32_t*>(a.col_idx);
  const int32_t e1 = __ldg(a.row_ptr + r + 1);
  int32_t e = __ldg(a.row_ptr + r);
  if (OVERLAP) {
    if (e < e1) {
      asm volatile("prefetch.global.L1 [%0];" ::"l"(col + e));
      if (WMODE == W_GENERAL) asm volatile("prefetch.global.L1 [%0];" ::"l"(a.w + e));
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
  }
  auto vector = [](const char* at) {
    const uint4* const q = reinterpret_cast<const uint4*>(at);
    return OVERLAP ? *q : __ldg(q);
  };
  // own row ahead of the gathers, which hide its latency
  const size_t base = (size_t)r * a.ld + c0;
  const uint4 own = vector(static_cast<const char*>(a.yin) + base * (16 / VN));
  // where it was measured to help (+-1, 16-bit: 2 000 nodes of degree 64, 40 columns 9.8 -> 8.1 us; 700 000 of degree 5,
  // 3 columns 82 -> 94); general weights in 16 bits lose 13 %, FP32 up to 10 % on narrow blocks
  if (MOM && PREC == DECO_PREC_BF16 && WMODE == W_SIGN) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.v + base));
  const float dr = LAP ? __ldg(a.dnet + r) : 0.0f;
  const char* const yb = static_cast<const char*>(a.yin) + (size_t)c0 * (16 / VN);
  const uint32_t row_bytes = (uint32_t)a.ld * (16 / VN);
  auto gather = [&](uint32_t x) { return vector(yb + (size_t)(WMODE == W_SIGN ? x & 0x7FFFFFFFu : x) * row_bytes); };

  float acc[VN];
#pragma unroll
  for (int k = 0; k < VN; ++k) acc[k] = 0.0f;
  uint4 raw[U];
  uint32_t x[U];
  float w[U] = {};
  for (; e + U <= e1; e += U) {
#pragma unroll
    for (int q = 0; q < U; ++q) {
      x[q] = __ldg(col + e + q);
      if (WMODE == W_GENERAL) w[q] = __ldg(a.w + e + q);
      raw[q] = gather(x[q]);
    }
#pragma unroll
    for (int q = 0; q < U; ++q) add_entry<PREC, WMODE>(acc, raw[q], x[q], w[q]);
  }
  // the last entries, together
#pragma unroll
  for (int q = 0; q < U - 1; ++q) {
    if (e + q < e1) {
      x[q] = __ldg(col + e + q);
      if (WMODE == W_GENERAL) w[q] = __ldg(a.w + e + q);
      raw[q] = gather(x[q]);
    }
  }
#pragma unroll
  for (int q = 0; q < U - 1; ++q)
    if (e + q < e1) add_entry<PREC, WMODE>(acc, raw[q], x[q], w[q]);

  float vv[VN];
  if (MOM) {
#pragma unroll
    for (int k = 0; k < VN; k += 4) {
      const float4 q = *reinterpret_cast<const float4*>(a.v + base + k);
      vv[k] = q.x; vv[k + 1] = q.y; vv[k + 2] = q.z; vv[k + 3] = q.w;
    }
  }

  // ---- epilogue: gradient, momentum, step, projection
  float y[VN], out[VN];
  unpack(own, y);
  bool bad = false;
  const bool whole = c0 + VN <= a.C;
  if (whole && !a.alpha_cols && !a.steps_cols) {
#pragma unroll
    for (int k = 0; k < VN; ++k) {
      const float grad = LAP ? fmaf(dr, y[k], -acc[k]) : -acc[k];
      if (MOM) vv[k] = fmaf(a.mu, vv[k], grad);
      const float yn = fmaf(a.alpha_eff, MOM ? vv[k] : grad, y[k]);
      bad = bad || !isfinite(yn);
      out[k] = fminf(fmaxf(yn, -1.0f), 1.0f);
    }
  } else {
#pragma unroll
    for (int k = 0; k < VN; ++k) {
      const int32_t c = c0 + k;
      const float grad = LAP ? fmaf(dr, y[k], -acc[k]) : -acc[k];
      const float step = MOM ? fmaf(a.mu, vv[k], grad) : grad;
      const float alpha = a.alpha_cols ? a.afac * __ldg(a.alpha_cols + (c < a.C ? c : 0)) : a.alpha_eff;
      const bool active = (c < a.C) && (!a.steps_cols || a.t < __ldg(a.steps_cols + c));
      float yn = fmaf(alpha, step, y[k]);
      if (active && !isfinite(yn)) bad = true;
      yn = fminf(fmaxf(yn, -1.0f), 1.0f);
      out[k] = active ? yn : y[k];
      if (MOM && active) vv[k] = step;
    }
  }
  if (whole) {
    V::store(a.yout, base, out);
    if (MOM) {
#pragma unroll
      for (int k = 0; k < VN; k += 4)
        *reinterpret_cast<float4*>(a.v + base + k) = make_float4(vv[k], vv[k + 1], vv[k + 2], vv[k + 3]);
    }
  } else {
    // ragged last vector: only columns < C are written
#pragma unroll
    for (int k = 0; k < VN; ++k) {
      if (c0 + k >= a.C) continue;
      if (PREC == DECO_PREC_FP32) static_cast<float*>(a.yout)[base + k] = out[k];
      else static_cast<__nv_bfloat16*>(a.yout)[base + k] = __float2bfloat16_rn(out[k]);
      if (MOM) a.v[base + k] = vv[k];
    }
  }
  if (bad && a.flag) atomicExch(a.flag, 1);
}

void launch_k(void (*fn)(const KArgs), const KArgs& a, bool overlap, dim3 grid, cudaStream_t st) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(1u << (a.lr + a.lg), 1, 1);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = overlap ? 1 : 0;
  cudaLaunchKernelEx(&cfg, fn, a);   // the caller reads the error
}

template <int PREC, int WMODE, bool MOM, bool EIGHT>
void launch_o(const KArgs& a, bool lap, bool overlap, dim3 grid, cudaStream_t st) {
  if (lap) {
    if (overlap) launch_k(k_step_global<PREC, WMODE, MOM, true, EIGHT, true>, a, true, grid, st);
    else launch_k(k_step_global<PREC, WMODE, MOM, true, EIGHT, false>, a, false, grid, st);
  } else {
    if (overlap) launch_k(k_step_global<PREC, WMODE, MOM, false, EIGHT, true>, a, true, grid, st);
    else launch_k(k_step_global<PREC, WMODE, MOM, false, EIGHT, false>, a, false, grid, st);
  }
}

template <int PREC, int WMODE>
void launch_w(const KArgs& a, bool mom, bool lap, bool eight, bool overlap, dim3 grid, cudaStream_t st) {
  if (mom) launch_o<PREC, WMODE, true, true>(a, lap, overlap, grid, st);
  else if (eight) launch_o<PREC, WMODE, false, true>(a, lap, overlap, grid, st);
  else launch_o<PREC, WMODE, false, false>(a, lap, overlap, grid, st);
}

template <int PREC>
void launch_p(const KArgs& a, int wmode, bool mom, bool lap, bool eight, bool overlap, dim3 grid, cudaStream_t st) {
  if (wmode == W_UNIT) launch_w<PREC, W_UNIT>(a, mom, lap, eight, overlap, grid, st);
  else if (wmode == W_SIGN) launch_w<PREC, W_SIGN>(a, mom, lap, eight, overlap, grid, st);
  else launch_w<PREC, W_GENERAL>(a, mom, lap, eight, overlap, grid, st);
}

}  // namespace

int launch_step_global(const StepLaunch& s, cudaStream_t st) {
  KArgs a{};
  const int VN = s.precision == DECO_PREC_BF16 ? 8 : 4;
  const int nvec = (s.C + VN - 1) / VN;
  int G = 1;
  for (; G < nvec && G < 32; G <<= 1) ++a.lg;
  a.n = s.n;
  a.C = s.C;
  a.ld = s.ld;
  a.G = G;
  a.row_ptr = s.row_ptr;
  a.col_idx = s.col_idx;
  a.col_sw = s.col_sw;
  a.w = s.w;
  a.dnet = s.dnet;
  a.yin = s.yin;
  a.yout = s.yout;
  a.v = s.v;
  const float fac = s.objective == DECO_OBJ_MULTILINEAR01 ? 2.0f : 1.0f;
  a.alpha_eff = fac * s.alpha;
  a.afac = fac;
  a.mu = s.mu;
  a.alpha_cols = s.alpha_cols;
  a.steps_cols = s.steps_cols;
  a.t = s.t;
  a.flag = s.flag;
  if (s.n == 0 || s.C == 0) return DECO_OK;
  const bool mom = s.mu != 0.0f;
  const bool lap = s.objective == DECO_OBJ_LAPLACIAN;
  const int32_t nchunks = (nvec + G - 1) / G;
  const int64_t threads = (int64_t)s.n * G * nchunks, sms = device_sm_count();
  // long rows, and grids that leave warps' slots empty anyway: eight gathers in flight; not where the long rows fill one
  // wave with four and a second, nearly empty one with eight (3 000 nodes of degree 300, 256 columns: 49 us, here 39)
  const bool long_rows = s.nnz >= (int64_t)64 * s.n;
  const bool eight = long_rows ? threads <= 1024 * sms || threads > 1536 * sms : (int64_t)s.n * s.C <= sms * 2048 * VN;
  // steps of up to 64 MB of block and momentum (10 - 70 us): the gap between two launches is worth the wait.  Not on
  // longer rows, whose lanes find most of their index words in L1: the waits of the blocks that come in drop them.  The
  // fewer lanes a row has, the shorter the rows on which this costs more than the gap.  us per step, overlapping and
  // not: 60 000 nodes of degree 32, 3 columns 27 / 16; 20 000 of degree 24, 11 columns, 16-bit 9.4 / 8.7; 3 000 of
  // degree 300, 40 columns 37 / 21; 5 000 of degree 100, 40 columns, 16-bit 13 / 11; but 120 000 of degree 6, 3 columns
  // 10.5 / 10.9; 60 000 of degree 48, 100 columns 62 / 64; 1 000 of degree 200, 40 columns 13.2 / 14.9
  const int64_t longest = G >= 2 && threads <= 256 * sms                                       ? 1024
                          : G >= 8 || s.n <= 64 * sms || (G == 4 && threads >= 1024 * sms) ? 80
                          : G == 4 || (G == 2 && threads >= 1024 * sms)                     ? 28
                                                                                            : 16;
  const bool overlap = s.overlap && nchunks <= 65535 && s.nnz < longest * s.n &&
                       (int64_t)s.n * s.C * ((s.precision == DECO_PREC_BF16 ? 2 : 4) + (mom ? 8 : 0)) <= (64 << 20);
  // blocks of two warps free their slots sooner (200 003 nodes, 100 columns, momentum, multilinear: eight warps 172 us,
  // two 160; with the Laplacian's degrees 170 and 170); where every block waits for the step before, fewer and larger
  a.lr = (overlap ? (G == 1 ? 8 : 7) : 6) - a.lg;
  const unsigned rows = (unsigned)(((int64_t)s.n + ((int64_t)1 << a.lr) - 1) >> a.lr);
  for (a.ch0 = 0; a.ch0 < nchunks; a.ch0 += 65535) {
    const dim3 grid(rows, (unsigned)std::min(nchunks - a.ch0, 65535));
    if (s.precision == DECO_PREC_BF16) launch_p<DECO_PREC_BF16>(a, s.wmode, mom, lap, eight, overlap, grid, st);
    else launch_p<DECO_PREC_FP32>(a, s.wmode, mom, lap, eight, overlap, grid, st);
    DECO_CUDA_TRY(cudaGetLastError());
  }
  return DECO_OK;
}

// ---- slab-major layout: row-major n x ld  <->  S slabs of dense n x w
// element (r, c) of the row-major block is element (r, c % w) of slab c / w.
namespace {
template <typename T>
__global__ void k_to_slabs(int32_t n, int32_t ld, int32_t C, int32_t w, int32_t S, const T* __restrict__ src,
                           T* __restrict__ dst, int to_slabs) {
  const int64_t total = (int64_t)n * C;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = i / C;
    const int32_t c = (int32_t)(i % C);   // column of the row-major block
    const int64_t slab_idx = (int64_t)(c / w) * n * w + r * w + (c % w);
    if (to_slabs) dst[slab_idx] = src[r * ld + c];
    else dst[r * ld + c] = src[slab_idx];
  }
}
}  // namespace

int launch_slab_layout(int32_t n, int32_t ld, int32_t C, int32_t w, int32_t S, size_t esz, const void* src,
                       void* dst, bool to_slabs, cudaStream_t st) {
  const int64_t total = (int64_t)n * C;
  if (total == 0) return DECO_OK;
  (void)S;
  const int block = 256;
  const unsigned grid = (unsigned)std::min<int64_t>((total + block - 1) / block, 152 * 32);
  if (esz == 2)
    k_to_slabs<uint16_t><<<grid, block, 0, st>>>(n, ld, C, w, S, static_cast<const uint16_t*>(src),
                                                  static_cast<uint16_t*>(dst), to_slabs ? 1 : 0);
  else
    k_to_slabs<uint32_t><<<grid, block, 0, st>>>(n, ld, C, w, S, static_cast<const uint32_t*>(src),
                                                  static_cast<uint32_t*>(dst), to_slabs ? 1 : 0);
  DECO_CUDA_TRY(cudaGetLastError());
  return DECO_OK;
}

}  // namespace deco
