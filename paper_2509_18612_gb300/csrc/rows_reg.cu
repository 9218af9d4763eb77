// Row-vector form of the persistent on-chip kernel (rows.cu) for graphs whose
// slices are at most a warp each and whose rows have at most 32 entries: what
// belongs to a row stays in its lane's registers through the phase.
//
// k_rows reads its slice table and entry lists, the own row and the momentum
// from shared memory in every step, one after another.  With one slice per
// warp they never change hands: a lane keeps its entries' offsets (two to a
// register), its own vector, momentum and net degree, and a step is its
// gathers, the update, one 16-byte store and a barrier.  The iterates are
// bit-identical to k_rows'.  Bound by the gathers' bank conflicts and, below
// some 200 rows, by the latency of gathers, update and barrier (0.35 us).
// Measured us per step, k_rows and here:
//   ER(100), degree 10, 64 columns, FP32        0.75 -> 0.49
//   ER(300), degree 6, 256 columns, 16-bit      0.98 -> 0.69
//   ER(500), degree 12, 64 columns, FP32        1.55 -> 1.29
//   ER(1000), degree 16, 256 columns, FP32      3.35 -> 3.06
//   40 x 20 torus, +-1, 1 024 columns, 16-bit   1.51 -> 1.17
#include <algorithm>

#include "rows.cuh"

namespace deco {
namespace {

__device__ __forceinline__ uint4 lds128(uint32_t a) {
  uint4 q;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(q.x), "=r"(q.y), "=r"(q.z), "=r"(q.w) : "r"(a));
  return q;
}

template <int VN>
__device__ __forceinline__ void unpack(const uint4 q, float (&v)[VN]) {
  if constexpr (VN == 4) {
    v[0] = __uint_as_float(q.x); v[1] = __uint_as_float(q.y); v[2] = __uint_as_float(q.z); v[3] = __uint_as_float(q.w);
  } else {
    v[0] = bf16lo(q.x); v[1] = bf16hi(q.x); v[2] = bf16lo(q.y); v[3] = bf16hi(q.y);
    v[4] = bf16lo(q.z); v[5] = bf16hi(q.z); v[6] = bf16lo(q.w); v[7] = bf16hi(q.w);
  }
}

// E: entries held per lane; B: gathers in flight
template <int PREC, int WMODE, int E, int B, int NT>
__global__ void __launch_bounds__(NT) k_rows_reg(const __grid_constant__ RowsParams P) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr int VN = PREC == DECO_PREC_BF16 ? 8 : 4;     // columns of a vector
  constexpr size_t ESZ = 16 / VN;
  const RowsGraph& G = P.g0;
  const int lpr = P.lpr, SR = 32 / lpr;                  // vectors of a slab row, rows of a slice
  const int n = G.n, ld = G.ld, C = G.C;
  const int lane = threadIdx.x & 31, s = threadIdx.x >> 5;
  const int sub = lane % lpr, ri = lane / lpr;
  const int p = s * SR + ri;                             // position of the lane's row
  const bool row = p < n;
  const bool lap = P.objective == DECO_OBJ_LAPLACIAN, mom = P.mu != 0.0f;
  const uint32_t rep_bytes = (uint32_t)(n + 1) * 16u * lpr;
  const int c0 = blockIdx.x * lpr * VN + sub * VN;       // the lane's first column
  const bool in = c0 < ld;

  // ---- this lane's entries (+ entries, then - entries of a +-1 graph): byte offsets into a replica, two to a register
  const int4 si = __ldg(reinterpret_cast<const int4*>(G.image) + s);
  const uint16_t* const lists = reinterpret_cast<const uint16_t*>(G.image + G.nslices);
  const int kp = si.y, total = si.y + (WMODE == W_SIGN ? si.z : 0);
  uint32_t ent[E / 2];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    uint32_t off = (uint32_t)n * lpr;                    // the row of zeros
    if (e < total) {
      const int chunk = e < kp ? e / 8 : (kp + 7) / 8 + (e - kp) / 8, k = e < kp ? e % 8 : (e - kp) % 8;
      off = __ldg(lists + ((size_t)si.x + (size_t)chunk * SR + ri) * 8 + k);
    }
    if (e & 1) ent[e / 2] |= off << 20;
    else ent[e / 2] = off << 4;
  }

  // ---- own row, momentum, replicas
  const int r = row ? __ldg(G.order + p) : 0;
  unsigned char* const yg = static_cast<unsigned char*>(G.y) + ((size_t)r * ld + c0) * ESZ;
  uint4 own = make_uint4(0u, 0u, 0u, 0u);
  if (row && in) own = *reinterpret_cast<const uint4*>(yg);
  const float dr = lap && row ? __ldg(G.dnet + r) : 0.0f;
  float v[VN] = {};
  if (mom && P.load_v && row && in) {
#pragma unroll
    for (int h = 0; h < VN; h += 4) {
      const float4 q = *reinterpret_cast<const float4*>(G.v + (size_t)r * ld + c0 + h);
      v[h] = q.x; v[h + 1] = q.y; v[h + 2] = q.z; v[h + 3] = q.w;
    }
  }
  const uint32_t mine = (uint32_t)(p * lpr + sub) * 16u;
  if (row) *reinterpret_cast<uint4*>(smem + mine) = own;
  if (threadIdx.x < 2u * lpr)
    *reinterpret_cast<uint4*>(smem + (threadIdx.x / lpr) * (size_t)rep_bytes + (size_t)n * 16 * lpr + (threadIdx.x % lpr) * 16) =
        make_uint4(0u, 0u, 0u, 0u);
  uint32_t live = 0u;                                    // columns below C
#pragma unroll
  for (int h = 0; h < VN; ++h)
    if (c0 + h < C) live |= 1u << h;
  __syncthreads();

  const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem);
  uint32_t cur = base, next = base + rep_bytes;
  bool bad = false;
  for (int t = 0; t < P.steps; ++t) {
    float acc[VN];
#pragma unroll
    for (int h = 0; h < VN; ++h) acc[h] = 0.0f;
    const uint32_t rep = cur + sub * 16u;
#pragma unroll
    for (int eb = 0; eb < E; eb += B) {
      if (eb >= total) break;                            // the same for the warp
      uint4 q[B];
#pragma unroll
      for (int e = 0; e < B; ++e) {
        const uint32_t x = ent[(eb + e) / 2];
        if (eb + e < total) q[e] = lds128(rep + ((eb + e) & 1 ? x >> 16 : x & 0xFFFFu));
      }
#pragma unroll
      for (int e = 0; e < B; ++e) {
        if (eb + e < total) {
          if constexpr (PREC == DECO_PREC_BF16) {
            // widened exactly, one rounding: the mixed-precision add
            const uint32_t flip = WMODE == W_SIGN && eb + e >= kp ? 0x80008000u : 0u;
            const uint32_t u[4] = {q[e].x ^ flip, q[e].y ^ flip, q[e].z ^ flip, q[e].w ^ flip};
#pragma unroll
            for (int h = 0; h < 4; ++h)
              asm("{\n .reg .b16 lo, hi;\n mov.b32 {lo, hi}, %2;\n add.rn.f32.bf16 %0, lo, %0;\n add.rn.f32.bf16 %1, hi, %1;\n}"
                  : "+f"(acc[(2 * h) % VN]), "+f"(acc[(2 * h + 1) % VN])
                  : "r"(u[h]));
          } else {
            const float y[4] = {__uint_as_float(q[e].x), __uint_as_float(q[e].y), __uint_as_float(q[e].z), __uint_as_float(q[e].w)};
            const float w = WMODE == W_SIGN && eb + e >= kp ? -1.0f : 1.0f;
#pragma unroll
            for (int h = 0; h < 4; ++h) acc[h] = WMODE == W_SIGN ? fmaf(w, y[h], acc[h]) : acc[h] + y[h];
          }
        }
      }
    }
    // fused update: gradient, momentum, step, projection
    float y[VN], out[VN];
    unpack<VN>(own, y);
#pragma unroll
    for (int h = 0; h < VN; ++h) {
      const float grad = lap ? fmaf(dr, y[h], -acc[h]) : -acc[h];
      const float step = mom ? fmaf(P.mu, v[h], grad) : grad;
      const bool active = ((live >> h) & 1u) != 0;
      float yn = fmaf(P.alpha, step, y[h]);
      if (active && !isfinite(yn)) bad = true;
      yn = fminf(fmaxf(yn, -1.0f), 1.0f);
      out[h] = active ? yn : y[h];
      if (active) v[h] = step;
    }
    if constexpr (PREC == DECO_PREC_FP32)
      own = make_uint4(__float_as_uint(out[0]), __float_as_uint(out[1]), __float_as_uint(out[2]), __float_as_uint(out[3]));
    else
      own = make_uint4(pack_bf16x2(out[0], out[1]), pack_bf16x2(out[2], out[3]), pack_bf16x2(out[4 % VN], out[5 % VN]),
                       pack_bf16x2(out[6 % VN], out[7 % VN]));
    if (row)
      asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(next + mine), "r"(own.x), "r"(own.y), "r"(own.z), "r"(own.w)
                   : "memory");
    __syncthreads();
    const uint32_t other = cur;
    cur = next;
    next = other;
  }
  if (row && in) {
    *reinterpret_cast<uint4*>(yg) = own;
    if (mom && P.store_v) {
#pragma unroll
      for (int h = 0; h < VN; h += 4)
        *reinterpret_cast<float4*>(G.v + (size_t)r * ld + c0 + h) = make_float4(v[h], v[h + 1], v[h + 2], v[h + 3]);
    }
  }
  if (bad && row && P.flag) atomicOr(P.flag, 1);
}

template <int PREC, int WMODE, int E>
cudaError_t launch_e(const RowsParams& p, int n_items, int threads, size_t smem, cudaStream_t st) {
  // up to 16 warps: eight gathers in flight; up to 32 leave 64 registers a thread
  auto fn = threads <= 512 ? k_rows_reg<PREC, WMODE, E, 8, 512> : k_rows_reg<PREC, WMODE, E, 4, 1024>;
  const cudaError_t e = allow_smem(fn);
  if (e != cudaSuccess) return e;
  fn<<<(unsigned)n_items, threads, smem, st>>>(p);
  return cudaGetLastError();
}

template <int PREC, int WMODE>
cudaError_t launch_w(const RowsParams& p, int longest, int n_items, int threads, size_t smem, cudaStream_t st) {
  if (longest <= 8) return launch_e<PREC, WMODE, 8>(p, n_items, threads, smem, st);
  if (longest <= 16) return launch_e<PREC, WMODE, 16>(p, n_items, threads, smem, st);
  return launch_e<PREC, WMODE, 32>(p, n_items, threads, smem, st);
}

template <int PREC>
cudaError_t launch_p(const RowsParams& p, int wmode, int longest, int n_items, int threads, size_t smem, cudaStream_t st) {
  return wmode == W_UNIT ? launch_w<PREC, W_UNIT>(p, longest, n_items, threads, smem, st)
                         : launch_w<PREC, W_SIGN>(p, longest, n_items, threads, smem, st);
}

}  // namespace

// More than 16 warps leave 64 registers, which +-1 rows of more than 8 entries overflow (800 rows of degree 4, 16-bit:
// 2.5 us a step here, 1.8 in k_rows).
bool rows_reg_fits(const RowsImage& im, int wmode) {
  if (wmode == W_GENERAL || im.nslices > 32 || im.longest > 32) return false;
  return wmode == W_UNIT || im.nslices <= 16 || im.longest <= 8;
}

size_t rows_reg_smem_bytes(const RowsImage& im) { return 2 * (size_t)(im.n + 1) * 16 * im.lpr; }

int launch_rows_reg(const RowsParams& p, const RowsImage& im, int n_items, int prec, int wmode, cudaStream_t st) {
  if (n_items < 1) return DECO_OK;
  const size_t smem = rows_reg_smem_bytes(im);
  const int threads = 32 * im.nslices;
  const cudaError_t e = prec == DECO_PREC_BF16
                            ? launch_p<DECO_PREC_BF16>(p, wmode, im.longest, n_items, threads, smem, st)
                            : launch_p<DECO_PREC_FP32>(p, wmode, im.longest, n_items, threads, smem, st);
  if (e != cudaSuccess) return cuda_fail(e, "k_rows_reg launch");
  return DECO_OK;
}

}  // namespace deco
