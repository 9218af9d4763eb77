// 16-byte vectors of the iterate (the per-step kernels), and the CSR gather
// (one row of A Y for one lane's vector of columns) of the learned proposal's
// message passing.
#pragma once

#include "deco_internal.cuh"

namespace deco {

template <int PREC>
struct VecT;
template <>
struct VecT<DECO_PREC_FP32> {
  static constexpr int N = 4;
  __device__ static void store(void* base, size_t idx, const float* in) {
    *reinterpret_cast<float4*>(static_cast<float*>(base) + idx) = make_float4(in[0], in[1], in[2], in[3]);
  }
};
template <>
struct VecT<DECO_PREC_BF16> {
  static constexpr int N = 8;
  __device__ static void store(void* base, size_t idx, const float* in) {
    uint4 q = make_uint4(pack_bf16x2(in[0], in[1]), pack_bf16x2(in[2], in[3]),
                         pack_bf16x2(in[4], in[5]), pack_bf16x2(in[6], in[7]));
    *reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(base) + idx) = q;
  }
};

struct CsrView {
  const int32_t* col_idx;
  const uint32_t* col_sw;   // index | sign bit (W_SIGN)
  const float* w;           // weights (W_GENERAL)
};

template <int WMODE>
__device__ __forceinline__ void csr_edge(const CsrView& A, int32_t e, int32_t& j, float& wt) {
  if (WMODE == W_UNIT) {
    j = __ldg(A.col_idx + e);
    wt = 1.0f;
  } else if (WMODE == W_SIGN) {
    uint32_t s = __ldg(A.col_sw + e);
    j = (int32_t)(s & 0x7FFFFFFFu);
    wt = (s & 0x80000000u) ? -1.0f : 1.0f;
  } else {
    j = __ldg(A.col_idx + e);
    wt = __ldg(A.w + e);
  }
}

// acc[k] += sum over entries e in [e0, e1) of w_e * Y[j_e, c0 + k], in CSR
// order, for this lane's four FP32 columns.  Eight gathers are kept in flight
// per lane, then four, then one.
template <int WMODE>
__device__ __forceinline__ void csr_gather_row(const CsrView& A, const float* Y, int32_t ld, int32_t c0, int32_t e0,
                                               int32_t e1, float* acc) {
  auto gather = [&](int32_t j) { return __ldg(reinterpret_cast<const float4*>(Y + (size_t)j * ld + c0)); };
  auto add = [&](const float4& y, float w) {
    const float v[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[k] = WMODE == W_UNIT ? acc[k] + v[k] : fmaf(w, v[k], acc[k]);
  };
  int32_t e = e0;
  for (; e + 8 <= e1; e += 8) {
    int32_t j[8];
    float w[8];
    float4 y[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) csr_edge<WMODE>(A, e + q, j[q], w[q]);
#pragma unroll
    for (int q = 0; q < 8; ++q) y[q] = gather(j[q]);
#pragma unroll
    for (int q = 0; q < 8; ++q) add(y[q], w[q]);
  }
  for (; e + 4 <= e1; e += 4) {
    int32_t j[4];
    float w[4];
    float4 y[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) csr_edge<WMODE>(A, e + q, j[q], w[q]);
#pragma unroll
    for (int q = 0; q < 4; ++q) y[q] = gather(j[q]);
#pragma unroll
    for (int q = 0; q < 4; ++q) add(y[q], w[q]);
  }
  for (; e < e1; ++e) {
    int32_t j;
    float w;
    csr_edge<WMODE>(A, e, j, w);
    add(gather(j), w);
  }
}

}  // namespace deco
