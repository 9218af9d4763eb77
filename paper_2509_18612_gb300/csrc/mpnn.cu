// Learned initial-mean proposal: a small message-passing network whose
// output h = tanh(o) in (-1,1)^n becomes the mean of the Gaussian starts of
// the solver (Sec. 4.2's "Gaussian around a mean vector", with a learned mean
// instead of IDI).  Inference, loss, backward pass and Adam run in these
// kernels; the neighbour aggregation is the CSR gather of spmm.cuh.
//
//   X  = node features [d/Delta, d/mean(d), 1/sqrt(d+1), 5 x U(-1,1)]   (n x 8)
//   H0 = relu(X W0 + b0)
//   M  = D^-1 A H_{l-1};   H_l = relu(H_{l-1} Ws_l + M Wn_l + b_l),  l = 1..L
//   o  = H_L wo + bo,      h = tanh(o)
//   loss per graph: min over the two labellings z, 1 - z of the mean
//   logistic loss softplus(-t o), t = 2z - 1 (a cut does not change when
//   both sides swap); batch loss = mean over graphs.
// Weight gradients are reductions over nodes in a fixed order (chunks of
// nodes in node order, then the chunks in order), so they are deterministic.
#include <algorithm>
#include <cmath>
#include <vector>

#include "api_util.cuh"
#include "deco_internal.cuh"
#include "spmm.cuh"

using namespace deco;

namespace {
constexpr int F_IN = 8;
constexpr int N_RANDOM = 5;
constexpr uint32_t STREAM_FEAT = 4, STREAM_PARAM = 5;
}  // namespace

struct deco_mpnn {
  int32_t hidden = 64, layers = 3;
  int64_t n_params = 0;
  float* theta = nullptr;   // device parameters (flat, see mpnn oracle layout)
  float* m = nullptr;       // Adam first moment
  float* v = nullptr;       // Adam second moment, behind the first
  int64_t t = 0;            // Adam step count
};

namespace {

struct Layout {
  int64_t W0, b0, wo, bo, total;
  std::vector<int64_t> Ws, Wn, b;
};

Layout layout(int32_t H, int32_t L) {
  Layout o;
  int64_t p = 0;
  o.W0 = p; p += (int64_t)F_IN * H;
  o.b0 = p; p += H;
  for (int l = 0; l < L; ++l) {
    o.Ws.push_back(p); p += (int64_t)H * H;
    o.Wn.push_back(p); p += (int64_t)H * H;
    o.b.push_back(p); p += H;
  }
  o.wo = p; p += H;
  o.bo = p; p += 1;
  o.total = p;
  return o;
}

// ---------------------------------------------------------------- kernels

__global__ void k_init_params(int64_t count, const int64_t* starts, const double* bounds, int32_t n_ranges,
                              uint32_t k0, uint32_t k1, float* theta) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  double a = 0.0;
  for (int r = 0; r < n_ranges; ++r)
    if (i >= starts[2 * r] && i < starts[2 * r + 1]) a = bounds[r];
  if (a == 0.0) { theta[i] = 0.0f; return; }
  const uint4 x = philox4x32_10(make_uint4((uint32_t)i, 0u, 0u, STREAM_PARAM), k0, k1);
  // (2u - 1) a with u exact in FP32; the product is formed in FP64 and rounded
  theta[i] = (float)((2.0 * (double)u01(x.x) - 1.0) * a);
}

__global__ void k_features(int32_t n, const int32_t* deg, const int32_t* gid, const int32_t* goff,
                           const int32_t* gmax, const double* gmean, int32_t max_deg, double mean_deg,
                           uint32_t k0, uint32_t k1, float* X, float* dinv) {
  const int32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  uint32_t kk0 = k0, kk1 = k1, vr = (uint32_t)v;
  double delta = max_deg > 0 ? (double)max_deg : 1.0, mean = mean_deg > 0 ? mean_deg : 1.0;
  if (gid) {
    const int32_t g = gid[v];
    delta = gmax[g] > 0 ? (double)gmax[g] : 1.0;
    mean = gmean[g] > 0 ? gmean[g] : 1.0;
    batch_key(gid, goff, v, kk0, kk1, vr);
  }
  const double d = (double)deg[v];
  float* x = X + (size_t)v * F_IN;
  x[0] = (float)(d / delta);
  x[1] = (float)(d / mean);
  x[2] = (float)(1.0 / sqrt(d + 1.0));
  dinv[v] = d > 0.0 ? (float)(1.0 / d) : 0.0f;
  for (int j = 0; j < N_RANDOM; ++j) {
    const uint4 r = philox4x32_10(make_uint4(vr, (uint32_t)j, 0u, STREAM_FEAT), kk0, kk1);
    x[3 + j] = (float)(2.0 * (double)u01(r.x) - 1.0);
  }
}

// ---- layer kernels.  A block of 4 H threads owns LTILE nodes; thread (ty, tx)
// computes nodes ty, ty + 16, ... of the tile (four of them) times columns
// 4 tx ... 4 tx + 3 from operands in shared memory: 8 16-byte shared loads feed
// 64 fused multiply-adds.  The sums run over the inputs in ascending order, as
// one thread per output would form them.  Bound by the neighbour gather's
// latency and the FP32 pipe.  Measured, n = 50 000, H = 64, degree 10: a layer
// (gather + both products) 45 us, as separate gather and one-output-per-thread
// kernels 14.6 + 160 us.  Four rows per thread: on the 48-graph training batch
// (20 000 nodes) two rows, twice the blocks, take 2.86 instead of 3.23 ms for 11 passes,
// but at n = 50 000 four rows take 150 us an inference and two take 183 (one: 3.48 ms, 219 us).
constexpr int RPT = 4;               // tile rows per thread
constexpr int LTILE = 16 * RPT;

// what the last layer adds: o = H_L wo + bo, h = tanh(o), and the loss sums
struct Head {
  const float* wo = nullptr;     // null: not the last layer
  const float* bo = nullptr;
  float* o = nullptr;            // n, or null
  float* h = nullptr;            // n, or null
  const uint8_t* z = nullptr;    // labels: add the loss terms to lp / lm
  const int32_t* gid = nullptr;
  double *lp = nullptr, *lm = nullptr;
};

struct LayerArgs {
  int32_t n, H, F1;              // in1 is n x F1
  const float* in1;
  const int32_t* row_ptr;        // aggregation over in1's rows (null: the first layer has none)
  CsrView A;
  const float* dinv;
  const float *W1, *W2, *b;
  float* agg;                    // n x H aggregated inputs, kept for the weight gradients, or null
  float* post;                   // n x H, or null (the last layer of an inference)
  int32_t bf16;
  double *zlp, *zlm;             // loss sums zeroed by the first layer
  int32_t n_graphs;
  Head head;
};

__device__ __forceinline__ double sigmoid_d(double x) {
  return x >= 0 ? 1.0 / (1.0 + exp(-x)) : exp(x) / (1.0 + exp(x));
}

// sum over the warp's lanes of (a, b) per graph into lp / lm: one atomic per
// warp where its nodes share a graph (lanes without a node pass g = -1)
__device__ __forceinline__ void add_loss(unsigned mask, int32_t g, double a, double b, double* lp, double* lm) {
  const int32_t g0 = __shfl_sync(mask, g, __ffs(mask) - 1);
  if (__all_sync(mask, g == g0) && mask == 0xFFFFFFFFu) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_xor_sync(mask, a, o);
      b += __shfl_xor_sync(mask, b, o);
    }
    if ((threadIdx.x & 31) == 0 && g0 >= 0) {
      atomicAdd(lp + g0, a);
      atomicAdd(lm + g0, b);
    }
  } else if (g >= 0) {
    atomicAdd(lp + g, a);
    atomicAdd(lm + g, b);
  }
}

// acc[i][c] += sum_k sA[(ty + 16 i) P + k] sW[k H + 4 tx + c], k ascending, K a multiple of 4
__device__ __forceinline__ void tile_gemm(const float* sA, int P, const float* sW, int ldw, int K, int ty, int tx,
                                          float (&acc)[RPT][4]) {
#pragma unroll 2
  for (int k = 0; k < K; k += 4) {
    float4 a[RPT], w[4];
#pragma unroll
    for (int i = 0; i < RPT; ++i) a[i] = *reinterpret_cast<const float4*>(sA + (ty + 16 * i) * P + k);
#pragma unroll
    for (int q = 0; q < 4; ++q) w[q] = *reinterpret_cast<const float4*>(sW + (k + q) * ldw + 4 * tx);
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      const float av[4] = {a[i].x, a[i].y, a[i].z, a[i].w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        acc[i][0] = fmaf(av[q], w[q].x, acc[i][0]);
        acc[i][1] = fmaf(av[q], w[q].y, acc[i][1]);
        acc[i][2] = fmaf(av[q], w[q].z, acc[i][2]);
        acc[i][3] = fmaf(av[q], w[q].w, acc[i][3]);
      }
    }
  }
}

// post = relu(in1 W1 + (D^-1 A in1) W2 + b), optionally rounded to BF16
template <int WMODE>
__global__ void __launch_bounds__(512) k_layer(const __grid_constant__ LayerArgs a) {
  extern __shared__ __align__(16) float sm[];
  const int H = a.H, F1 = a.F1, F2 = a.row_ptr ? H : 0, K = F1 + F2, P = K + 4;
  float* sW = sm;                 // K x H
  float* sA = sm + K * H;         // LTILE x P
  const int TX = H / 4, tx = threadIdx.x % TX, ty = threadIdx.x / TX, nt = blockDim.x;
  const int32_t v0 = blockIdx.x * LTILE;
  if (a.zlp && blockIdx.x == 0)
    for (int g = threadIdx.x; g < a.n_graphs; g += nt) a.zlp[g] = a.zlm[g] = 0.0;
  for (int i = threadIdx.x; i < F1 * H / 4; i += nt)
    reinterpret_cast<float4*>(sW)[i] = __ldg(reinterpret_cast<const float4*>(a.W1) + i);
  for (int i = threadIdx.x; i < F2 * H / 4; i += nt)
    reinterpret_cast<float4*>(sW + F1 * H)[i] = __ldg(reinterpret_cast<const float4*>(a.W2) + i);
  for (int i = threadIdx.x; i < LTILE * F1 / 4; i += nt) {
    const int r = i / (F1 / 4), q = i % (F1 / 4);
    const float4 x = v0 + r < a.n ? __ldg(reinterpret_cast<const float4*>(a.in1 + (size_t)(v0 + r) * F1) + q)
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
    *reinterpret_cast<float4*>(sA + r * P + 4 * q) = x;
  }
  if (F2) {
#pragma unroll 1
    for (int i = 0; i < RPT; ++i) {
      const int r = ty + 16 * i, v = v0 + r;
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
      if (v < a.n) {
        csr_gather_row<WMODE>(a.A, a.in1, H, 4 * tx, __ldg(a.row_ptr + v), __ldg(a.row_ptr + v + 1), acc);
        const float s = __ldg(a.dinv + v);
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[c] *= s;
        if (a.agg)
          *reinterpret_cast<float4*>(a.agg + (size_t)v * H + 4 * tx) = make_float4(acc[0], acc[1], acc[2], acc[3]);
      }
      *reinterpret_cast<float4*>(sA + r * P + F1 + 4 * tx) = make_float4(acc[0], acc[1], acc[2], acc[3]);
    }
  }
  __syncthreads();
  float acc[RPT][4] = {};
  tile_gemm(sA, P, sW, H, K, ty, tx, acc);
  const float bb[4] = {a.b[4 * tx], a.b[4 * tx + 1], a.b[4 * tx + 2], a.b[4 * tx + 3]};
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const int v = v0 + ty + 16 * i;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float y = fmaxf(acc[i][c] + bb[c], 0.0f);
      if (a.bf16) y = __bfloat162float(__float2bfloat16_rn(y));
      acc[i][c] = y;
    }
    if (a.post && v < a.n)
      *reinterpret_cast<float4*>(a.post + (size_t)v * H + 4 * tx) =
          make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
  }
  if (!a.head.wo) return;
  // head: one thread per node of the tile, columns in ascending order
  __syncthreads();   // sA is free
  const int PH = H + 1;
#pragma unroll
  for (int i = 0; i < RPT; ++i)
#pragma unroll
    for (int c = 0; c < 4; ++c) sA[(ty + 16 * i) * PH + 4 * tx + c] = acc[i][c];
  __syncthreads();
  for (int r = threadIdx.x; r < LTILE; r += nt) {
    const int v = v0 + r;
    float o = 0.0f;
    for (int j = 0; j < H; ++j) o = fmaf(sA[r * PH + j], __ldg(a.head.wo + j), o);
    o += __ldg(a.head.bo);
    const bool have = v < a.n;
    if (have && a.head.o) a.head.o[v] = o;
    if (have && a.head.h) a.head.h[v] = tanhf(o);
    if (a.head.z) {
      // softplus(-t o) and softplus(t o), t = +-1, in FP64: they share log1p(exp(-|o|))
      const double x = (double)o, l = log1p(exp(-fabs(x)));
      const double tx_ = have && a.head.z[v] ? x : -x;
      const int32_t g = have ? (a.head.gid ? a.head.gid[v] : 0) : -1;
      add_loss(__activemask(), g, fmax(-tx_, 0.0) + l, fmax(tx_, 0.0) + l, a.head.lp, a.head.lm);
    }
  }
}

// Backward of one layer for a tile of nodes: the gradient of the layer's
// inputs to its ReLU,
//   first (the last layer): dpre = (dout wo) masked by H_l > 0, dout from the loss
//   else:                   dpre = (S + A T) masked by H_l > 0
// and what the next layer down needs, S' = dpre Ws^T and T' = D^-1 (dpre Wn^T).
struct BackArgs {
  int32_t n, H;
  const int32_t* row_ptr;
  CsrView A;
  const float* dinv;
  const float* Hl;               // n x H activations of this layer (its mask)
  const float *S, *T;            // from the layer above, or null (first)
  const float *o, *wo;           // first: outputs, head weights
  const uint8_t* z;
  const int32_t* gid;
  const int32_t* gsize;
  const double *lp, *lm;
  int32_t n_graphs;
  float* dout;                   // first: n, written
  float* dpre;                   // n x H, written
  const float *Ws, *Wn;          // null: layer 0 passes nothing further down
  float *So, *To;                // n x H, written
};

template <int WMODE>
__global__ void __launch_bounds__(512) k_back(const __grid_constant__ BackArgs a) {
  extern __shared__ __align__(16) float sm[];
  const int H = a.H, P = H + 4;
  float* sA = sm;                 // LTILE x P
  float* sW = sm + LTILE * P;     // H x 2H: column i of row j = Ws[i][j], column H + i = Wn[i][j]
  __shared__ float s_dout[LTILE];
  const int TX = H / 4, tx = threadIdx.x % TX, ty = threadIdx.x / TX, nt = blockDim.x;
  const int32_t v0 = blockIdx.x * LTILE;
  if (a.Ws) {
    for (int i = threadIdx.x; i < 2 * H * TX; i += nt) {
      const int c = i % (2 * H), j4 = i / (2 * H);
      const float4 w = __ldg(reinterpret_cast<const float4*>((c < H ? a.Ws + (size_t)c * H : a.Wn + (size_t)(c - H) * H)) + j4);
      sW[(4 * j4) * 2 * H + c] = w.x;
      sW[(4 * j4 + 1) * 2 * H + c] = w.y;
      sW[(4 * j4 + 2) * 2 * H + c] = w.z;
      sW[(4 * j4 + 3) * 2 * H + c] = w.w;
    }
  }
  if (a.o) {
    for (int r = threadIdx.x; r < LTILE; r += nt) {
      const int v = v0 + r;
      float d = 0.0f;
      if (v < a.n) {
        const int32_t g = a.gid ? a.gid[v] : 0;
        const double ng = a.gsize ? (double)a.gsize[g] : (double)a.n;
        const double s = (a.lp[g] / ng <= a.lm[g] / ng) ? 1.0 : -1.0;
        const double t = a.z[v] ? 1.0 : -1.0;
        d = (float)(-s * t * sigmoid_d(-s * t * (double)a.o[v]) / (ng * (double)a.n_graphs));
        a.dout[v] = d;
      }
      s_dout[r] = d;
    }
    __syncthreads();
  }
#pragma unroll 1
  for (int i = 0; i < RPT; ++i) {
    const int r = ty + 16 * i, v = v0 + r;
    float d[4] = {0.f, 0.f, 0.f, 0.f};
    if (v < a.n) {
      if (a.o) {
#pragma unroll
        for (int c = 0; c < 4; ++c) d[c] = s_dout[r] * __ldg(a.wo + 4 * tx + c);
      } else {
        csr_gather_row<WMODE>(a.A, a.T, H, 4 * tx, __ldg(a.row_ptr + v), __ldg(a.row_ptr + v + 1), d);
        const float4 s = *reinterpret_cast<const float4*>(a.S + (size_t)v * H + 4 * tx);
        d[0] += s.x; d[1] += s.y; d[2] += s.z; d[3] += s.w;
      }
      const float4 h = *reinterpret_cast<const float4*>(a.Hl + (size_t)v * H + 4 * tx);
      d[0] = h.x > 0.0f ? d[0] : 0.0f;
      d[1] = h.y > 0.0f ? d[1] : 0.0f;
      d[2] = h.z > 0.0f ? d[2] : 0.0f;
      d[3] = h.w > 0.0f ? d[3] : 0.0f;
      *reinterpret_cast<float4*>(a.dpre + (size_t)v * H + 4 * tx) = make_float4(d[0], d[1], d[2], d[3]);
    }
    *reinterpret_cast<float4*>(sA + r * P + 4 * tx) = make_float4(d[0], d[1], d[2], d[3]);
  }
  if (!a.Ws) return;
  __syncthreads();
#pragma unroll 1
  for (int half = 0; half < 2; ++half) {
    float acc[RPT][4] = {};
    tile_gemm(sA, P, sW + half * H, 2 * H, H, ty, tx, acc);
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      const int v = v0 + ty + 16 * i;
      if (v >= a.n) continue;
      const float s = half ? __ldg(a.dinv + v) : 1.0f;
      *reinterpret_cast<float4*>((half ? a.To : a.So) + (size_t)v * H + 4 * tx) =
          make_float4(acc[i][0] * s, acc[i][1] * s, acc[i][2] * s, acc[i][3] * s);
    }
  }
}

__device__ __forceinline__ void loss_total(int32_t n, int32_t n_graphs, const int32_t* gsize, const double* lp,
                                           const double* lm, double* out) {
  // batch loss = mean over graphs of min(lp, lm) / n_g, summed in graph order
  __shared__ double s[128];
  double tot = 0.0;
  for (int32_t g0 = 0; g0 < n_graphs; g0 += 128) {
    const int32_t g = g0 + (int32_t)threadIdx.x;
    __syncthreads();
    if (threadIdx.x < 128 && g < n_graphs) s[threadIdx.x] = fmin(lp[g], lm[g]) / (gsize ? (double)gsize[g] : (double)n);
    __syncthreads();
    if (threadIdx.x == 0)
      for (int32_t i = 0; i < 128 && g0 + i < n_graphs; ++i) tot += s[i];
  }
  if (threadIdx.x == 0) *out = tot / (double)n_graphs;
}

__global__ void k_loss_reduce(int32_t n, int32_t n_graphs, const int32_t* gsize, const double* lp, const double* lm,
                              double* out) {
  loss_total(n, n_graphs, gsize, lp, lm, out);
}

// Weight gradients dW[i][j] = sum_v in[v][i] d[v][j] and the bias gradients
// (column sums of d) of every layer in one launch, as a two-level reduction
// with a fixed order: chunks of nodes summed in node order into `part`
// (chunk x parameter), then the chunks in order (k_wgrad_sum).  A thread holds
// 8 x 4 sums in registers (3 16-byte shared loads per 32 fused multiply-adds).
// Measured, 48 graphs (23 000 nodes), H = 64, 3 layers: all of them 55 us,
// as one kernel per matrix with a division per product 4 070 us.
constexpr int WG_TILE = 32, WG_THREADS = 256, WG_MAX_JOBS = 9;

struct WgradJob {
  const float *in1, *in2, *d;
  int32_t F1, F2;
  int64_t oW1, oW2, ob;          // parameter offsets
};

struct WgradArgs {
  int32_t n, H, chunk, n_jobs, passes;   // passes: row groups of the widest job
  int64_t n_params;
  WgradJob job[WG_MAX_JOBS];
  const float *HL, *dout;        // the head: dwo = H_L^T dout, dbo = sum dout
  int64_t owo, obo;
  float* part;
};

__global__ void __launch_bounds__(WG_THREADS) k_wgrad_part(const __grid_constant__ WgradArgs a) {
  extern __shared__ __align__(16) float sm[];
  const int H = a.H, tid = threadIdx.x;
  const int32_t v0 = blockIdx.x * a.chunk, v1 = min(a.n, v0 + a.chunk);
  float* const part = a.part + (size_t)blockIdx.x * a.n_params;
  const int jb = blockIdx.y / a.passes, pass = blockIdx.y % a.passes;
  if (jb == a.n_jobs) {
    // head: `groups` row ranges of the chunk, then the ranges in order
    if (pass) return;
    const int groups = WG_THREADS / (H + 1), j = tid % (H + 1), g = tid / (H + 1);
    float acc = 0.0f;
    if (g < groups) {
      const int32_t span = (v1 - v0 + groups - 1) / groups, r0 = v0 + g * span, r1 = min(v1, r0 + span);
#pragma unroll 8
      for (int32_t v = r0; v < r1; ++v) acc = fmaf(j < H ? a.HL[(size_t)v * H + j] : 1.0f, a.dout[v], acc);
      sm[g * (H + 1) + j] = acc;
    }
    __syncthreads();
    if (tid <= H) {
      acc = 0.0f;
      for (int q = 0; q < groups; ++q) acc += sm[q * (H + 1) + tid];
      part[tid < H ? a.owo + tid : a.obo] = acc;
    }
    return;
  }
  const WgradJob& J = a.job[jb];
  const int TX = H / 4, TY = WG_THREADS / TX, tx = tid % TX, ty = tid / TX;
  const int R = J.F1 + J.F2, i0 = pass * TY * 8;
  if (i0 >= R) return;
  const int RW = min(R - i0, TY * 8);        // rows of this pass (a multiple of 4)
  const int P = (RW + 7) / 8 * 8 + 4;
  float* sA = sm;                            // WG_TILE x P
  float* sD = sm + WG_TILE * P;              // WG_TILE x H
  const bool on = ty * 8 < RW && ty < TY;
  const bool bias = pass == 0 && ty == 0;
  float acc[8][4] = {}, bs[4] = {};
  for (int i = tid; i < WG_TILE * P; i += WG_THREADS) sA[i] = 0.0f;   // the padding columns
  for (int32_t t0 = v0; t0 < v1; t0 += WG_TILE) {
    const int cnt = min(WG_TILE, v1 - t0);
    __syncthreads();
    for (int x = tid; x < cnt * (RW / 4); x += WG_THREADS) {
      const int r = x / (RW / 4), i = i0 + 4 * (x % (RW / 4));
      const float* src = i < J.F1 ? J.in1 + (size_t)(t0 + r) * J.F1 + i : J.in2 + (size_t)(t0 + r) * J.F2 + (i - J.F1);
      *reinterpret_cast<float4*>(sA + r * P + (i - i0)) = __ldg(reinterpret_cast<const float4*>(src));
    }
    for (int x = tid; x < cnt * TX; x += WG_THREADS)
      reinterpret_cast<float4*>(sD)[x] = __ldg(reinterpret_cast<const float4*>(J.d + (size_t)t0 * H) + x);
    __syncthreads();
    if (on) {
#pragma unroll 4
      for (int r = 0; r < cnt; ++r) {
        const float4 d = *reinterpret_cast<const float4*>(sD + r * H + 4 * tx);
        const float4 x0 = *reinterpret_cast<const float4*>(sA + r * P + 8 * ty);
        const float4 x1 = *reinterpret_cast<const float4*>(sA + r * P + 8 * ty + 4);
        const float xv[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          acc[q][0] = fmaf(xv[q], d.x, acc[q][0]);
          acc[q][1] = fmaf(xv[q], d.y, acc[q][1]);
          acc[q][2] = fmaf(xv[q], d.z, acc[q][2]);
          acc[q][3] = fmaf(xv[q], d.w, acc[q][3]);
        }
        if (bias) { bs[0] += d.x; bs[1] += d.y; bs[2] += d.z; bs[3] += d.w; }
      }
    }
  }
  if (!on) return;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int i = i0 + 8 * ty + q;
    if (8 * ty + q >= RW) break;
    float* dst = part + (i < J.F1 ? J.oW1 + (size_t)i * H : J.oW2 + (size_t)(i - J.F1) * H) + 4 * tx;
#pragma unroll
    for (int c = 0; c < 4; ++c) dst[c] = acc[q][c];
  }
  if (bias) {
#pragma unroll
    for (int c = 0; c < 4; ++c) part[J.ob + 4 * tx + c] = bs[c];
  }
}

__device__ __forceinline__ void adam(float gi, float& m, float& v, float& theta, float lr, float c1, float c2) {
  const float mi = 0.9f * m + 0.1f * gi;
  const float vi = 0.999f * v + 0.001f * gi * gi;
  m = mi;
  v = vi;
  const float mh = mi / c1, vh = vi / c2;
  theta -= lr * mh / (sqrtf(vh) + 1e-8f);
}

// The chunks' sums in order: 8 threads per parameter take consecutive ranges
// of chunks, then the 8 in order.  grad (or null) receives the gradient; an
// Adam step follows where theta is given.  One more block totals the loss.
struct SumArgs {
  int32_t chunks;
  int64_t n_params;
  const float* part;
  float* grad;
  float *theta, *m, *v;
  float lr, c1, c2;
  int32_t n, n_graphs;
  const int32_t* gsize;
  const double *lp, *lm;
  double* loss;                  // device, or null
};

__global__ void __launch_bounds__(256) k_wgrad_sum(const __grid_constant__ SumArgs a) {
  __shared__ float s[8][32];
  if (blockIdx.x == gridDim.x - 1) {
    if (a.loss) loss_total(a.n, a.n_graphs, a.gsize, a.lp, a.lm, a.loss);
    return;
  }
  const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
  const int64_t e = (int64_t)blockIdx.x * 32 + lane;
  const int span = (a.chunks + 7) / 8, c0 = q * span, c1 = min(a.chunks, c0 + span);
  float acc = 0.0f;
  if (e < a.n_params) {
#pragma unroll 8
    for (int c = c0; c < c1; ++c) acc += __ldg(a.part + (size_t)c * a.n_params + e);
  }
  s[q][lane] = acc;
  __syncthreads();
  if (q || e >= a.n_params) return;
  acc = 0.0f;
#pragma unroll
  for (int i = 0; i < 8; ++i) acc += s[i][lane];
  if (a.grad) a.grad[e] = acc;
  if (a.theta) adam(acc, a.m[e], a.v[e], a.theta[e], a.lr, a.c1, a.c2);
}

unsigned nb(int64_t count, int block = 256) { return (unsigned)((count + block - 1) / block); }

// ---------------------------------------------------------------- forward / backward

struct FeatureInfo {
  const int32_t* gid = nullptr;
  const int32_t* goff = nullptr;
  const int32_t* gmax = nullptr;
  const double* gmean = nullptr;
  const int32_t* gsize = nullptr;
  int32_t n_graphs = 1;
};

// Device buffers of one call, allocated once and used by every step.
struct Acts {
  float *X = nullptr, *dinv = nullptr, *o = nullptr, *dout = nullptr, *part = nullptr;
  std::vector<float*> Hs, Ms, dpre;   // H[l], dpre[l] for l = 0..L;  M[l] for l = 1..L (index l-1)
  float *S[2] = {nullptr, nullptr}, *T[2] = {nullptr, nullptr};
  double *lp = nullptr, *lm = nullptr, *loss = nullptr;
  int32_t chunk = 0, chunks = 0;
};

// picks the kernel of the graph's weight storage and launches it over the node tiles
#define DECO_LAUNCH_TILES(kernel, g, H, smem, st, args)                                                      \
  do {                                                                                                       \
    auto fn_ = (g)->wmode == W_UNIT ? kernel<W_UNIT> : (g)->wmode == W_SIGN ? kernel<W_SIGN> : kernel<W_GENERAL>; \
    DECO_CUDA_TRY(allow_smem(fn_));                                                                          \
    fn_<<<nb((g)->n, LTILE), 4 * (H), smem, st>>>(args);                                                     \
    DECO_CUDA_TRY(cudaGetLastError());                                                                       \
  } while (0)

// buffers, features and inverse degrees; `train`: also what the backward pass needs
int prepare_acts(const deco_mpnn* m, const deco_graph* g, const FeatureInfo& fi, uint64_t feat_seed, bool train,
                 Scratch& s, Acts& a, cudaStream_t st) {
  const int32_t n = g->n, H = m->hidden, L = m->layers;
  const size_t nh = sizeof(float) * (size_t)n * H;
  int rc;
  if ((rc = s.alloc(&a.X, sizeof(float) * (size_t)n * F_IN)) || (rc = s.alloc(&a.dinv, sizeof(float) * n))) return rc;
  a.Hs.assign(L + 1, nullptr);
  a.Ms.assign(L, nullptr);
  a.dpre.assign(L + 1, nullptr);
  if (train) {
    for (int l = 0; l <= L; ++l) {
      if ((rc = s.alloc(&a.Hs[l], nh)) || (rc = s.alloc(&a.dpre[l], nh))) return rc;
      if (l < L && (rc = s.alloc(&a.Ms[l], nh))) return rc;
    }
    for (int i = 0; i < 2; ++i)
      if ((rc = s.alloc(&a.S[i], nh)) || (rc = s.alloc(&a.T[i], nh))) return rc;
    // at most 1024 chunks, of at least 256 nodes: enough blocks, and partial sums that stay small
    a.chunk = std::max(256, (n + 1023) / 1024);
    a.chunks = (n + a.chunk - 1) / a.chunk;
    if ((rc = s.alloc(&a.o, sizeof(float) * n)) || (rc = s.alloc(&a.dout, sizeof(float) * n)) ||
        (rc = s.alloc(&a.part, sizeof(float) * (size_t)a.chunks * m->n_params)) ||
        (rc = s.alloc(&a.lp, sizeof(double) * fi.n_graphs)) || (rc = s.alloc(&a.lm, sizeof(double) * fi.n_graphs)) ||
        (rc = s.alloc(&a.loss, sizeof(double))))
      return rc;
  } else {
    // an inference keeps two layers' activations (none of the last)
    float* two[2] = {nullptr, nullptr};
    if ((rc = s.alloc(&two[0], nh)) || (L > 1 && (rc = s.alloc(&two[1], nh)))) return rc;
    for (int l = 0; l < L; ++l) a.Hs[l] = two[l & 1];
  }
  const double mean = g->n ? (double)g->deg_s1 / (double)g->n : 1.0;
  k_features<<<nb(n), 256, 0, st>>>(n, g->deg, fi.gid, fi.goff, fi.gmax, fi.gmean, g->max_deg, mean,
                                    (uint32_t)feat_seed, (uint32_t)(feat_seed >> 32), a.X, a.dinv);
  DECO_CUDA_TRY(cudaGetLastError());
  return DECO_OK;
}

// h (or null) receives tanh(o); with labels z the loss sums are formed too
int forward(const deco_mpnn* m, const deco_graph* g, const FeatureInfo& fi, bool bf16, const Acts& a,
            const uint8_t* z, float* h, cudaStream_t st) {
  const int32_t n = g->n, H = m->hidden, L = m->layers;
  const Layout lo = layout(H, L);
  const float* th = m->theta;
  for (int l = 0; l <= L; ++l) {
    LayerArgs p{};
    p.n = n;
    p.H = H;
    p.A = CsrView{g->col_idx, g->col_sw, g->w};
    p.bf16 = bf16 ? 1 : 0;
    p.post = a.Hs[l];
    if (l == 0) {
      p.F1 = F_IN;
      p.in1 = a.X;
      p.W1 = th + lo.W0;
      p.b = th + lo.b0;
      p.n_graphs = fi.n_graphs;
      if (z) { p.zlp = a.lp; p.zlm = a.lm; }
    } else {
      p.F1 = H;
      p.in1 = a.Hs[l - 1];
      p.row_ptr = g->row_ptr;
      p.dinv = a.dinv;
      p.W1 = th + lo.Ws[l - 1];
      p.W2 = th + lo.Wn[l - 1];
      p.b = th + lo.b[l - 1];
      p.agg = a.Ms[l - 1];
    }
    if (l == L) {
      p.head.wo = th + lo.wo;
      p.head.bo = th + lo.bo;
      p.head.o = a.o;
      p.head.h = h;
      p.head.z = z;
      p.head.gid = fi.gid;
      p.head.lp = a.lp;
      p.head.lm = a.lm;
    }
    const int K = p.F1 + (l ? H : 0);
    const size_t smem = sizeof(float) * ((size_t)K * H + (size_t)LTILE * (K + 4));
    DECO_LAUNCH_TILES(k_layer, g, H, smem, st, p);
  }
  return DECO_OK;
}

// gradients of the loss whose sums `forward` formed: into grad (or null), an
// Adam step when adam_t > 0, the loss into *loss_dev (device, or null)
int backward(deco_mpnn* m, const deco_graph* g, const FeatureInfo& fi, const uint8_t* z, const Acts& a, float* grad,
             float lr, int64_t adam_t, double* loss_dev, cudaStream_t st) {
  const int32_t n = g->n, H = m->hidden, L = m->layers;
  const Layout lo = layout(H, L);
  const float* th = m->theta;
  for (int l = L; l >= 0; --l) {
    BackArgs p{};
    p.n = n;
    p.H = H;
    p.row_ptr = g->row_ptr;
    p.A = CsrView{g->col_idx, g->col_sw, g->w};
    p.dinv = a.dinv;
    p.Hl = a.Hs[l];
    p.dpre = a.dpre[l];
    if (l == L) {
      p.o = a.o;
      p.wo = th + lo.wo;
      p.z = z;
      p.gid = fi.gid;
      p.gsize = fi.gsize;
      p.lp = a.lp;
      p.lm = a.lm;
      p.n_graphs = fi.n_graphs;
      p.dout = a.dout;
    } else {
      p.S = a.S[(l + 1) & 1];
      p.T = a.T[(l + 1) & 1];
    }
    if (l > 0) {
      p.Ws = th + lo.Ws[l - 1];
      p.Wn = th + lo.Wn[l - 1];
      p.So = a.S[l & 1];
      p.To = a.T[l & 1];
    }
    const size_t smem = sizeof(float) * ((size_t)LTILE * (H + 4) + (l > 0 ? 2 * (size_t)H * H : 0));
    DECO_LAUNCH_TILES(k_back, g, H, smem, st, p);
  }
  WgradArgs w{};
  w.n = n;
  w.H = H;
  w.chunk = a.chunk;
  w.n_jobs = L + 1;
  w.n_params = m->n_params;
  const int rows = WG_THREADS / (H / 4) * 8;   // weight rows of one pass
  w.passes = (2 * H + rows - 1) / rows;
  w.job[0] = WgradJob{a.X, nullptr, a.dpre[0], F_IN, 0, lo.W0, 0, lo.b0};
  for (int l = 1; l <= L; ++l)
    w.job[l] = WgradJob{a.Hs[l - 1], a.Ms[l - 1], a.dpre[l], H, H, lo.Ws[l - 1], lo.Wn[l - 1], lo.b[l - 1]};
  w.HL = a.Hs[L];
  w.dout = a.dout;
  w.owo = lo.wo;
  w.obo = lo.bo;
  w.part = a.part;
  const size_t wsm = sizeof(float) * std::max<size_t>((size_t)WG_TILE * (std::min(2 * H, rows) + 12 + H), WG_THREADS);
  DECO_CUDA_TRY(allow_smem(k_wgrad_part));
  k_wgrad_part<<<dim3((unsigned)a.chunks, (unsigned)((L + 2) * w.passes)), WG_THREADS, wsm, st>>>(w);
  DECO_CUDA_TRY(cudaGetLastError());
  SumArgs sa{};
  sa.chunks = a.chunks;
  sa.n_params = m->n_params;
  sa.part = a.part;
  sa.grad = grad;
  if (adam_t > 0) {
    sa.theta = m->theta;
    sa.m = m->m;
    sa.v = m->v;
    sa.lr = lr;
    sa.c1 = 1.0f - std::pow(0.9f, (float)adam_t);
    sa.c2 = 1.0f - std::pow(0.999f, (float)adam_t);
  }
  sa.n = n;
  sa.n_graphs = fi.n_graphs;
  sa.gsize = fi.gsize;
  sa.lp = a.lp;
  sa.lm = a.lm;
  sa.loss = loss_dev;
  k_wgrad_sum<<<nb(m->n_params, 32) + 1, 256, 0, st>>>(sa);
  DECO_CUDA_TRY(cudaGetLastError());
  return DECO_OK;
}

// the loss to the host: synchronises the stream
int read_loss(const double* dev, double* host, cudaStream_t st) {
  double v = 0.0;
  DECO_CUDA_TRY(cudaMemcpyAsync(&v, dev, sizeof(double), cudaMemcpyDeviceToHost, st));
  DECO_CUDA_TRY(cudaStreamSynchronize(st));
  *host = v;
  return DECO_OK;
}

int check_model(const deco_mpnn* m) {
  if (!m) { set_error("model is NULL"); return DECO_ERR_ARG; }
  return DECO_OK;
}

}  // namespace

// Batch side-information for the features and the per-graph loss (batch.cu).
namespace deco {
int batch_feature_info(const deco_batch* b, const deco_graph** g, const int32_t** gid, const int32_t** goff,
                       const int32_t** gmax, const double** gmean, const int32_t** gsize, int32_t* n_graphs);
}

static int resolve(const deco_graph* g, const deco_batch* b, const deco_graph** G, FeatureInfo* fi) {
  if ((g == nullptr) == (b == nullptr)) { set_error("pass exactly one of a graph and a batch"); return DECO_ERR_ARG; }
  *fi = FeatureInfo{};
  if (g) { *G = g; return DECO_OK; }
  return batch_feature_info(b, G, &fi->gid, &fi->goff, &fi->gmax, &fi->gmean, &fi->gsize, &fi->n_graphs);
}

extern "C" int deco_mpnn_create(int32_t hidden, int32_t layers, uint64_t seed, deco_mpnn** out) {
  clear_error();
  if (!out || hidden < 4 || hidden > 128 || hidden % 4 || layers < 1 || layers > 8) {
    set_error("need hidden in [4, 128], a multiple of 4, and 1 <= layers <= 8");
    return DECO_ERR_ARG;
  }
  deco_mpnn* m = new deco_mpnn();
  m->hidden = hidden;
  m->layers = layers;
  const Layout lo = layout(hidden, layers);
  m->n_params = lo.total;
  cudaError_t e = cudaMalloc((void**)&m->theta, sizeof(float) * lo.total);
  if (e == cudaSuccess) e = cudaMalloc((void**)&m->m, 2 * sizeof(float) * lo.total);   // both moments
  if (e == cudaSuccess) e = cudaMemset(m->m, 0, 2 * sizeof(float) * lo.total);
  if (e == cudaSuccess) m->v = m->m + lo.total;
  if (e != cudaSuccess) {
    cudaFree(m->theta); cudaFree(m->m);
    delete m;
    return cuda_fail(e, "model allocation");
  }
  // Xavier-uniform weight ranges: [start, end) and bound per weight matrix
  std::vector<int64_t> ranges;
  std::vector<double> bounds;
  auto add = [&](int64_t s, int64_t count, int fi, int fo) {
    ranges.push_back(s);
    ranges.push_back(s + count);
    bounds.push_back(std::sqrt(6.0 / (double)(fi + fo)));
  };
  add(lo.W0, (int64_t)F_IN * hidden, F_IN, hidden);
  for (int l = 0; l < layers; ++l) {
    add(lo.Ws[l], (int64_t)hidden * hidden, hidden, hidden);
    add(lo.Wn[l], (int64_t)hidden * hidden, hidden, hidden);
  }
  add(lo.wo, hidden, hidden, 1);
  int64_t* dr = nullptr;
  double* db = nullptr;
  e = cudaMalloc((void**)&dr, sizeof(int64_t) * ranges.size());
  if (e == cudaSuccess) e = cudaMalloc((void**)&db, sizeof(double) * bounds.size());
  if (e == cudaSuccess) e = cudaMemcpy(dr, ranges.data(), sizeof(int64_t) * ranges.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(db, bounds.data(), sizeof(double) * bounds.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    k_init_params<<<nb(lo.total), 256>>>(lo.total, dr, db, (int32_t)bounds.size(), (uint32_t)seed,
                                         (uint32_t)(seed >> 32), m->theta);
    e = cudaDeviceSynchronize();
  }
  cudaFree(dr);
  cudaFree(db);
  if (e != cudaSuccess) {
    cudaFree(m->theta); cudaFree(m->m);
    delete m;
    return cuda_fail(e, "model initialisation");
  }
  *out = m;
  return DECO_OK;
}

extern "C" void deco_mpnn_destroy(deco_mpnn* m) {
  if (!m) return;
  cudaFree(m->theta);
  cudaFree(m->m);
  delete m;
}

extern "C" int deco_mpnn_num_params(const deco_mpnn* m, int64_t* count) {
  clear_error();
  int rc = check_model(m);
  if (rc) return rc;
  if (!count) { set_error("count is NULL"); return DECO_ERR_ARG; }
  *count = m->n_params;
  return DECO_OK;
}

extern "C" int deco_mpnn_get_params(const deco_mpnn* m, float* host, int64_t count) {
  clear_error();
  int rc = check_model(m);
  if (rc) return rc;
  if (!host || count != m->n_params) { set_error("need a host buffer of %lld floats", (long long)m->n_params); return DECO_ERR_ARG; }
  DECO_CUDA_TRY(cudaMemcpy(host, m->theta, sizeof(float) * count, cudaMemcpyDeviceToHost));
  return DECO_OK;
}

extern "C" int deco_mpnn_set_params(deco_mpnn* m, const float* host, int64_t count) {
  clear_error();
  int rc = check_model(m);
  if (rc) return rc;
  if (!host || count != m->n_params) { set_error("need a host buffer of %lld floats", (long long)m->n_params); return DECO_ERR_ARG; }
  DECO_CUDA_TRY(cudaMemset(m->m, 0, 2 * sizeof(float) * count));
  DECO_CUDA_TRY(upload(m->theta, host, sizeof(float) * count));   // and the moments: there for every stream
  m->t = 0;
  return DECO_OK;
}

extern "C" int deco_mpnn_infer(const deco_mpnn* m, const deco_graph* g, const deco_batch* b, uint64_t feat_seed,
                               int32_t precision, float* h, void* stream) {
  clear_error();
  int rc = check_model(m);
  if (rc) return rc;
  if (!h || (rc = check_prec(precision))) { if (!rc) set_error("h is NULL"); return rc ? rc : DECO_ERR_ARG; }
  const deco_graph* G = nullptr;
  FeatureInfo fi;
  if ((rc = resolve(g, b, &G, &fi))) return rc;
  cudaStream_t st = as_stream(stream);
  Scratch s(st);
  Acts a;
  if ((rc = prepare_acts(m, G, fi, feat_seed, false, s, a, st))) return rc;
  return forward(m, G, fi, precision == DECO_PREC_BF16, a, nullptr, h, st);
}

extern "C" int deco_mpnn_loss_grad(const deco_mpnn* m, const deco_graph* g, const deco_batch* b, const uint8_t* z,
                                   uint64_t feat_seed, double* loss, float* grad, void* stream) {
  clear_error();
  int rc = check_model(m);
  if (rc) return rc;
  if (!z) { set_error("labels are NULL"); return DECO_ERR_ARG; }
  const deco_graph* G = nullptr;
  FeatureInfo fi;
  if ((rc = resolve(g, b, &G, &fi))) return rc;
  cudaStream_t st = as_stream(stream);
  Scratch s(st);
  Acts a;
  if ((rc = prepare_acts(m, G, fi, feat_seed, true, s, a, st)) || (rc = forward(m, G, fi, false, a, z, nullptr, st)))
    return rc;
  if (grad) {
    if ((rc = backward(const_cast<deco_mpnn*>(m), G, fi, z, a, grad, 0.0f, 0, a.loss, st))) return rc;
  } else {
    k_loss_reduce<<<1, 128, 0, st>>>(G->n, fi.n_graphs, fi.gsize, a.lp, a.lm, a.loss);
    DECO_CUDA_TRY(cudaGetLastError());
  }
  return loss ? read_loss(a.loss, loss, st) : DECO_OK;
}

extern "C" int deco_mpnn_train(deco_mpnn* m, const deco_graph* g, const deco_batch* b, const uint8_t* z,
                               uint64_t feat_seed, float lr, int32_t steps, double* losses, void* stream) {
  clear_error();
  int rc = check_model(m);
  if (rc) return rc;
  if (!z || !(lr > 0.0f) || steps < 0) { set_error("need labels, lr > 0 and steps >= 0"); return DECO_ERR_ARG; }
  const deco_graph* G = nullptr;
  FeatureInfo fi;
  if ((rc = resolve(g, b, &G, &fi))) return rc;
  cudaStream_t st = as_stream(stream);
  Scratch s(st);
  double* ldev = nullptr;
  if ((rc = s.alloc(&ldev, sizeof(double) * (size_t)(steps > 0 ? steps : 1)))) return rc;
  Acts a;
  if (steps > 0 && (rc = prepare_acts(m, G, fi, feat_seed, true, s, a, st))) return rc;
  for (int32_t it = 0; it < steps; ++it) {
    if ((rc = forward(m, G, fi, false, a, z, nullptr, st))) return rc;
    m->t += 1;
    if ((rc = backward(m, G, fi, z, a, nullptr, lr, m->t, ldev + it, st))) return rc;
  }
  if (losses && steps > 0) {
    DECO_CUDA_TRY(cudaMemcpyAsync(losses, ldev, sizeof(double) * steps, cudaMemcpyDeviceToHost, st));
    DECO_CUDA_TRY(cudaStreamSynchronize(st));
  }
  return DECO_OK;
}

extern "C" int deco_mpnn_train_step(deco_mpnn* m, const deco_graph* g, const deco_batch* b, const uint8_t* z,
                                    uint64_t feat_seed, float lr, double* loss, void* stream) {
  clear_error();
  int rc = check_model(m);
  if (rc) return rc;
  if (!z || !(lr > 0.0f)) { set_error("need labels and lr > 0"); return DECO_ERR_ARG; }
  const deco_graph* G = nullptr;
  FeatureInfo fi;
  if ((rc = resolve(g, b, &G, &fi))) return rc;
  cudaStream_t st = as_stream(stream);
  Scratch s(st);
  Acts a;
  if ((rc = prepare_acts(m, G, fi, feat_seed, true, s, a, st)) || (rc = forward(m, G, fi, false, a, z, nullptr, st)))
    return rc;
  m->t += 1;
  if ((rc = backward(m, G, fi, z, a, nullptr, lr, m->t, a.loss, st))) return rc;
  return loss ? read_loss(a.loss, loss, st) : DECO_OK;
}
