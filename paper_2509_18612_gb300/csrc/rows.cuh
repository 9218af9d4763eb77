// Row-vector form of the persistent on-chip kernel (rows.cu): parameter
// blocks, cost estimate and host helpers.
#pragma once

#include <stdint.h>

#include "deco_internal.cuh"

namespace deco {

struct RowsGraph {
  int32_t n, ld, C;
  int32_t nslices, list16, wts16;
  const uint4* image;
  const int32_t* order;
  const float* dnet;
  void* y;                    // n x ld iterate in global memory (in/out)
  float* v;                   // n x ld momentum or null (a batched launch: its scratch, zeroed by the kernel)
  const float* alpha_cols;    // per column or null
  const int32_t* steps_cols;  // per column or null
};

struct RowsParams {
  RowsGraph g0;                // the graph of a single-graph launch (graphs == null)
  const RowsGraph* graphs;     // device array of a batched launch, or null
  const int2* items;           // batched launch: (graph, first column) per item
  int32_t lpr, threads;
  uint32_t smem;               // dynamic shared memory of the launch
  int32_t steps;
  const int32_t* steps_dev;    // device value bounding the steps (min with `steps`), or null
  float alpha, afac, mu;
  int32_t objective;
  int32_t load_v, store_v;
  int32_t* flag;
};

constexpr int ROWS_MAX_LPR = 8;

// shared memory of a launch: the replicas, image, (lap) net degrees and (mom) momentum
size_t rows_smem_bytes(const RowsImage& im, int prec, bool lap, bool mom);
// a lower bound of it (gradients with net degrees, momentum) over all widths, known without the image
size_t rows_smem_least(int32_t n, int64_t nnz, int prec, int wmode);
// sizes and counts of the images of rows [row0, row0 + n) for every lpr, nothing uploaded
void rows_measure(const int32_t* row_ptr, const float* w, int wmode, int32_t row0, int32_t n,
                  std::vector<RowsImage>* out);
// one image: its sizes and its words (table, lists, weights, order), nothing uploaded
void rows_build(const int32_t* row_ptr, const int32_t* col, const float* w, int wmode, int32_t row0, int32_t n,
                int lpr, RowsImage* im, std::vector<uint32_t>* words);
int rows_image(deco_graph* g, int lpr, const RowsImage** out);   // built once and kept with the graph
// cycles of one step of one CTA that has its SM to itself, and the shared-memory cycles among them; registers: of the
// form with a row's data in registers
double rows_cycles(const RowsImage& im, bool registers, double* pipe);
int rows_threads(int32_t n, int lpr);
// threads of an SM: 1024 leave 64 registers, enough but for 8 columns with their own step sizes and budgets
constexpr int rows_max_threads(int prec, bool percol) { return prec == DECO_PREC_BF16 && percol ? 512 : 1024; }
RowsGraph rows_graph(const RowsImage& im);
int launch_rows(const RowsParams& p, int n_items, int prec, int wmode, cudaStream_t st);
// the form with a row's data in registers (rows_reg.cu): one graph, a slice per warp, at most 32 entries a row, no
// general weights, the same step size and budget for every column
bool rows_reg_fits(const RowsImage& im, int wmode);
size_t rows_reg_smem_bytes(const RowsImage& im);
int launch_rows_reg(const RowsParams& p, const RowsImage& im, int n_items, int prec, int wmode, cudaStream_t st);

}  // namespace deco
