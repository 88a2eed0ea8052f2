// Host interface of the FP64 predictor with the M_i^-1 product on the tensor cores
// (predictor_f64.cuh): plan, launches and set-up.  The kernels of each order are a translation
// unit of their own (predictor_f64.cu compiled with AFE_ORDER = 1, 2, 3).
#pragma once

#include <cuda_runtime.h>

#include "kernels.cuh"

namespace afe {

// Time-basis constants.
struct PdRef {
  double w[4];      // Gauss-Legendre weights
  double kw[4][4];  // K1t^-1[s][t] w_t
  double kws[4];    // sum_t K1t^-1[s][t] w_t
  // digits of S^ and of S^ transposed (rows m, columns (d, j)), 16 x 16 tiles of 512 words, for
  // |entries| < 2^sexp
  const uint32_t *sdig, *sdig_t;
  int sexp;
};

// Words of one of the two digit tables of S^, and the tables (host).
int pd_stiffness_words(int N);
int pd_stiffness_digits(const RefData& ref, bool transposed, uint32_t* out);  // returns the exponent

// Blocks per SM (0: the cells do not fit) and dynamic shared memory of a block.
struct PdPlan {
  int blocks = 0;
  size_t smem = 0;
};

template <int N>
cudaError_t pd_plan(int device, int Nmax, int Smax, int Fmax, PdPlan* out);

template <int N>
void pd_launch(const PdPlan& plan, const Batch& b, const PdRef& ref, bool inviscid, bool viscous, int diag, int n_sm,
               cudaStream_t st);

// The corrector on the digits of M_i^-1, for cells of up to Nmax nodes.
template <int N>
void pd_correct(const Batch& b, const RefData* ref, int Nmax, cudaStream_t st);

// Digit blocks of M_i^-1 (m.m16) from m.minv64.
void pd_set_up(const DevMesh& m, int grid, cudaStream_t st);

}  // namespace afe
