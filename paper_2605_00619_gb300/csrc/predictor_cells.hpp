// Host interface of the FP32 predictor with several cells in flight per SM (predictor_cells.cuh):
// its plan, its launches and the set-up of the data it reads.  The kernels of each order are a
// translation unit of their own (predictor_cells.cu compiled with AFE_ORDER = 1, 2, 3).
#pragma once

#include <cuda_runtime.h>

#include "kernels.cuh"

namespace afe {

// Time-basis constants.
struct PcRef {
  float w[4];       // Gauss-Legendre weights
  float kw[4][4];   // K1t^-1[s][t] w_t
  float kws[4];     // sum_t K1t^-1[s][t] w_t
};

// Constants of the corrector on the split M_i^-1.
struct CorrRef {
  float Z[10][10];   // face mass on the unit right triangle
  double zs[10];     // its column sums
};

// Launch plan: block shape (0: few cells, more warps each; 1: many cells), blocks per SM and
// dynamic shared memory of a block; most face slots of a cell.  blocks = 0: the cells do not fit.
struct PcPlan {
  int shape = 0;
  int blocks = 0;
  size_t smem = 0;
  int Fmax = 0;
};

// What the plan needs to know of a set of cells: maxima of their nodes, sub-tets and face slots, and the
// shared memory the most demanding one asks for by block shape.  Sets merge by maxima, so a union
// fits whenever its parts do.  (The corrector's shared memory is a sum of two maxima, of nodes and of face
// slots; it stays below 140 KB for all cells that the gather slots admit, because a closed surface of f
// triangles has f / 2 + 2 vertices and more nodes: at N = 3 f <= N_i / 4.5.)
struct PcCells {
  int Nmax = 0, Smax = 0, Fmax = 0;
  size_t need[2] = {0, 0};
};
template <int N>
void pc_add_cell(int n, int s, int ns, PcCells* q);

// Plan for `cells` cells (`viscous`: every one with viscous fluxes) with the properties q on n_sm SMs.
template <int N>
cudaError_t pc_plan(int device, int n_sm, int64_t cells, bool viscous, const PcCells& q, PcPlan* out);

// Launches the kernel for the kinds of cells that may be present.
template <int N>
void pc_launch(const PcPlan& plan, const Batch& b, const PcRef& ref, bool inviscid, bool viscous, int diag, int n_sm,
               cudaStream_t st);

// The corrector on the split M_i^-1 for cells of up to Nmax nodes and Fmax face slots.
template <int N>
void pc_correct(const Batch& b, const CorrRef& ref, int Nmax, int Fmax, cudaStream_t st);

// Bytes of the gather blocks of a mesh, and the set-up of m.m16 and m.gat (of m.gat alone).
size_t pc_gather_bytes(const DevMesh& m, int64_t n_subtets, int np, int nf);
void pc_set_up(const DevMesh& m, int np, int nf, int grid, cudaStream_t st);
void pc_gather_set_up(const DevMesh& m, int np, int nf, int grid, cudaStream_t st);

}  // namespace afe
