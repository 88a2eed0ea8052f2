// Device kernels of the ADER-AFE-DG step (sm_103a).  Included by afe.cu only.
//
// Layouts (all in HBM, resident for the life of a mesh handle):
//   u        [n_nodes][5] FP64 master state, node-major, contiguous per cell
//   minv     per cell a dense N_i x N_i block (symmetric), FP64 or FP32 copy
//   A        [T][Np] cell-local node of every sub-tet node (uint16)
//   geo      [T][10] adj(J_ik) (row-major, = det J J^-1) and det J_ik (FP64)
//   slot_*   one entry per cell-boundary sub-triangle ("face slot"), cell-major
// Per-step intermediates (Real = double or float):
//   vol      [n_nodes][5]            volume term of the corrector
//   slot_q   [n_slots][Nf][5]        time-integrated predictor at the face nodes
//   slot_fn  [n_slots][Nf][5]        time-integrated flux . (own outward normal)
//   slot_G   [n_slots][Nf][5]        Rusanov flux, own-side orientation
#pragma once

#include <cstdint>

#include "refelem.hpp"
#include "topology.hpp"

namespace afe {

constexpr int np_of(int N) { return (N + 1) * (N + 2) * (N + 3) / 6; }
constexpr int nf_of(int N) { return (N + 1) * (N + 2) / 2; }

enum FlagIndex { F_NONCONV = 0, F_NONFINITE = 1, F_TROUBLED = 2, F_ITERSUM = 3, F_TIMEOUT = 4, F_COUNT = 8 };

struct DevMesh {
  int N;
  int64_t C, n_nodes, n_slots, n_groups;
  int Nmax, Smax;
  const int64_t* node_ptr;
  const int64_t* sub_ptr;
  const int64_t* slot_ptr;
  const int64_t* minv_ptr;
  const uint16_t* A;
  const double* geo;
  unsigned char* sub32;  // packed FP32 sub-tet records, reduced-precision path only
  const int64_t* inc_ptr;
  const uint32_t* inc;
  const int32_t* slot_cell;
  const uint16_t* slot_sub;
  const uint8_t* slot_loc;
  const uint16_t* slot_node;
  const double* slot_geo;
  const int32_t* slot_nbr;
  const int64_t* finc_ptr;
  const uint32_t* finc;
  const int64_t* group_ptr;
  const int2* group_pair;  // own-side slot and its partner (-1: domain boundary) of every sub-triangle
  const double* cell_vol;
  const double* cell_h;
  const double* cell_hv;  // length in the viscous term of the time step (cell_h or the sub-tet length)
  double* wvec;
  double* minv64;
  float* minv32;
  uint32_t* m16;       // M_i^-1 as pairs of FP16 values (reduced precision) or digits, in matrix-fragment
                       // order, behind the offsets of the cells' blocks (see m16_block)
  unsigned char* gat;  // per cell: gather lists and face data of the reduced-precision predictor
  double* u;
  void* vol;
  void* slot_q;
  void* slot_fn;
  void* slot_G;
  int32_t* iters;
  double* beta;
  double* mu;     // per-cell dynamic viscosity mu_i (physical + artificial)
  double* means;  // [C][5] density, velocity and sound speed of the cell means
  double* dt;     // device scalars: time step of the current step, its inverse rounded to FP32, and the
                  // face fluxes' viscous constants (see ViscFace)
  double* tacc;   // device scalar: accumulated time
  unsigned long long* maxbits;
  int* flags;
  int* work;      // work counters of the persistent predictors (three), blocks done of the CFL launch
  double* qbar_diag;
  // physics
  double gamma, Rgas, cv, cfl, m1, mu0, Pr, kappa0, tol, h_min;
  int picard_max, limiter, eq;
  int first_wait_polls;  // poll limit of the FP32 predictor's first bounded wait per cell
};

// A set of meshes stepped by one launch per stage (one mesh is a batch of one).  The whole
// table travels as one __grid_constant__ kernel parameter (about 31 KB, below the 32 KB
// parameter limit), so every field read stays a constant-bank load as with a single DevMesh
// passed by value, and a captured graph node carries its own copy of the table.
constexpr int kMaxBatch = 64;
struct Batch {
  int nh;                        // members in use
  int Nmax, Smax;                // maxima over the members (shared-memory layout)
  int ring_cap;                  // FP32 predictor: most M_i^-1 ring stages (0: as many as fit)
  int narrow;                    // FP32 predictor: 1 = narrow right-hand-side chunks everywhere
  int pad;
  int* work;                     // work counters of the persistent predictors (three), blocks done of the CFL launch
  const int32_t* order;          // global cells in the order the predictor takes them (NULL: index order)
  int64_t cpre[kMaxBatch + 1];   // prefix sums of the members' cells
  int64_t gpre[kMaxBatch + 1];   // prefix sums of the members' polygonal faces
  DevMesh tab[kMaxBatch];
};

// Member holding global item x of a prefix-sum array (largest h with pre[h] <= x).
__device__ __forceinline__ int batch_find(const int64_t* __restrict__ pre, int nh, int64_t x) {
  int lo = 0, hi = nh - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (pre[mid] <= x) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

__device__ __forceinline__ double cell_kappa(const DevMesh& m, double mu_i) {
  return m.kappa0 >= 0.0 ? m.kappa0 : mu_i * m.gamma * m.cv / m.Pr;
}

// Physical flux F_e(Q, grad Q) of Sec. 2: F[e][var].  gq[e][var] = dQ_var/dx_e (only read
// when visc).  sigma = (p + 2/3 mu div v) I - mu (grad v + grad v^T); energy flux
// v . (rho E I + sigma) - kappa grad T, T = p / (rho R).
template <typename Real>
__device__ __forceinline__ void phys_flux(const Real* Q, const Real (*gq)[5], bool visc, Real mu, Real kap,
                                          Real gam, Real Rg, Real F[3][5]) {
  const Real rho = Q[0];
  const Real ir = Real(1) / rho;
  const Real v[3] = {Q[1] * ir, Q[2] * ir, Q[3] * ir};
  const Real vv = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
  const Real p = (gam - Real(1)) * (Q[4] - Real(0.5) * rho * vv);
  Real sig[3][3] = {{p, 0, 0}, {0, p, 0}, {0, 0, p}};
  Real heat[3] = {0, 0, 0};
  if (visc) {
    Real dv[3][3];  // dv[e][a] = d v_a / d x_e
#pragma unroll
    for (int e = 0; e < 3; ++e)
#pragma unroll
      for (int a = 0; a < 3; ++a) dv[e][a] = (gq[e][1 + a] - v[a] * gq[e][0]) * ir;
    const Real div = dv[0][0] + dv[1][1] + dv[2][2];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
#pragma unroll
      for (int e = 0; e < 3; ++e) sig[a][e] -= mu * (dv[e][a] + dv[a][e]);
      sig[a][a] += Real(2.0 / 3.0) * mu * div;
    }
#pragma unroll
    for (int e = 0; e < 3; ++e) {
      const Real dp = (gam - Real(1)) *
                      (gq[e][4] - Real(0.5) * vv * gq[e][0] - rho * (v[0] * dv[e][0] + v[1] * dv[e][1] + v[2] * dv[e][2]));
      const Real dT = (dp * ir - p * gq[e][0] * ir * ir) / Rg;
      heat[e] = kap * dT;
    }
  }
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    F[e][0] = Q[1 + e];
#pragma unroll
    for (int a = 0; a < 3; ++a) F[e][1 + a] = Q[1 + a] * v[e] + sig[a][e];
    F[e][4] = Q[4] * v[e] + v[0] * sig[0][e] + v[1] * sig[1][e] + v[2] * sig[2][e] - heat[e];
  }
}

// A cell's block of M_i^-1 in fragment order.
__device__ __forceinline__ uint32_t* m16_block(const DevMesh& m, int64_t c) {
  return m.m16 + reinterpret_cast<const int64_t*>(m.m16)[c];
}

__device__ __forceinline__ void store_dt(const DevMesh& m, double dt) {
  m.dt[0] = dt;
  m.dt[1] = (double)(float)(1.0 / dt);
}
// max(4 mu / 3, kappa / c_v) = max(mu factor, least): factor = 4/3, least = kappa / c_v with kappa given,
// factor = max(4/3, gamma / Pr), least = 0 with kappa = mu gamma c_v / Pr.
struct ViscFace {
  double factor, least;
};

// Block-wide max of two values (blockDim.x a multiple of 32, <= 1024).
__device__ __forceinline__ void block_max2(double& a, double& b, double* sh /* >= 64 */) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a = fmax(a, __shfl_xor_sync(0xffffffffu, a, o));
    b = fmax(b, __shfl_xor_sync(0xffffffffu, b, o));
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
  __syncthreads();
  if (l == 0) {
    sh[w] = a;
    sh[32 + w] = b;
  }
  __syncthreads();
  a = l < nw ? sh[l] : 0.0;
  b = l < nw ? sh[32 + l] : 0.0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a = fmax(a, __shfl_xor_sync(0xffffffffu, a, o));
    b = fmax(b, __shfl_xor_sync(0xffffffffu, b, o));
  }
}

// ----------------------------------------------------------------------------------------
// Set-up (FP64): cell mass matrices M_i = sum_k |J_ik| A_k^T M^ A_k (Sec. 4.4), written
// into the per-cell dense blocks, and w_i = M_i 1.  One block per cell; sub-tets are added
// in order (within one sub-tet the gather A_k is injective, so there is no write conflict).
static __global__ void assemble_mass_kernel(DevMesh m, const RefData* __restrict__ ref) {
  const int Np = ref->Np;
  for (int64_t c = blockIdx.x; c < m.C; c += gridDim.x) {
    const int64_t n0 = m.node_ptr[c];
    const int Ni = (int)(m.node_ptr[c + 1] - n0);
    double* M = m.minv64 + m.minv_ptr[c];
    const int LD = minv_ld(Ni);
    for (int64_t e = threadIdx.x; e < m.minv_ptr[c + 1] - m.minv_ptr[c]; e += blockDim.x) M[e] = 0.0;
    __syncthreads();
    for (int64_t k = m.sub_ptr[c]; k < m.sub_ptr[c + 1]; ++k) {
      const double det = m.geo[k * 10 + 9];
      const uint16_t* Ak = m.A + k * Np;
      for (int e = threadIdx.x; e < Np * Np; e += blockDim.x) {
        const int j = e / Np, l = e % Np;
        M[(int64_t)Ak[j] * LD + Ak[l]] += det * ref->M[j][l];
      }
      __syncthreads();
    }
    for (int n = threadIdx.x; n < Ni; n += blockDim.x) {
      double s = 0.0;
      for (int l = 0; l < Ni; ++l) s += M[(int64_t)n * LD + l];
      m.wvec[n0 + n] = s;
    }
    __syncthreads();
  }
}

// In-place inverse of each cell's SPD mass matrix by tiled Gauss-Jordan elimination in FP64
// (no pivoting is needed for SPD matrices; every pivot block is a Schur complement of an
// SPD matrix).  One block of 256 threads per cell, 32 x 32 tiles staged in shared memory.
// A non-positive pivot raises flags[F_NONFINITE].
static __global__ void __launch_bounds__(256) invert_spd_kernel(DevMesh m) {
  constexpr int B = 32;
  __shared__ double sD[B][B + 1];
  __shared__ double sX[B][B + 1];
  __shared__ double sY[B][B + 1];
  __shared__ double sPiv;
  const int tid = threadIdx.x;
  for (int64_t c = blockIdx.x; c < m.C; c += gridDim.x) {
    const int n = (int)(m.node_ptr[c + 1] - m.node_ptr[c]);
    const int LD = minv_ld(n);
    double* A = m.minv64 + m.minv_ptr[c];
    const int T = (n + B - 1) / B;
    auto load = [&](double (*dst)[B + 1], int ib, int jb, bool ident) {
      for (int e = tid; e < B * B; e += blockDim.x) {
        const int r = e / B, q = e % B;
        const int gr = ib * B + r, gq = jb * B + q;
        double v = (ident && r == q) ? 1.0 : 0.0;
        if (gr < n && gq < n) v = A[(int64_t)gr * LD + gq];
        dst[r][q] = v;
      }
    };
    auto store = [&](double (*src)[B + 1], int ib, int jb) {
      for (int e = tid; e < B * B; e += blockDim.x) {
        const int r = e / B, q = e % B;
        const int gr = ib * B + r, gq = jb * B + q;
        if (gr < n && gq < n) A[(int64_t)gr * LD + gq] = src[r][q];
      }
    };
    for (int kb = 0; kb < T; ++kb) {
      // 1. invert the diagonal tile (padding rows/cols act as identity)
      load(sD, kb, kb, true);
      __syncthreads();
      for (int p = 0; p < B; ++p) {
        if (tid == 0) {
          const double piv = sD[p][p];
          if (!(piv > 0.0)) atomicOr(&m.flags[F_NONFINITE], 2);
          sPiv = 1.0 / piv;
        }
        __syncthreads();
        const double ip = sPiv;
        // row p scaled; other rows eliminated (classic in-place sweep).  Every thread reads
        // the pivot row and column entries it needs before any entry is overwritten.
        double colp[4], rowp[4];
        int cnt = 0;
        for (int e = tid; e < B * B; e += blockDim.x, ++cnt) {
          colp[cnt] = sD[e / B][p];
          rowp[cnt] = sD[p][e % B];
        }
        __syncthreads();
        cnt = 0;
        for (int e = tid; e < B * B; e += blockDim.x, ++cnt) {
          const int r = e / B, q = e % B;
          const double arp = colp[cnt], apq = rowp[cnt];
          if (r == p) {
            sD[r][q] = (q == p) ? ip : apq * ip;
          } else {
            // new a_rq = a_rq - a_rp a_pq / a_pp ; new a_rp = -a_rp / a_pp
            sD[r][q] = (q == p) ? -arp * ip : sD[r][q] - arp * apq * ip;
          }
        }
        __syncthreads();
      }
      // 2. row panel: A[K, J] <- Dinv A[K, J]
      for (int jb = 0; jb < T; ++jb) {
        if (jb == kb) continue;
        load(sX, kb, jb, false);
        __syncthreads();
        for (int e = tid; e < B * B; e += blockDim.x) {
          const int r = e / B, q = e % B;
          double s = 0.0;
#pragma unroll 8
          for (int k = 0; k < B; ++k) s += sD[r][k] * sX[k][q];
          sY[r][q] = s;
        }
        __syncthreads();
        store(sY, kb, jb);
        __syncthreads();
      }
      // 3. trailing update: A[I, J] -= A[I, K] A[K, J]
      for (int ib = 0; ib < T; ++ib) {
        if (ib == kb) continue;
        load(sY, ib, kb, false);  // A[I, K] (not yet updated)
        for (int jb = 0; jb < T; ++jb) {
          if (jb == kb) continue;
          load(sX, kb, jb, false);  // updated row panel
          __syncthreads();
          for (int e = tid; e < B * B; e += blockDim.x) {
            const int r = e / B, q = e % B;
            const int gr = ib * B + r, gq = jb * B + q;
            if (gr < n && gq < n) {
              double s = 0.0;
#pragma unroll 8
              for (int k = 0; k < B; ++k) s += sY[r][k] * sX[k][q];
              A[(int64_t)gr * LD + gq] -= s;
            }
          }
          __syncthreads();
        }
        // 4. column panel: A[I, K] <- -A[I, K] Dinv
        for (int e = tid; e < B * B; e += blockDim.x) {
          const int r = e / B, q = e % B;
          const int gr = ib * B + r, gq = kb * B + q;
          if (gr < n && gq < n) {
            double s = 0.0;
#pragma unroll 8
            for (int k = 0; k < B; ++k) s += sY[r][k] * sD[k][q];
            A[(int64_t)gr * LD + gq] = -s;
          }
        }
        __syncthreads();
      }
      // 5. diagonal tile
      store(sD, kb, kb);
      __syncthreads();
    }
  }
}

// Symmetrise in FP64.
static __global__ void symmetrize_kernel(DevMesh m) {
  for (int64_t c = blockIdx.x; c < m.C; c += gridDim.x) {
    const int n = (int)(m.node_ptr[c + 1] - m.node_ptr[c]);
    const int LD = minv_ld(n);
    double* A = m.minv64 + m.minv_ptr[c];
    for (int64_t e = threadIdx.x; e < (int64_t)n * n; e += blockDim.x) {
      const int r = (int)(e / n), q = (int)(e % n);
      if (q < r) continue;
      const double v = 0.5 * (A[(int64_t)r * LD + q] + A[(int64_t)q * LD + r]);
      A[(int64_t)r * LD + q] = v;
      A[(int64_t)q * LD + r] = v;
    }
  }
}

// FP32 rows of the inverses; padding (columns >= n, rows >= n) written as zeros.
static __global__ void round_rows_kernel(DevMesh m) {
  for (int64_t c = blockIdx.x; c < m.C; c += gridDim.x) {
    const int n = (int)(m.node_ptr[c + 1] - m.node_ptr[c]), LD = minv_ld(n);
    const int64_t at = m.minv_ptr[c];
    for (int64_t e = threadIdx.x; e < m.minv_ptr[c + 1] - at; e += blockDim.x) {
      const int64_t r = e / LD, q = e % LD;
      m.minv32[at + e] = (r < n && q < n) ? (float)m.minv64[at + e] : 0.f;
    }
  }
}

// ----------------------------------------------------------------------------------------
// Per-step kernels over a batch of meshes (one mesh is a batch of one).
//
// Start of a series of steps: clear every member's status flags (they then accumulate over
// the steps until the host reads them).
static __global__ void flags_clear_kernel(const __grid_constant__ Batch bt) {
  for (int h = threadIdx.x; h < bt.nh; h += blockDim.x) {
#pragma unroll
    for (int f = 0; f < F_COUNT; ++f) bt.tab[h].flags[f] = 0;
  }
}

// Sec. 4.5: cell means u_bar_i = w_i . u_i / |P_i| (w_i = M_i 1), one warp per cell, kept as what the
// detector reads of them, once per cell instead of once per neighbour: density, velocity and
// sound speed.
static __global__ void __launch_bounds__(256) cell_means_kernel(const __grid_constant__ Batch bt) {
  const int64_t gc = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (gc >= bt.cpre[bt.nh]) return;
  const int hh = batch_find(bt.cpre, bt.nh, gc);
  const DevMesh& m = bt.tab[hh];
  if (!m.limiter) return;  // warp-uniform
  const int64_t c = gc - bt.cpre[hh];
  double acc[5] = {0, 0, 0, 0, 0};
  for (int64_t n = m.node_ptr[c] + lane; n < m.node_ptr[c + 1]; n += 32) {
    const double w = m.wvec[n];
#pragma unroll
    for (int v = 0; v < 5; ++v) acc[v] += w * m.u[n * 5 + v];
  }
#pragma unroll
  for (int v = 0; v < 5; ++v)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc[v] += __shfl_xor_sync(0xffffffffu, acc[v], o);
  if (lane) return;
  const double vol = m.cell_vol[c];
  double q[5], vel[3];
#pragma unroll
  for (int v = 0; v < 5; ++v) q[v] = acc[v] / vol;
#pragma unroll
  for (int d = 0; d < 3; ++d) vel[d] = q[1 + d] / q[0];
  const double p = (m.gamma - 1.0) * (q[4] - 0.5 * q[0] * (vel[0] * vel[0] + vel[1] * vel[1] + vel[2] * vel[2]));
  double* out = m.means + c * 5;
  out[0] = q[0];
#pragma unroll
  for (int d = 0; d < 3; ++d) out[1 + d] = vel[d];
  out[4] = sqrt(m.gamma * p / q[0]);
}

// Artificial-viscosity limiter (Sec. 4.5, Eq. beta3D): beta_i from the discrete velocity
// divergence of the cell means over the faces of P_i, mu_i = mu + beta_i rho_i lambda_i h_i/(2N+1).
// One warp per cell, its lanes on the face slots: with a thread per cell the some 45 slots, each with
// its neighbour's divisions and square root in FP64, were one serial chain (limiter stage 270 us
// whatever the size of the mesh; before and after with the time step: 15^3 P3 338 and 165 us, batch of ten P2 3,676 and 3,077 us per pass).
static __global__ void __launch_bounds__(256) limiter_kernel(const __grid_constant__ Batch bt) {
  const int64_t gc = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (gc >= bt.cpre[bt.nh]) return;
  const int hh = batch_find(bt.cpre, bt.nh, gc);
  const DevMesh& m = bt.tab[hh];
  if (!m.limiter) return;  // a batch member without the limiter keeps beta = 0, mu_i = mu
  const int64_t c = gc - bt.cpre[hh];
  double own[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) own[v] = m.means[c * 5 + v];
  double div = 0.0, cmin = own[4];
  for (int64_t s = m.slot_ptr[c] + lane; s < m.slot_ptr[c + 1]; s += 32) {
    const int32_t nb = m.slot_nbr[s];
    if (nb < 0) continue;
    const double* q = m.means + (int64_t)nb * 5;
    const double* g = m.slot_geo + s * 4;
    div += g[3] * ((q[1] - own[1]) * g[0] + (q[2] - own[2]) * g[1] + (q[3] - own[3]) * g[2]);
    cmin = fmin(cmin, q[4]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    div += __shfl_xor_sync(0xffffffffu, div, o);
    cmin = fmin(cmin, __shfl_xor_sync(0xffffffffu, cmin, o));
  }
  if (lane) return;
  div /= m.cell_vol[c];
  const double b = fmin(1.0, fmax(0.0, -(div + m.m1 * cmin) / (m.m1 * cmin)));
  m.beta[c] = b;
  const double lam = sqrt(own[1] * own[1] + own[2] * own[2] + own[3] * own[3]) + own[4];
  m.mu[c] = m.mu0 + b * own[0] * lam * m.cell_h[c] / (2 * m.N + 1);
  if (b > 0.0) atomicAdd(&m.flags[F_TROUBLED], 1);
}

// FP32 value of x by truncation, from its bits (integer instructions: the FP64 pipe, conversions
// included, takes one lane or two per cycle and SM).  Relative error below 2^-23 when the result is
// true in `ok`: x is zero or its exponent lies within +-100.
__device__ __forceinline__ float f32_head(double x, bool& ok) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const int e = (hi >> 20) & 0x7ff;
  const bool zero = ((hi << 1) | lo) == 0;
  ok = ok && (zero || (unsigned)(e - 923) <= 200u);
  const unsigned bits = (unsigned)(hi & 0x80000000) | (unsigned)((e - 896) << 23) |
                        (__funnelshift_l((unsigned)lo, (unsigned)hi, 3) & 0x7fffffu);
  return zero ? 0.f : __uint_as_float(bits);
}

// CFL bound (Sec. 4.6): max over nodes of lambda + 2 lambda_v (2N+1)/h_i, one warp per cell,
// folded into the member's maximum by an integer atomicMax on the bits of a non-negative
// double (order-independent, hence deterministic).
// The bound itself is FP64 arithmetic (a division and two square roots per node), and the FP64
// pipe is what the kernel would wait for: on the 10.2 M nodes of a 32^3 P3 mesh 890 us, and 120 us as
// it stands (62 us for the state's bytes at the copy rate); 24^3 P1 95 -> 38 us.  So every node first gets an interval around its bound in FP32; only nodes
// whose upper end reaches the largest lower end seen (of the cell's nodes, and the maximum folded
// so far) can be the maximum and are evaluated in FP64.  A node whose interval is in doubt (an
// exponent out of range, a pressure that is not positive beyond its error) always is, so that
// the maximum and the report of inadmissible states are those of evaluating every node.
__device__ __forceinline__ void cfl_cell(const Batch& bt, int64_t gc, int lane) {
  const int hh = batch_find(bt.cpre, bt.nh, gc);
  const DevMesh& m = bt.tab[hh];
  const int64_t c = gc - bt.cpre[hh];
  const int64_t n0 = m.node_ptr[c], n1 = m.node_ptr[c + 1];
  const double mu_i = m.mu[c], kap = cell_kappa(m, mu_i);
  // per cell: lambda_v = max(4 mu / 3, kappa / c_v) / rho, weighted by 2 (2N+1) / h
  const double gam = m.gamma;
  const double visc =
      mu_i == 0.0 && kap == 0.0 ? 0.0 : fmax(4.0 * mu_i / 3.0, kap / m.cv) * (2.0 * (2 * m.N + 1) / m.cell_hv[c]);
  // gamma (gamma - 1) is rounded once: near gamma = 1 the difference of rounded values is off by far more than kEps
  const float vf = (float)visc, gg = (float)fma(gam, gam, -gam);
  const bool vis_ok = vf >= 0x1p-120f || visc == 0.0;  // else too small for FP32
  // interval of a node's bound: relative errors are a few 2^-23 of each term, kEps covers them
  constexpr float kEps = 0x1p-18f;
  auto interval = [&](const double (&q)[5], float& lower) {
    bool ok = true;
    const float r = f32_head(q[0], ok), a = f32_head(q[1], ok), b = f32_head(q[2], ok), d = f32_head(q[3], ok),
                e = f32_head(q[4], ok);
    const float ir = 1.f / r, m2 = (a * a + b * b + d * d) * ir;
    const float c2 = gg * ir * (e - 0.5f * m2), err = kEps * gg * ir * (fabsf(e) + m2);
    const float s = sqrtf(m2 * ir) + vf * ir;
    const float lo = sqrtf(c2 - err), up = s + sqrtf(c2 + err);
    // rho > 0, a pressure that is positive whatever the error, everything in range.  The squares of the
    // momentum lose up to 2^-148 to underflow, 2^-74 / rho of |v|: below 2^-25 c when gamma (gamma - 1)
    // rho E > 2^-80 and the pressure passes its test (c^2 > 2^-18 gamma (gamma - 1) E / rho).
    ok = ok && r > 0.f && c2 > err && c2 > 0x1p-100f && gg * (e * r) > 0x1p-80f && vis_ok && up < 1e30f && s >= 0.f;
    lower = ok ? (s + lo) * (1.f - kEps) : 0.f;
    return ok ? up * (1.f + kEps) : __int_as_float(0x7f800000);
  };
  auto load = [&](int64_t n, double (&q)[5]) {
#pragma unroll
    for (int v = 0; v < 5; ++v) q[v] = m.u[n * 5 + v];
  };
  float most = 0.f, least = 0.f;  // largest upper and lower end of this lane's nodes
  for (int64_t n = n0 + lane; n < n1; n += 32) {
    double q[5];
    load(n, q);
    float lower;
    most = fmaxf(most, interval(q, lower));
    least = fmaxf(least, lower);
  }
  least = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(least)));
  const double seen = __longlong_as_double((long long)*(volatile unsigned long long*)m.maxbits);
  const float floor_ = fmaxf(least, (float)seen * (1.f - kEps));
  if (!__any_sync(0xffffffffu, most >= floor_)) return;
  double best = 0.0, last[5] = {0, 0, 0, 0, 0};
  bool bad = false, any = false;
  for (int64_t n = n0 + lane; n < n1; n += 32) {
    double q[5];
    load(n, q);
    float lower;
    if (interval(q, lower) < floor_) continue;
    // in a uniform region every node is a candidate: a state equal to the lane's last, bit for
    // bit, has its bound already
    bool same = any;
    any = true;
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      same = same && __double_as_longlong(q[v]) == __double_as_longlong(last[v]);
      last[v] = q[v];
    }
    if (same) continue;
    const double rho = q[0], ir = 1.0 / rho;  // one division per node
    const double m2 = q[1] * q[1] + q[2] * q[2] + q[3] * q[3];
    const double p = (gam - 1.0) * (q[4] - 0.5 * m2 * ir);
    double br = sqrt(m2) * ir + sqrt(gam * p * ir) + visc * ir;
    if (!(rho > 0.0) || !(br >= 0.0) || !isfinite(br)) {  // inadmissible state: report, keep dt finite
      bad = true;
      br = 0.0;
    }
    best = fmax(best, br);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) best = fmax(best, __shfl_xor_sync(0xffffffffu, best, o));
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(&m.flags[F_NONFINITE], 1);
  if (lane == 0) atomicMax(m.maxbits, (unsigned long long)__double_as_longlong(best));
}

// What a CFL launch does once the maximum is complete: nothing, dt, or dt and the step's clock.
enum CflMode { CFL_BOUND = 0, CFL_DT = 1, CFL_STEP = 2 };

// CFL bound of every cell; the last block to finish (bt.work[3] counts them) turns the members' maxima into
// dt = CFL h_min / ((2N+1) max_bound) (Sec. 4.6), leaves the maxima zero for the next launch and
// starts the step's clock.  Launches of their own for the start of a step, dt and the clock took 6 to
// 11 us of a step (us per four steps, with them and here: 4^3 P1 541 and 495, 8^3 P2 732 and 709,
// 24^3 P1 2,429 and 2,406; 32^3 P3 within 0.1 %).
static __global__ void __launch_bounds__(256) cfl_kernel(const __grid_constant__ Batch bt, int mode) {
  const int64_t gc = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (gc < bt.cpre[bt.nh]) cfl_cell(bt, gc, threadIdx.x & 31);
  if (mode == CFL_BOUND) return;
  __shared__ int last;
  __syncthreads();  // the block's maxima are folded
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(&bt.work[3], 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int h = threadIdx.x; h < bt.nh; h += blockDim.x) {
    const DevMesh& m = bt.tab[h];
    const double mx = __longlong_as_double((long long)atomicExch(m.maxbits, 0ull));
    double dt = mx > 0.0 ? m.cfl * m.h_min / ((2 * m.N + 1) * mx) : 0.0;
    if (!(dt > 0.0)) atomicOr(&m.flags[F_NONFINITE], 4);
    store_dt(m, dt);
    if (mode == CFL_STEP) *m.tacc += dt;
  }
  if (threadIdx.x < 4) bt.work[threadIdx.x] = 0;
}

// Start of a step of a given size.
static __global__ void set_dt_kernel(const __grid_constant__ Batch bt, double dt) {
  for (int h = threadIdx.x; h < bt.nh; h += blockDim.x) {
    store_dt(bt.tab[h], dt);
    *bt.tab[h].tacc += dt;
  }
  if (threadIdx.x < 4) bt.work[threadIdx.x] = 0;
}

// ----------------------------------------------------------------------------------------
// Space-time predictor (Sec. 4.3).  Persistent: each block takes cells from a work
// counter.  Per cell, with q [N_i][Nt][5] the space-time nodal coefficients:
//   q^0 = u^  at every time node;
//   repeat:  B_{k,t}  = dt adj(J_ik) . F(q at the nodes of T_ik, time t)          (f*, g*, h*)
//            R_{k,t}  = w_t sum_d S^_d B_{k,t,d}                                     (K_d terms)
//            RHS_t    = sum_k A_k^T R_{k,t}           (fixed-order gather: deterministic)
//            Y        = M_i^-1 RHS                    (all Nt*5 columns at once)
//            q^{r+1}[n,s] = u^[n] - sum_t K1t^-1[s,t] Y[n,t]        (K_1,i^-1 = M_i^-1 (x) K1t^-1,
//                                                                      K1t^-1 psi(0) = 1)
//   until max|q^{r+1}-q^r| <= tol max(1, max|q^r|) or picard_max.
// Epilogue (Eq. TAvectors and the corrector's volume term of Sec. 4.4):
//   vol[n]     = sum_k A_k^T sum_d S^_d^T adj(J_ik) F_bar_k,  F_bar = dt sum_t w_t F(q_t)
//   slot_q     = dt sum_t w_t q_t at the face nodes
//   slot_fn    = F_bar . n at the face nodes (flux of the sub-tet owning the triangle)
// Per-block scratch in global memory (L2-resident): q, RHS, Y, B, R.
template <int N, typename Real>
__global__ void __launch_bounds__(256) predictor_kernel(DevMesh m, const RefData* __restrict__ ref, Real* scratch,
                                                        int64_t scratch_stride, int diag) {
  constexpr int NP = np_of(N), NT = N + 1, NF = nf_of(N);
  // the nodal derivative matrices stay in global memory (L1-cached) when both reference
  // matrices would not fit the static shared-memory limit (FP64 at N = 4)
  constexpr bool kDShared = 2 * 3 * NP * NP * sizeof(Real) <= 44 * 1024;
  constexpr int DS = kDShared ? NP : 1;
  __shared__ Real sS[3][NP][NP];
  __shared__ Real sD[3][DS][DS];
  __shared__ Real sK[NT][NT];
  __shared__ Real sW[NT];
  __shared__ double sred[64];
  __shared__ int64_t sCell;
  // FP32 at N = 4: the stiffness with its rows innermost, and a tile of right-hand-side rows, both read as
  // vectors (what the scalar loads of the general form are bound by; us per launch at 8^3: 11,770
  // without, 6,680 with both)
  constexpr bool kTiled = N == 4 && sizeof(Real) == 4;
  constexpr int MP = (NP + 3) / 4 * 4, CP = (NT * 5 + 3) / 4 * 4, LT = 32;
  __shared__ __align__(16) float sST[kTiled ? 3 * NP : 1][MP];
  __shared__ __align__(16) float sRT[kTiled ? LT : 1][CP];
  const int tid = threadIdx.x, nthr = blockDim.x;
  if constexpr (kTiled) {
    for (int e = tid; e < 3 * NP * MP; e += nthr) {
      const int kk = e / MP, r = e % MP;
      sST[kk][r] = r < NP ? (float)ref->S[kk / NP][r][kk % NP] : 0.f;
    }
    for (int e = tid; e < LT * CP; e += nthr) sRT[e / CP][e % CP] = 0.f;
  }
  for (int e = tid; e < 3 * NP * NP; e += nthr) {
    const int d = e / (NP * NP), r = (e / NP) % NP, q = e % NP;
    sS[d][r][q] = (Real)ref->S[d][r][q];
    if constexpr (kDShared) sD[d][r % DS][q % DS] = (Real)ref->D[d][r][q];
  }
  auto Dv = [&](int d, int j, int l) -> Real {
    if constexpr (kDShared) return sD[d][j % DS][l % DS];
    else return (Real)ref->D[d][j][l];
  };
  if (tid < NT * NT) sK[tid / NT][tid % NT] = (Real)ref->K1tinv[tid / NT][tid % NT];
  if (tid < NT) sW[tid] = (Real)ref->w[tid];
  const int Nmax = m.Nmax, Smax = m.Smax;
  Real* q = scratch + blockIdx.x * scratch_stride;
  Real* RHS = q + (int64_t)Nmax * NT * 5;
  Real* Y = RHS + (int64_t)Nmax * NT * 5;
  Real* Bf = Y + (int64_t)Nmax * NT * 5;        // [Smax][NT][3][NP][5]
  Real* Rb = Bf + (int64_t)Smax * NT * 3 * NP * 5;  // [Smax][NT][NP][5]
  const double dt = *m.dt;
  const Real gam = (Real)m.gamma, Rg = (Real)m.Rgas;
  const Real* minv = nullptr;
  __syncthreads();
  for (;;) {
    if (tid == 0) sCell = atomicAdd(m.work, 1);
    __syncthreads();
    const int64_t c = sCell;
    __syncthreads();
    if (c >= m.C) break;
    const int64_t n0 = m.node_ptr[c];
    const int Ni = (int)(m.node_ptr[c + 1] - n0);
    const int64_t k0 = m.sub_ptr[c];
    const int S = (int)(m.sub_ptr[c + 1] - k0);
    const double mu_d = m.mu[c];
    const double kap_d = cell_kappa(m, mu_d);
    const bool visc = (mu_d != 0.0) || (kap_d != 0.0);
    const Real mu = (Real)mu_d, kap = (Real)kap_d;
    if constexpr (sizeof(Real) == 8) minv = (const Real*)(m.minv64 + m.minv_ptr[c]);
    else minv = (const Real*)(m.minv32 + m.minv_ptr[c]);
    const double* uh = m.u + n0 * 5;
    for (int e = tid; e < Ni * NT * 5; e += nthr) {
      const int n = e / (NT * 5), v = e % 5;
      q[e] = (Real)uh[n * 5 + v];
    }
    __syncthreads();

    // flux pre-contraction at one (sub-tet k, time t, local node j): out[d][v] = sum_e G[d][e] F_e[v]
    auto flux_item = [&](int k, int t, int j, Real out[3][5], bool scale_dt) {
      const int64_t kg = k0 + k;
      const uint16_t* Ak = m.A + kg * NP;
      const double* g = m.geo + kg * 10;
      Real Q[5];
      const int node = Ak[j];
#pragma unroll
      for (int v = 0; v < 5; ++v) Q[v] = q[(node * NT + t) * 5 + v];
      Real gq[3][5];
      if (visc) {
        Real gx[3][5];
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
          for (int v = 0; v < 5; ++v) gx[d][v] = 0;
        for (int l = 0; l < NP; ++l) {
          const Real* ql = q + (Ak[l] * NT + t) * 5;
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const Real dd = Dv(d, j, l);
#pragma unroll
            for (int v = 0; v < 5; ++v) gx[d][v] += dd * ql[v];
          }
        }
        // grad_x = J^-T grad_xi, J^-1 = adj / det
        const Real idet = Real(1) / (Real)g[9];
#pragma unroll
        for (int e = 0; e < 3; ++e)
#pragma unroll
          for (int v = 0; v < 5; ++v)
            gq[e][v] = ((Real)g[0 * 3 + e] * gx[0][v] + (Real)g[1 * 3 + e] * gx[1][v] + (Real)g[2 * 3 + e] * gx[2][v]) * idet;
      }
      Real F[3][5];
      phys_flux<Real>(Q, gq, visc, mu, kap, gam, Rg, F);
      const Real sc = scale_dt ? (Real)dt : Real(1);
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int v = 0; v < 5; ++v)
          out[d][v] = sc * ((Real)g[d * 3 + 0] * F[0][v] + (Real)g[d * 3 + 1] * F[1][v] + (Real)g[d * 3 + 2] * F[2][v]);
    };

    int it = 0;
    bool conv = false;
    while (!conv && it < m.picard_max) {
      ++it;
      // A: B[k][t][d][j][v]
      for (int e = tid; e < S * NT * NP; e += nthr) {
        const int k = e / (NT * NP), t = (e / NP) % NT, j = e % NP;
        Real out[3][5];
        flux_item(k, t, j, out, true);
        Real* dst = Bf + ((int64_t)(k * NT + t) * 3) * NP * 5 + j * 5;
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
          for (int v = 0; v < 5; ++v) dst[d * NP * 5 + v] = out[d][v];
      }
      __syncthreads();
      // B: R[k][t][m][v] = w_t sum_d sum_j S[d][m][j] B[k][t][d][j][v]
      if constexpr (kTiled) {  // a column (k, t, v) per thread, all rows m in registers
        for (int e = tid; e < S * NT * 5; e += nthr) {
          const int kt = e / 5, v = e % 5;
          const Real* src = Bf + (int64_t)kt * 3 * NP * 5 + v;
          float acc[MP];
#pragma unroll
          for (int i = 0; i < MP; ++i) acc[i] = 0.f;
#pragma unroll 3
          for (int kk = 0; kk < 3 * NP; ++kk) {
            const float x = src[kk * 5];
#pragma unroll
            for (int i = 0; i < MP; i += 4) {
              const float4 c = *reinterpret_cast<const float4*>(&sST[kk][i]);
              acc[i] += c.x * x, acc[i + 1] += c.y * x, acc[i + 2] += c.z * x, acc[i + 3] += c.w * x;
            }
          }
          const float wt = sW[kt % NT];
#pragma unroll
          for (int i = 0; i < NP; ++i) Rb[((int64_t)kt * NP + i) * 5 + v] = wt * acc[i];
        }
      } else for (int e = tid; e < S * NT * NP * 5; e += nthr) {
        const int k = e / (NT * NP * 5), t = (e / (NP * 5)) % NT, mm = (e / 5) % NP, v = e % 5;
        const Real* src = Bf + ((int64_t)(k * NT + t) * 3) * NP * 5 + v;
        Real acc = 0;
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
          for (int j = 0; j < NP; ++j) acc += sS[d][mm][j] * src[(d * NP + j) * 5];
        Rb[e] = sW[t] * acc;
      }
      __syncthreads();
      // C: RHS[n][t][v] = sum over incidences (k, j) of node n
      for (int e = tid; e < Ni * NT * 5; e += nthr) {
        const int n = e / (NT * 5), t = (e / 5) % NT, v = e % 5;
        Real acc = 0;
        for (int64_t p = m.inc_ptr[n0 + n]; p < m.inc_ptr[n0 + n + 1]; ++p) {
          const uint32_t w = m.inc[p];
          const int k = (int)(w >> 6), j = (int)(w & 63);
          acc += Rb[((int64_t)(k * NT + t) * NP + j) * 5 + v];
        }
        RHS[e] = acc;
      }
      __syncthreads();
      // D: Y = M_i^-1 RHS (M_i^-1 symmetric: row n read as column n, coalesced)
      if constexpr (kTiled) {  // four nodes per thread against tiles of 32 right-hand-side rows
        const int LD = minv_ld(Ni);
        for (int g0 = 0; 4 * g0 < Ni; g0 += nthr) {
          const int g = g0 + tid;
          float acc[4][NT * 5];
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int c2 = 0; c2 < NT * 5; ++c2) acc[i][c2] = 0.f;
          for (int l0 = 0; l0 < Ni; l0 += LT) {
            __syncthreads();
            for (int e = tid; e < LT * NT * 5; e += nthr) {
              const int l = e / (NT * 5);
              sRT[l][e - l * NT * 5] = l0 + l < Ni ? RHS[l0 * NT * 5 + e] : 0.f;
            }
            __syncthreads();
            if (4 * g >= Ni) continue;
            const float* col = (const float*)minv + 4 * g;
#pragma unroll 2
            for (int l = 0; l < min(LT, Ni - l0); ++l) {
              const float4 a = *reinterpret_cast<const float4*>(col + (int64_t)(l0 + l) * LD);
#pragma unroll
              for (int q = 0; q < CP; q += 4) {
                const float4 r = *reinterpret_cast<const float4*>(&sRT[l][q]);
                const float rv[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
                for (int u = 0; u < 4; ++u)
                  if (q + u < NT * 5) {
                    acc[0][q + u] += a.x * rv[u];
                    acc[1][q + u] += a.y * rv[u];
                    acc[2][q + u] += a.z * rv[u];
                    acc[3][q + u] += a.w * rv[u];
                  }
              }
            }
          }
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (4 * g + i < Ni)
#pragma unroll
              for (int c2 = 0; c2 < NT * 5; ++c2) Y[(4 * g + i) * NT * 5 + c2] = acc[i][c2];
        }
      } else for (int n = tid; n < Ni; n += nthr) {
        Real acc[NT * 5];
#pragma unroll
        for (int c2 = 0; c2 < NT * 5; ++c2) acc[c2] = 0;
        const int LD = minv_ld(Ni);
        for (int l = 0; l < Ni; ++l) {
          const Real a = minv[(int64_t)l * LD + n];
          const Real* r = RHS + l * NT * 5;
#pragma unroll
          for (int c2 = 0; c2 < NT * 5; ++c2) acc[c2] += a * r[c2];
        }
#pragma unroll
        for (int c2 = 0; c2 < NT * 5; ++c2) Y[n * NT * 5 + c2] = acc[c2];
      }
      __syncthreads();
      // E: update and residual
      double res = 0.0, qmax = 0.0;
      for (int e = tid; e < Ni * NT * 5; e += nthr) {
        const int n = e / (NT * 5), s = (e / 5) % NT, v = e % 5;
        Real acc = (Real)uh[n * 5 + v];
#pragma unroll
        for (int t = 0; t < NT; ++t) acc -= sK[s][t] * Y[(n * NT + t) * 5 + v];
        const Real old = q[e];
        res = fmax(res, (double)fabs(acc - old));
        qmax = fmax(qmax, (double)fabs(old));
        q[e] = acc;
      }
      block_max2(res, qmax, sred);
      conv = res <= m.tol * fmax(1.0, qmax);
      __syncthreads();
    }
    if (tid == 0) {
      m.iters[c] = it;
      if (!conv) atomicAdd(&m.flags[F_NONCONV], 1);
    }

    // epilogue: B_bar[k][d][j][v] = sum_t w_t dt adj F(q_t) = adj F_bar  (stored in Bf)
    for (int e = tid; e < S * NP; e += nthr) {
      const int k = e / NP, j = e % NP;
      Real accb[3][5];
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int v = 0; v < 5; ++v) accb[d][v] = 0;
      for (int t = 0; t < NT; ++t) {
        Real out[3][5];
        flux_item(k, t, j, out, true);
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
          for (int v = 0; v < 5; ++v) accb[d][v] += sW[t] * out[d][v];
      }
      Real* dst = Bf + ((int64_t)k * 3) * NP * 5 + j * 5;
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int v = 0; v < 5; ++v) dst[d * NP * 5 + v] = accb[d][v];
    }
    __syncthreads();
    // R_bar[k][mm][v] = sum_d sum_j S[d][j][mm] B_bar[k][d][j][v]   (V_d = S^_d^T)
    for (int e = tid; e < S * NP * 5; e += nthr) {
      const int k = e / (NP * 5), mm = (e / 5) % NP, v = e % 5;
      const Real* src = Bf + ((int64_t)k * 3) * NP * 5 + v;
      Real acc = 0;
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int j = 0; j < NP; ++j) acc += sS[d][j][mm] * src[(d * NP + j) * 5];
      Rb[e] = acc;
    }
    __syncthreads();
    Real* vol = (Real*)m.vol;
    for (int e = tid; e < Ni * 5; e += nthr) {
      const int n = e / 5, v = e % 5;
      Real acc = 0;
      for (int64_t p = m.inc_ptr[n0 + n]; p < m.inc_ptr[n0 + n + 1]; ++p) {
        const uint32_t w = m.inc[p];
        acc += Rb[((int64_t)(w >> 6) * NP + (w & 63)) * 5 + v];
      }
      vol[(n0 + n) * 5 + v] = acc;
    }
    // face slots: q_bar and F_bar . n at every face node
    const int64_t s0 = m.slot_ptr[c];
    const int ns = (int)(m.slot_ptr[c + 1] - s0);
    Real* sq = (Real*)m.slot_q;
    Real* sfn = (Real*)m.slot_fn;
    for (int e = tid; e < ns * NF; e += nthr) {
      const int s = e / NF, a = e % NF;
      const int64_t sg = s0 + s;
      const int k = m.slot_sub[sg];
      const int j = m.slot_loc[sg * NF + a];
      const int node = m.slot_node[sg * NF + a];
      const double* g = m.slot_geo + sg * 4;
      Real qb[5] = {0, 0, 0, 0, 0}, fb[5] = {0, 0, 0, 0, 0};
      // F . n from the owning sub-tet: reuse flux_item with unit geometry is not possible,
      // so evaluate the physical flux directly.
      const int64_t kg = k0 + k;
      const uint16_t* Ak = m.A + kg * NP;
      const double* gk = m.geo + kg * 10;
      for (int t = 0; t < NT; ++t) {
        Real Q[5];
#pragma unroll
        for (int v = 0; v < 5; ++v) Q[v] = q[(node * NT + t) * 5 + v];
        Real gq[3][5];
        if (visc) {
          Real gx[3][5];
#pragma unroll
          for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int v = 0; v < 5; ++v) gx[d][v] = 0;
          for (int l = 0; l < NP; ++l) {
            const Real* ql = q + (Ak[l] * NT + t) * 5;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
              const Real dd = Dv(d, j, l);
#pragma unroll
              for (int v = 0; v < 5; ++v) gx[d][v] += dd * ql[v];
            }
          }
          const Real idet = Real(1) / (Real)gk[9];
#pragma unroll
          for (int e2 = 0; e2 < 3; ++e2)
#pragma unroll
            for (int v = 0; v < 5; ++v)
              gq[e2][v] = ((Real)gk[0 * 3 + e2] * gx[0][v] + (Real)gk[1 * 3 + e2] * gx[1][v] + (Real)gk[2 * 3 + e2] * gx[2][v]) * idet;
        }
        Real F[3][5];
        phys_flux<Real>(Q, gq, visc, mu, kap, gam, Rg, F);
        const Real wt = sW[t] * (Real)dt;
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          qb[v] += wt * Q[v];
          fb[v] += wt * ((Real)g[0] * F[0][v] + (Real)g[1] * F[1][v] + (Real)g[2] * F[2][v]);
        }
      }
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        sq[(sg * NF + a) * 5 + v] = qb[v];
        sfn[(sg * NF + a) * 5 + v] = fb[v];
      }
    }
    if (diag && m.qbar_diag) {
      for (int e = tid; e < Ni * 5; e += nthr) {
        const int n = e / 5, v = e % 5;
        double acc = 0.0;
        for (int t = 0; t < NT; ++t) acc += (double)sW[t] * (double)q[(n * NT + t) * 5 + v];
        m.qbar_diag[(n0 + n) * 5 + v] = dt * acc;
      }
    }
    __syncthreads();
  }
}

// ----------------------------------------------------------------------------------------
// Rusanov fluxes (Eq. 3.33) on the face nodes, FP64 form; one warp per polygonal face (all its
// sub-triangles, both sides).  The wave speeds are reduced over the face with warp
// shuffles; G is written for the own side and, negated, for the matched side.
template <int N, typename Real>
__global__ void face_kernel(const __grid_constant__ Batch bt) {
  constexpr int NF = nf_of(N);
  const int64_t ggw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (ggw >= bt.gpre[bt.nh]) return;
  const int h = batch_find(bt.gpre, bt.nh, ggw);
  const DevMesh& m = bt.tab[h];
  const int64_t gw = ggw - bt.gpre[h];
  const int64_t g0 = m.group_ptr[gw], g1 = m.group_ptr[gw + 1];
  const int nitems = (int)(g1 - g0) * NF;
  const Real* sq = (const Real*)m.slot_q;
  const Real* sfn = (const Real*)m.slot_fn;
  Real* sG = (Real*)m.slot_G;
  const double dt = *m.dt;
  const Real idt = Real(1.0 / dt);
  const Real gam = (Real)m.gamma;
  const int2 p_first = m.group_pair[g0];
  const int32_t ci = m.slot_cell[p_first.x];
  const int32_t cj = p_first.y >= 0 ? m.slot_cell[p_first.y] : -1;
  const double mu_i = m.mu[ci], kap_i = cell_kappa(m, mu_i);
  const double mu_j = cj >= 0 ? m.mu[cj] : mu_i, kap_j = cell_kappa(m, mu_j);
  const double h_i = m.cell_h[ci], h_j = cj >= 0 ? m.cell_h[cj] : h_i;
  // |lambda_v| = max(4 mu / 3, kappa / c_v) / rho: the coefficient once per side, then one
  // reciprocal per face node (1 / rho = dt / q_bar_rho)
  const Real cvis_i = (Real)fmax(4.0 * mu_i / 3.0, kap_i / m.cv), cvis_j = (Real)fmax(4.0 * mu_j / 3.0, kap_j / m.cv);
  const Real rdt = (Real)dt;
  Real smax = 0, vmax = 0;
  for (int e = lane; e < nitems; e += 32) {
    const int2 pair = m.group_pair[g0 + e / NF];
    const int64_t s = pair.x, ps = pair.y;
    const int a = e % NF;
    const double* g = m.slot_geo + s * 4;
    for (int side = 0; side < 2; ++side) {
      const int64_t ss = side == 0 ? s : ps;
      if (ss < 0) continue;
      const Real* Q = sq + (ss * NF + a) * 5;
      const Real rho = Q[0] * idt;
      const Real ir = Real(1) / Q[0];
      const Real v0 = Q[1] * ir, v1 = Q[2] * ir, v2 = Q[3] * ir;  // q_bar / dt ratios
      const Real p = (gam - 1) * (Q[4] * idt - Real(0.5) * rho * (v0 * v0 + v1 * v1 + v2 * v2));
      const Real vn = fabs(v0 * (Real)g[0] + v1 * (Real)g[1] + v2 * (Real)g[2]);
      const Real irho = ir * rdt;  // 1 / rho
      smax = fmax(smax, vn + sqrt(gam * p * irho));
      vmax = fmax(vmax, (side == 0 ? cvis_i : cvis_j) * irho);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    smax = fmax(smax, __shfl_xor_sync(0xffffffffu, smax, o));
    vmax = fmax(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
  }
  const Real eps = (Real)((2 * N + 1) / ((h_i + h_j) * sqrt(3.14159265358979323846 / 2.0)));
  const Real diss = Real(0.5) * (smax + Real(2) * eps * vmax);
  for (int e = lane; e < nitems * 5; e += 32) {
    const int item = e / 5, v = e % 5;
    const int2 pair = m.group_pair[g0 + item / NF];
    const int64_t s = pair.x, ps = pair.y;
    const int a = item % NF;
    const int64_t io = (s * NF + a) * 5 + v;
    if (ps < 0) {  // transmissive boundary: q+ = q-, F+ = F-
      sG[io] = sfn[io];
      continue;
    }
    const int64_t ip = (ps * NF + a) * 5 + v;
    // the matched side stores F_bar . (its own normal) = -F_bar+ . n
    const Real G = Real(0.5) * (sfn[io] - sfn[ip]) - diss * (sq[ip] - sq[io]);
    sG[io] = G;
    sG[ip] = -G;
  }
}

// FP32 value of x to nearest, by integer instructions where x is zero or normal in FP32.
__device__ __forceinline__ float f32_of(double x) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const int e = (hi >> 20) & 0x7ff;
  if (((hi << 1) | lo) == 0) return 0.f;
  if ((unsigned)(e - 898) > 250u) return (float)x;
  unsigned bits = (unsigned)(hi & 0x80000000) | (unsigned)((e - 896) << 23) |
                  (__funnelshift_l((unsigned)lo, (unsigned)hi, 3) & 0x7fffffu);
  const unsigned rest = (unsigned)lo & 0x1fffffffu;  // the 29 bits dropped
  if (rest > 0x10000000u || (rest == 0x10000000u && (bits & 1u))) ++bits;
  return __uint_as_float(bits);
}

// x as the sum of two FP32 values, the first of them x to nearest (48 bits; the first alone where the
// second would leave FP32's normal range).
__device__ __forceinline__ float2 f32_pair(double x) {
  const float h = f32_of(x);
  const int rest = __double2loint(x) & 0x1fffffff;  // the 29 bits dropped, of weight 2^(e - 127 - 52)
  const int hi = __double2hiint(x), ex = (hi >> 20) & 0x7ff;
  if ((unsigned)(ex - 950) > 200u) return make_float2(h, 0.f);
  const bool up = (__float_as_uint(h) & 0x7fffffffu) !=
                  ((unsigned)((ex - 896) << 23) | (__funnelshift_l((unsigned)__double2loint(x), (unsigned)hi, 3) & 0x7fffffu));
  const float l = (float)(up ? rest - 0x20000000 : rest) * __uint_as_float((unsigned)(ex - 896 - 52) << 23);
  return make_float2(h, hi < 0 ? -l : l);
}
// x y rounded once.
__device__ __forceinline__ float f32_product(double x, double y) {
  const float2 a = f32_pair(x), b = f32_pair(y);
  const float p = a.x * b.x;
  return p + (fmaf(a.x, b.x, -p) + (a.x * b.y + a.y * b.x));
}
// (2N+1) / ((h_i + h_j) sqrt(pi / 2)) rounded once.
template <int N>
__device__ __forceinline__ float f32_face_eps(double hi, double hj) {
  constexpr double c = (2 * N + 1) * 0.79788456080286535588;  // sqrt(2 / pi)
  constexpr float c0 = (float)c, c1 = (float)(c - (double)c0), ic = (float)(1.0 / c);
  const float2 a = f32_pair(hi), b = f32_pair(hj);
  const float s = a.x + b.x, t = s - a.x;
  const float rest = ((a.x - (s - t)) + (b.x - t)) + (a.y + b.y);
  const float q = c0 / s;
  return q + (fmaf(-q, s, c0) + fmaf(-q, rest, c1)) * (q * ic);
}

// The FP32 form's fluxes: L lanes per polygonal face (8, 16, 32 at N = 1, 2, 3: about the face nodes of
// three sub-triangles), the states and fluxes of a lane's first two face nodes held in registers
// from the wave speeds to the fluxes.  What it waited for before: the FP64 pipe (1 / dt, eps and the
// conversions of mu, h and the normals, per lane), then chains of dependent loads; the
// conversions are integer instructions now, 1 / dt comes with dt, eps and the viscous coefficients are
// formed in pairs of FP32 values, to the same single rounding, and slots and partners come as one pair.
// us per launch before and after: 32^3 P3 1,177 and 440 (127 for the bytes at
// the copy rate), 21^3 P2 258 and 90, 24^3 P1 479 and 76, 4^3 P1 18 and 12.
template <int N>
__global__ void __launch_bounds__(256) face_f32_kernel(const __grid_constant__ Batch bt) {
  constexpr int NF = nf_of(N), L = N == 1 ? 8 : (N == 2 ? 16 : 32), R = 2;
  const int64_t ggw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / L;
  const int lane = threadIdx.x % L;
  const bool on = ggw < bt.gpre[bt.nh];  // whole groups of lanes; the others only take part in the shuffles
  const int h = batch_find(bt.gpre, bt.nh, on ? ggw : 0);
  const DevMesh& m = bt.tab[h];
  const int64_t gw = on ? ggw - bt.gpre[h] : 0;
  const int64_t g0 = m.group_ptr[gw], g1 = on ? m.group_ptr[gw + 1] : g0;
  const int nitems = (int)(g1 - g0) * NF;
  const float* sq = (const float*)m.slot_q;
  const float* sfn = (const float*)m.slot_fn;
  float* sG = (float*)m.slot_G;
  const int2* pairs = m.group_pair + g0;
  const float rdt = f32_of(m.dt[0]), idt = f32_of(m.dt[1]), gam = f32_of(m.gamma);
  const int2 first = pairs[0];
  const int32_t ci = m.slot_cell[first.x];
  const int32_t cj = first.y >= 0 ? m.slot_cell[first.y] : ci;
  // |lambda_v| = max(4 mu / 3, kappa / c_v) / rho: the coefficient per side
  const ViscFace vf = *reinterpret_cast<const ViscFace*>(m.dt + 2);
  const double mu_i = m.mu[ci], mu_j = m.mu[cj], h_i = m.cell_h[ci], h_j = m.cell_h[cj];
  const float least = f32_of(vf.least);
  const float cvis_i = fmaxf(f32_product(mu_i, vf.factor), least), cvis_j = fmaxf(f32_product(mu_j, vf.factor), least);
  float smax = 0.f, vmax = 0.f;
  auto speeds = [&](const float* Q, const float (&n)[3], float cvis) {
    const float ir = 1.f / Q[0], rho = Q[0] * idt;
    const float v0 = Q[1] * ir, v1 = Q[2] * ir, v2 = Q[3] * ir;  // q_bar / dt ratios
    const float p = (gam - 1.f) * (Q[4] * idt - 0.5f * rho * (v0 * v0 + v1 * v1 + v2 * v2));
    const float irho = ir * rdt;  // 1 / rho
    smax = fmaxf(smax, fabsf(v0 * n[0] + v1 * n[1] + v2 * n[2]) + sqrtf(gam * p * irho));
    vmax = fmaxf(vmax, cvis * irho);
  };
  auto load = [&](int e, int2& ps, int& a, float (&qo)[5], float (&qp)[5]) {
    const int k = e / NF;
    a = e - k * NF;
    ps = pairs[k];
    const double* g = m.slot_geo + (int64_t)ps.x * 4;
    const float n[3] = {f32_of(g[0]), f32_of(g[1]), f32_of(g[2])};
    const float* po = sq + ((int64_t)ps.x * NF + a) * 5;
    const float* pp = sq + ((int64_t)max(ps.y, 0) * NF + a) * 5;
#pragma unroll
    for (int v = 0; v < 5; ++v) qo[v] = po[v], qp[v] = pp[v];
    speeds(qo, n, cvis_i);
    if (ps.y >= 0) speeds(qp, n, cvis_j);
  };
  int2 ps[R];
  int a[R];
  float qo[R][5], qp[R][5], fo[R][5], fp[R][5];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int e = lane + r * L;
    if (e >= nitems) continue;
    load(e, ps[r], a[r], qo[r], qp[r]);
    const float* po = sfn + ((int64_t)ps[r].x * NF + a[r]) * 5;
    const float* pp = sfn + ((int64_t)max(ps[r].y, 0) * NF + a[r]) * 5;
#pragma unroll
    for (int v = 0; v < 5; ++v) fo[r][v] = po[v], fp[r][v] = pp[v];
  }
  for (int e = lane + R * L; e < nitems; e += L) {
    int2 p2;
    int a2;
    float q1[5], q2[5];
    load(e, p2, a2, q1, q2);
  }
#pragma unroll
  for (int o = L / 2; o > 0; o >>= 1) {
    smax = fmaxf(smax, __shfl_xor_sync(0xffffffffu, smax, o));
    vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
  }
  const float eps = f32_face_eps<N>(h_i, h_j);
  const float diss = 0.5f * (smax + 2.f * eps * vmax);
  auto flux = [&](int2 p, int a1, const float* q1, const float* q2, const float* f1, const float* f2) {
    float* go = sG + ((int64_t)p.x * NF + a1) * 5;
    if (p.y < 0) {  // transmissive boundary: q+ = q-, F+ = F-
#pragma unroll
      for (int v = 0; v < 5; ++v) go[v] = f1[v];
      return;
    }
    float* gp = sG + ((int64_t)p.y * NF + a1) * 5;
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      // the matched side stores F_bar . (its own normal) = -F_bar+ . n
      const float G = 0.5f * (f1[v] - f2[v]) - diss * (q2[v] - q1[v]);
      go[v] = G;
      gp[v] = -G;
    }
  };
#pragma unroll
  for (int r = 0; r < R; ++r)
    if (lane + r * L < nitems) flux(ps[r], a[r], qo[r], qp[r], fo[r], fp[r]);
  for (int e = lane + R * L; e < nitems; e += L) {
    const int k = e / NF, a2 = e - k * NF;
    const int2 p2 = pairs[k];
    const int64_t io = ((int64_t)p2.x * NF + a2) * 5, ip = ((int64_t)max(p2.y, 0) * NF + a2) * 5;
    flux(p2, a2, sq + io, sq + ip, sfn + io, sfn + ip);
  }
}

// ----------------------------------------------------------------------------------------
// Corrector (Sec. 4.4): r = vol - sum_slots 2 area Z^ G (fixed-order gather), then
// u^{n+1} = u^n + M_i^-1 r.  FP64 path: everything in FP64.  FP32 path: r and the apply in
// FP32, then an FP64 correction adds a constant to du so that w_i . du equals sum(r)
// exactly in FP64 (the conserved totals of the cell: 1^T M_i du = 1^T r).
template <int N, typename Real>
__global__ void __launch_bounds__(256) corrector_kernel(DevMesh m, const RefData* __restrict__ ref) {
  constexpr int NF = nf_of(N);
  extern __shared__ double smem_dbl[];
  Real* r = (Real*)smem_dbl;                       // [Nmax][5]
  double* du = smem_dbl + ((m.Nmax * 5 * sizeof(Real) + 7) / 8);  // [Nmax][5], FP32 path only
  __shared__ Real sZ[NF][NF];
  __shared__ double sfix[2][5][sizeof(Real) == 4 ? 256 : 1];
  const int tid = threadIdx.x;
  for (int e = tid; e < NF * NF; e += blockDim.x) sZ[e / NF][e % NF] = (Real)ref->Z[e / NF][e % NF];
  __syncthreads();
  const Real* vol = (const Real*)m.vol;
  const Real* sG = (const Real*)m.slot_G;
  for (int64_t c = blockIdx.x; c < m.C; c += gridDim.x) {
    const int64_t n0 = m.node_ptr[c];
    const int Ni = (int)(m.node_ptr[c + 1] - n0);
    const int64_t s0 = m.slot_ptr[c];
    double tot[5] = {0, 0, 0, 0, 0};
    for (int e = tid; e < Ni * 5; e += blockDim.x) {
      const int n = e / 5, v = e % 5;
      Real acc = vol[(n0 + n) * 5 + v];
      for (int64_t p = m.finc_ptr[n0 + n]; p < m.finc_ptr[n0 + n + 1]; ++p) {
        const uint32_t w = m.finc[p];
        const int64_t s = s0 + (w >> 4);
        const int a = w & 15;
        const Real twoA = Real(2) * (Real)m.slot_geo[s * 4 + 3];
        Real f = 0;
#pragma unroll
        for (int b = 0; b < NF; ++b) f += sZ[a][b] * sG[(s * NF + b) * 5 + v];
        acc -= twoA * f;
      }
      r[e] = acc;
    }
    if constexpr (sizeof(Real) == 4) {
      // exact cell total of the update in FP64: sum_m vol[m] = int grad(sum phi_m) . F = 0,
      // so 1^T r = -sum_slots 2 area sum_b (sum_a Z^[a][b]) G[b]; matched slots cancel.
      const int ns = (int)(m.slot_ptr[c + 1] - s0);
      for (int e = tid; e < ns * NF * 5; e += blockDim.x) {
        const int sl = e / (NF * 5), b = (e / 5) % NF, v = e % 5;
        const int64_t s = s0 + sl;
        double zs = 0.0;
#pragma unroll
        for (int a = 0; a < NF; ++a) zs += ref->Z[a][b];
        tot[v] -= 2.0 * m.slot_geo[s * 4 + 3] * zs * (double)sG[(s * NF + b) * 5 + v];
      }
    }
    __syncthreads();
    const Real* minv;
    if constexpr (sizeof(Real) == 8) minv = (const Real*)(m.minv64 + m.minv_ptr[c]);
    else minv = (const Real*)(m.minv32 + m.minv_ptr[c]);
    double wdu[5] = {0, 0, 0, 0, 0};
    for (int n = tid; n < Ni; n += blockDim.x) {
      Real acc[5] = {0, 0, 0, 0, 0};
      const int LD = minv_ld(Ni);
      for (int l = 0; l < Ni; ++l) {
        const Real a = minv[(int64_t)l * LD + n];
#pragma unroll
        for (int v = 0; v < 5; ++v) acc[v] += a * r[l * 5 + v];
      }
      if constexpr (sizeof(Real) == 8) {
        bool bad = false;
        double* un = m.u + (n0 + n) * 5;
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          un[v] += (double)acc[v];
          bad |= !isfinite(un[v]);
        }
        const double rho = un[0];
        const double p = (m.gamma - 1.0) * (un[4] - 0.5 * (un[1] * un[1] + un[2] * un[2] + un[3] * un[3]) / rho);
        if (bad || !(rho > 0.0) || !(p > 0.0)) atomicOr(&m.flags[F_NONFINITE], 8);
      } else {
        const double w = m.wvec[n0 + n];
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          wdu[v] += w * (double)acc[v];
          du[n * 5 + v] = (double)acc[v];
        }
      }
    }
    if constexpr (sizeof(Real) == 4) {
      // FP64 totals (target and w . du), block-reduced in a fixed order
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        sfix[0][v][tid] = tot[v];
        sfix[1][v][tid] = wdu[v];
      }
      __syncthreads();
      for (int st = blockDim.x / 2; st > 0; st >>= 1) {
        if (tid < st)
#pragma unroll
          for (int v = 0; v < 5; ++v) {
            sfix[0][v][tid] += sfix[0][v][tid + st];
            sfix[1][v][tid] += sfix[1][v][tid + st];
          }
        __syncthreads();
      }
      double corr[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) corr[v] = (sfix[0][v][0] - sfix[1][v][0]) / m.cell_vol[c];
      for (int n = tid; n < Ni; n += blockDim.x) {
        double* un = m.u + (n0 + n) * 5;
        bool bad = false;
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          un[v] += du[n * 5 + v] + corr[v];
          bad |= !isfinite(un[v]);
        }
        const double rho = un[0];
        const double p = (m.gamma - 1.0) * (un[4] - 0.5 * (un[1] * un[1] + un[2] * un[2] + un[3] * un[3]) / rho);
        if (bad || !(rho > 0.0) || !(p > 0.0)) atomicOr(&m.flags[F_NONFINITE], 8);
      }
    }
    __syncthreads();
  }
}

// FP64 conserved totals sum_i w_i . u_i: per-block partials over a fixed cell partition,
// then a single block sums the partials in order (bitwise reproducible).
static __global__ void totals_partial_kernel(DevMesh m, double* partial) {
  __shared__ double sh[5][256];
  double acc[5] = {0, 0, 0, 0, 0};
  const int64_t per = (m.n_nodes + gridDim.x - 1) / gridDim.x;
  const int64_t a = blockIdx.x * per, b = min(m.n_nodes, a + per);
  for (int64_t n = a + threadIdx.x; n < b; n += blockDim.x) {
    const double w = m.wvec[n];
#pragma unroll
    for (int v = 0; v < 5; ++v) acc[v] += w * m.u[n * 5 + v];
  }
#pragma unroll
  for (int v = 0; v < 5; ++v) sh[v][threadIdx.x] = acc[v];
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s)
#pragma unroll
      for (int v = 0; v < 5; ++v) sh[v][threadIdx.x] += sh[v][threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x < 5) partial[blockIdx.x * 5 + threadIdx.x] = sh[threadIdx.x][0];
}

static __global__ void totals_final_kernel(const double* partial, int nblk, double* out) {
  if (threadIdx.x < 5) {
    double s = 0.0;
    for (int b = 0; b < nblk; ++b) s += partial[b * 5 + threadIdx.x];
    out[threadIdx.x] = s;
  }
}

}  // namespace afe
