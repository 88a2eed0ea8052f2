// FP32 space-time predictor with several cells in flight per SM (Sec. 4.3, Eqs.
// ADER-localCauchy, ader4, TAvectors): the form of every mesh that its plan takes (pc_plan, predictor_cells.cu).
//
// One block of 32 W threads per cell, persistent (blocks take cells from a work counter), two
// blocks per SM at N = 3 (one of 16 warps where the largest cell needs the SM) and more at N = 1, 2, so that one cell's barriers, gathers and
// serial tails are covered by another cell's arithmetic.  What the cell needs on chip:
//   srec  [S][REC]       its packed sub-tet records (adj(J), det J, node ids)
//   sgat                 its node -> (sub-tet, local node) lists, 16 bits per entry
//   sexp  [N_i]          row exponents of M_i^-1, 8 bits
//   suh   [N_i][5]       u^, the state at t^n
//   sq    [N_i][5][NTP]  space-time coefficients q, time innermost (one vector load per variable)
// and a region that phase 1 uses for the pre-contracted fluxes of a chunk of sub-tets and
// phase 2 for the right-hand side as matrix fragments.
//
// Per fixed-point iteration:
//   1. for chunks of sub-tets: a thread takes a (sub-tet, node) and all its time slices, so that
//      adj(J) and the node index are read once; the flux goes straight to its contravariant
//      form adj(J)_d . F = (rho U_d, m U_d + p adj(J)_d, (E + p) U_d), U_d = adj(J)_d . v, half
//      the arithmetic of F followed by adj(J).  Then one column (k, v, t) per thread through
//      the written-out stiffness contraction (sref_gen.cuh); its Np results replace the column
//      in place, transposed over the time slices of (k, v) so that the gather reads one vector
//      per variable.  The gather adds a node's incidences in (k, j) order in the registers of
//      the thread that owns the node (no atomics; the order does not depend on the chunks).
//      The first iteration starts from q^0 = u^ at every time node: one time slice serves all.
//   2. Y = M_i^-1 RHS on the tensor cores.  M_i^-1 is kept as pairs of
//      FP16 values hi + lo of M_i^-1 scaled to a unit diagonal by powers of two per row and column (both
//      parts rounded to nearest: 22 bits and a sign, where the TF32 head and tail taken by truncation
//      carry 21) in the register layout of mma.sync.m16n8k16, so that a warp streams its own 16-row tiles from L2
//      straight into registers, 1 KB per tile and 16 columns, with no staging in shared memory
//      and no splitting arithmetic.  M_i^-1 is symmetric: only the tiles of its lower triangle are
//      kept (a tile above the diagonal is the mirrored one, transposed in registers), which
//      halves what the cells in flight hold in L2 between iterations and what comes from HBM.  The
//      right-hand side is split the same way, its rows scaled by the inverse powers, then with a power
//      of two per variable (taken from its maximum over the cell).  The products hi hi + lo hi + hi lo
//      are accumulated in FP32.
//      q^{r+1}[n,s] = u^[n] - dt sum_t K1t^-1[s,t] w_t Y[n,t] straight from the accumulators.
// Epilogue: vol, q_bar and F_bar . n as the FP64 kernel; F_bar . n comes from the volume term's
// adj(J)_d . F_bar, because the rows of adj(J) are the area normals of the sub-tet's faces.
//
// Why this split: in the one-block-per-SM form the M_i^-1 apply took 31 k of the 72 k cycles of a
// later iteration at N = 3 (the split into TF32 parts and the fragment loads, 50 instructions per
// 16 x 16 block, against 11 here), and phases separated by block barriers left half of the issue
// slots empty.  Measured, us per predictor launch (one block per SM -> here): 32^3 P3 13,880 ->
// 7,735; 16^3 P3 2,377 -> 1,391; 8^3 P2 193 -> 97; 21^3 P2 Navier-Stokes 2,559 -> 1,569; 24^3 P1
// 2,955 -> 386; 4^3 P1 82 -> 39.  What bounds it at N = 3: M_i^-1 from L2 and HBM (two reads of each
// tile per iteration; the cells in flight hold 66 MB of it, just more than the L2 keeps) for 45 %
// of a cell's cycles, then the shared-memory pipe and block barriers (issue slots 42 % used).
#pragma once

#include <cuda_fp16.h>

#include "predictor_cells.hpp"
#include "predictor_f32.cuh"

namespace afe {

template <int N>
struct Pc {
  static constexpr int NP = np_of(N), NT = N + 1, NF = nf_of(N), NTP = f32_ntp(N);
  static constexpr int SQ = 5 * NTP;              // floats of q per node
  static constexpr int REC = f32_rec_bytes(N);
  // Strides (floats) of the pre-contracted flux columns: a column (k, v, t) of 3 Np values, the NT
  // columns of one (k, v), and the one column of a (k, v) where all time slices share it.  Chosen
  // for the banks: the Np nodes of consecutive sub-tets (5 KV, 5 K1 apart) land in consecutive
  // banks when the fluxes are stored, and eight consecutive (k, v) fill the banks when columns are
  // loaded as vectors or their results are stored (KKS at N = 2 is 2 (mod 8) vectors, so that the
  // lanes of the next time slice complete the eight).
  static constexpr int KKS = N == 3 ? 60 : (N == 2 ? 40 : 12);
  static constexpr int KV = N == 3 ? 260 : (N == 2 ? 132 : 28);
  static constexpr int K1 = N == 3 ? 68 : (N == 2 ? 36 : 12);
  static_assert(KKS >= 3 * NP && KV >= NT * KKS && K1 >= 3 * NP && KKS % 4 + KV % 4 + K1 % 4 == 0, "column strides");
  static constexpr int NNT = N == 1 ? 2 : 3;      // 8-column tiles of RHS / Y: column v NTP + t
  static constexpr int FB = N == 1 ? 640 : 1280;  // bytes of the RHS fragments per 16 rows (full tiles of
                                                  // 512 bytes; the last tile's used lanes only)
  static constexpr int GK = 32 / NT;              // (k, v) groups of NT columns a warp takes at a time
};

// Tile (i, j) of the symmetric M_i^-1 in its block (see minv_split_words).
__host__ __device__ constexpr int tri_tile(int i, int j) { return j <= i ? i * (i + 1) / 2 + j : j * (j + 1) / 2 + i; }
__host__ __device__ constexpr size_t pc_up(size_t x) { return (x + 127) / 128 * 128; }
// A cell's gather block (bytes): the number of long lists, the N_i nodes in decreasing order of
// list length with the row offset of their list, and the offset past the last list (16 bits
// each); S Np entries (k << 6) | j (16 bits); per face slot 1 / (2 area) (float), (k << 2) | opposite
// vertex (16 bits) and the Nf sub-tet nodes (8 bits).  The three parts are padded to 16 bytes,
// and blocks start at multiples of 16 that leave room for every cell.  Entries are in the order
// of the lists, so that the list of the i-th node ends where the next begins.
__host__ __device__ constexpr size_t gat_up(size_t x) { return (x + 15) / 16 * 16; }
__host__ __device__ constexpr size_t gat_bytes(int n, int s, int ns, int np, int nf) {
  return gat_up(2 * (size_t)(2 * n + 3)) + gat_up(2 * (size_t)s * np) + gat_up((size_t)ns * (6 + nf));
}
__host__ __device__ constexpr size_t gat_start(int64_t n0, int64_t k0, int64_t s0, int64_t c, int np, int nf) {
  return gat_up((size_t)(4 * n0 + 2 * np * k0 + (6 + nf) * s0 + 80 * c));
}
// Lists longer than this are shared by the lanes of a warp (in a fan subgrid: the cell centre,
// which every sub-tet holds); one thread alone would leave the block waiting for its serial sum.
constexpr int kLongList = 24;
constexpr int kMaxLong = 2;
constexpr int kPcMaxSub = 1023;  // sub-tet index of a gather entry: 10 bits
constexpr int kPcOver = 2;  // gather slots a thread has at most beside its first
constexpr int kPcDeep = 4;  // 16-column steps of M_i^-1 a warp keeps in flight

template <int NTP>
__device__ __forceinline__ void load_sums(const float4* o, float (&a)[5][NTP]) {
  if constexpr (NTP == 4) {
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      const float4 x = o[v];
      a[v][0] = x.x, a[v][1] = x.y, a[v][2] = x.z, a[v][3] = x.w;
    }
  } else {
    const float2* q = reinterpret_cast<const float2*>(o);
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      const float2 x = q[v];
      a[v][0] = x.x, a[v][1] = x.y;
    }
  }
}
template <int NTP>
__device__ __forceinline__ void store_sums(float4* o, const float (&a)[5][NTP]) {
  if constexpr (NTP == 4) {
#pragma unroll
    for (int v = 0; v < 5; ++v) o[v] = make_float4(a[v][0], a[v][1], a[v][2], a[v][3]);
  } else {
    float2* q = reinterpret_cast<float2*>(o);
#pragma unroll
    for (int v = 0; v < 5; ++v) q[v] = make_float2(a[v][0], a[v][1]);
  }
}

__device__ __forceinline__ uint4 ldg_stream(const uint32_t* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}
// Transpose of an 8 x 8 block of 16-bit values held two per lane (lane 4 r + c: row r, columns 2 c, 2 c + 1).
__device__ __forceinline__ uint32_t transpose8(uint32_t x) {
  uint32_t y;
  asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
  return y;
}
// Fragment of the transposed 16 x 16 tile from the tile's.
__device__ __forceinline__ uint4 transpose16(const uint4& a) {
  return make_uint4(transpose8(a.x), transpose8(a.z), transpose8(a.y), transpose8(a.w));
}
// D += A B, m16n8k16, FP16 operands, FP32 accumulators.
__device__ __forceinline__ void mma_f16(float (&d)[4], const uint4& a, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}
// Biased exponent of the power of two that takes a maximum of magnitude x into [2^13, 2^14) (at most 2^126, so
// that its inverse is a normal number too).
__host__ __device__ __forceinline__ int f16_scale_exp(uint32_t bits) {
  const int e = 267 - (int)(bits >> 23 & 255u);
  return e > 253 ? 253 : e;
}
// 2^e, -126 <= e <= 127.
__device__ __forceinline__ float pow2f(int e) { return __uint_as_float((uint32_t)(127 + e) << 23); }

// adj(J)_d . F_e at one state, Euler: out[d][v].
__device__ __forceinline__ void contravariant_flux(const float (&Q)[5], const float (&g)[9], float gm1,
                                                   float out[3][5]) {
  const float ir = 1.f / Q[0];
  const float v0 = Q[1] * ir, v1 = Q[2] * ir, v2 = Q[3] * ir;
  const float p = gm1 * (Q[4] - 0.5f * Q[0] * (v0 * v0 + v1 * v1 + v2 * v2));
  const float H = Q[4] + p;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float U = g[3 * d] * v0 + g[3 * d + 1] * v1 + g[3 * d + 2] * v2;
    out[d][0] = Q[0] * U;
#pragma unroll
    for (int a = 0; a < 3; ++a) out[d][1 + a] = Q[1 + a] * U + p * g[3 * d + a];
    out[d][4] = H * U;
  }
}

// What the phases of a cell share, in shared memory: each phase is a function of its own that
// loads what it needs, so that none of them holds registers for the others (with everything
// inlined, the values that live across phases spilled to local memory, which the shared-memory
// carve-out leaves hardly any L1 for: 8.5 against 12.3 ms per launch at 32^3, N = 3).
struct PcCell {
  const DevMesh* m;
  const uint32_t* m16;    // fragments of the split M_i^-1
  int64_t c, n0, s0;
  int Ni, S, ns, nks, nlong, slots, room;
  uint32_t o_gat, o_inc, o_exp, o_uh, o_q, o_region;  // bytes from the start of dynamic shared memory
  float dt, gam, gm1, mu, kap;
  float isv[5];                         // 1 / (power of two of the right-hand side), per variable
};

// At the start of dynamic shared memory (every function names that memory itself, so that the
// accesses are known to be shared-memory ones, with 32-bit addresses).
struct PcShared {
  PcCell x;
  PcRef ref;
  float red[5][16];  // per-warp maxima
};
extern __shared__ __align__(128) unsigned char pc_smem[];
__device__ __forceinline__ PcShared& pc_shared() { return *reinterpret_cast<PcShared*>(pc_smem); }

// Bytes of the fixed part for a cell of n nodes and s sub-tets, and of its smallest region.
template <int N>
__host__ __device__ constexpr size_t pc_fixed(int n, int s, int ns) {
  return pc_up(sizeof(PcShared)) + pc_up((size_t)s * Pc<N>::REC) + pc_up(gat_bytes(n, s, ns, Pc<N>::NP, Pc<N>::NF)) +
         (size_t)minv_split_head(n) * 4 + pc_up((size_t)n * 20) + pc_up((size_t)n * Pc<N>::SQ * 4);
}
// Gather slots of a cell at most (a warp shares at most one long list).
__host__ __device__ constexpr int pc_slots(int n, int thr) { return n + 31 * (thr / 32 < kMaxLong ? thr / 32 : kMaxLong); }
template <int N>
__host__ __device__ constexpr size_t pc_over(int slots, int thr) {
  return slots > thr ? (size_t)(slots - thr) * Pc<N>::SQ * 4 : 0;
}
template <int N>
__host__ __device__ constexpr size_t pc_need(int n, int s, int ns, int thr) {
  const size_t frag = (size_t)((n + 15) / 16) * Pc<N>::FB + pc_over<N>(pc_slots(n, thr), 2 * thr);
  // four sub-tets at least, beside the sums of the gather slots past the first of each thread;
  // the fragments beside those past the second
  const size_t chunk = (size_t)4 * 5 * Pc<N>::KV * 4 + pc_over<N>(pc_slots(n, thr), thr);
  return pc_fixed<N>(n, s, ns) + (frag > chunk ? frag : chunk);
}
template <int N>
struct PcView {  // pointers into the cell's shared memory
  const unsigned char* srec;
  const uint16_t *slist, *sinc;
  const int8_t* sexp;
  const float* suh;
  float *sq, *region;
  __device__ __forceinline__ PcView()
      : srec(pc_smem + pc_up(sizeof(PcShared))),
        slist(reinterpret_cast<const uint16_t*>(pc_smem + pc_shared().x.o_gat)),
        sinc(reinterpret_cast<const uint16_t*>(pc_smem + pc_shared().x.o_inc)),
        sexp(reinterpret_cast<const int8_t*>(pc_smem + pc_shared().x.o_exp)),
        suh(reinterpret_cast<const float*>(pc_smem + pc_shared().x.o_uh)),
        sq(reinterpret_cast<float*>(pc_smem + pc_shared().x.o_q)),
        region(reinterpret_cast<float*>(pc_smem + pc_shared().x.o_region)) {}
  __device__ __forceinline__ const float* g(int k) const {
    return reinterpret_cast<const float*>(srec + k * Pc<N>::REC);
  }
  __device__ __forceinline__ const uint16_t* a(int k) const {
    return reinterpret_cast<const uint16_t*>(srec + k * Pc<N>::REC + 40);
  }
};

// Gather slots: slots 32 i .. 32 i + 31 share the i-th long list, the others take one node each.
// Returns the slot's node, or -1, and the entries cur, cur + step, ... < end of its list.
__device__ __forceinline__ int slot_list(const uint16_t* slist, int Ni, int nlong, int i, int& cur, int& end,
                                         int& step) {
  const bool share = i < 32 * nlong;
  const int q = share ? i >> 5 : i - 31 * nlong;
  cur = end = 0;
  step = share ? 32 : 1;
  if (q >= Ni) return -1;
  cur = slist[2 + 2 * q] + (share ? i & 31 : 0);
  end = slist[4 + 2 * q];
  return (int)slist[1 + 2 * q];
}

// Gradient columns of a chunk (viscous cells): column (k, v, t) of the buffer receives d/dxi_d of
// the sub-tet polynomial at node j, at row (d, j).
template <int N, int W>
__device__ __forceinline__ void pc_gradients(int kc, int nk, int nte, int kvs,
                                          bool first) {
  using P = Pc<N>;
  const PcView<N> V;
  const PcCell& x = pc_shared().x;
  const int cols = nk * 5 * nte;
  for (int col = threadIdx.x; col < cols; col += 32 * W) {
    const int kv = col / nte, t = col - kv * nte, kl = kv / 5, v = kv - kl * 5;
    const uint16_t* Ak = V.a(kc + kl);
    float q[P::NP];
#pragma unroll
    for (int l = 0; l < P::NP; ++l) q[l] = first ? V.suh[Ak[l] * 5 + v] : V.sq[Ak[l] * P::SQ + v * P::NTP + t];
    SrefFP32<N>::gradient(q, V.region + kv * kvs + t * P::KKS);
  }
}

// Physical flux of a viscous cell at a node whose reference gradients sit in the buffer columns.
template <int N>
__device__ __forceinline__ void pc_flux_visc(const PcCell& x, const float (&Q)[5], const float (&g)[9], float idet,
                                             const float* gcol, int vstride, float F[3][5]) {
  float gq[3][5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    const float x0 = gcol[v * vstride], x1 = gcol[v * vstride + Pc<N>::NP], x2 = gcol[v * vstride + 2 * Pc<N>::NP];
#pragma unroll
    for (int e = 0; e < 3; ++e) gq[e][v] = (g[e] * x0 + g[3 + e] * x1 + g[6 + e] * x2) * idet;
  }
  phys_flux<float>(Q, gq, true, x.mu, x.kap, x.gam, (float)x.m->Rgas, F);
}

template <int NTP>
__device__ __forceinline__ void load_q(const float* q, float (&qv)[5][NTP]) {
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    if constexpr (NTP == 4) {
      const float4 y = *reinterpret_cast<const float4*>(q + v * 4);
      qv[v][0] = y.x, qv[v][1] = y.y, qv[v][2] = y.z, qv[v][3] = y.w;
    } else {
      const float2 y = *reinterpret_cast<const float2*>(q + v * 2);
      qv[v][0] = y.x, qv[v][1] = y.y;
    }
  }
}

// Pre-contracted fluxes of a chunk: B[(k, v, t)][(d, j)] = adj(J_k)_d . F(q at node j, time t).
template <int N, int W, bool VISC>
__device__ __forceinline__ void pc_fluxes(int kc, int nk, bool first) {
  using P = Pc<N>;
  constexpr int NP = P::NP, NT = P::NT, NTP = P::NTP, KKS = P::KKS, KV = P::KV, K1 = P::K1;
  const PcView<N> V;
  const PcCell& x = pc_shared().x;
  const float gm1 = x.gm1;
  for (int e = threadIdx.x; e < nk * NP; e += 32 * W) {
    const int kl = e / NP, j = e - kl * NP;
    const float* gp = V.g(kc + kl);
    float g[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) g[i] = gp[i];
    const int node = V.a(kc + kl)[j];
    if (first) {
      float* dst = V.region + kl * 5 * K1 + j;
      float Q[5], out[3][5];
#pragma unroll
      for (int v = 0; v < 5; ++v) Q[v] = V.suh[node * 5 + v];
      if constexpr (VISC) {
        float F[3][5];
        pc_flux_visc<N>(x, Q, g, 1.f / gp[9], dst, K1, F);
        f32_contract_adj(g, 1.f, F, out);
      } else {
        contravariant_flux(Q, g, gm1, out);
      }
#pragma unroll
      for (int v = 0; v < 5; ++v)
#pragma unroll
        for (int d = 0; d < 3; ++d) dst[v * K1 + d * NP] = out[d][v];
    } else {
      float* dst = V.region + kl * 5 * KV + j;
      // one time slice at a time (not unrolled): the sums of the gather stay in registers here
      const float* qn = V.sq + node * P::SQ;
#pragma unroll 1
      for (int t = 0; t < NT; ++t) {
        const float Q[5] = {qn[t], qn[NTP + t], qn[2 * NTP + t], qn[3 * NTP + t], qn[4 * NTP + t]};
        float out[3][5];
        if constexpr (VISC) {
          float F[3][5];
          pc_flux_visc<N>(x, Q, g, 1.f / gp[9], dst + t * KKS, KV, F);
          f32_contract_adj(g, 1.f, F, out);
        } else {
          contravariant_flux(Q, g, gm1, out);
        }
#pragma unroll
        for (int v = 0; v < 5; ++v)
#pragma unroll
          for (int d = 0; d < 3; ++d) dst[v * KV + t * KKS + d * NP] = out[d][v];
      }
    }
  }
}

// The stiffness contraction, one column per thread; results replace the columns of (k, v) as
// [m][NTP] (one time slice: [m]).  The lanes of a group sit in one warp, so a warp barrier is all
// that separates the last read of a column from the first write over it.
template <int N, int W>
__device__ __forceinline__ void pc_contract(float* region, int nkv, bool one) {
  using P = Pc<N>;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int kvw = one ? 32 : P::GK;                      // (k, v) per warp; lanes t GK + (k, v)
  const int t = one ? 0 : lane / P::GK, kvs = one ? P::K1 : P::KV, st = one ? 1 : P::NTP;
  for (int kb = warp * kvw; kb < nkv; kb += W * kvw) {
    const int kv = kb + lane - t * kvw;
    const bool on = t < P::NT && kv < nkv;
    float acc[P::NP];
#pragma unroll
    for (int i = 0; i < P::NP; ++i) acc[i] = 0.f;
    if (on) SrefFP32<N>::contract(region + kv * kvs + t * P::KKS, acc);
    __syncwarp();
    if (on) {
      float* dst = region + kv * kvs + t;
#pragma unroll
      for (int i = 0; i < P::NP; ++i) dst[i * st] = acc[i];
    }
  }
}

// Adds the entries of a list that lie in the chunk of nk sub-tets from kc.
template <int N>
__device__ __forceinline__ void pc_gather(const PcView<N>& V, int kc, int nk, bool first, int& cur, int end, int step,
                                          float (&acc)[5][Pc<N>::NTP]) {
  using P = Pc<N>;
  const int lim = (kc + nk) << 6;
  int w = cur < end ? V.sinc[cur] : lim;
  while (w < lim) {
    const int kl = (w >> 6) - kc, j = w & 63;
    cur += step;
    w = cur < end ? V.sinc[cur] : lim;
    if (first) {
      const float* src = V.region + kl * 5 * P::K1 + j;
#pragma unroll
      for (int v = 0; v < 5; ++v) acc[v][0] += src[v * P::K1];
    } else {
      const float* src = V.region + kl * 5 * P::KV + j * P::NTP;
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        if constexpr (P::NTP == 4) {
          const float4 y = *reinterpret_cast<const float4*>(src + v * P::KV);
          acc[v][0] += y.x;
          acc[v][1] += y.y;
          acc[v][2] += y.z;
          if (P::NT == 4) acc[v][3] += y.w;
        } else {
          const float2 y = *reinterpret_cast<const float2*>(src + v * P::KV);
          acc[v][0] += y.x;
          acc[v][1] += y.y;
        }
      }
    }
  }
}

// ---- 1. Right-hand side of an iteration, left in the region as split fragments.
template <int N, int W, bool VISC>
__device__ __forceinline__ void pc_rhs(bool first) {
  using P = Pc<N>;
  constexpr int NT = P::NT, NTP = P::NTP, SQ = P::SQ, THR = 32 * W, FB = P::FB;
  const PcView<N> V;
  PcCell& x = pc_shared().x;
  auto& sred = pc_shared().red;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int S = x.S, over = max(x.slots - THR, 0);
  float* const sover = V.region + x.room / 4 - over * SQ;  // sums of the slots past THR
  const int kvs = first ? P::K1 : P::KV;                   // floats per (k, v)
  const int cap = (x.room - over * SQ * 4) / (5 * kvs * 4);
  const int nch = (S + cap - 1) / cap, CH = (S + nch - 1) / nch;  // chunks of equal width
  // sums of this thread's first slot in registers
  float racc[5][NTP];
  int cur, cend, cstep;
  const int node0 = slot_list(V.slist, x.Ni, x.nlong, tid, cur, cend, cstep);
#pragma unroll
  for (int v = 0; v < 5; ++v)
#pragma unroll
    for (int t = 0; t < NTP; ++t) racc[v][t] = 0.f;
  for (int e = tid; e < over * SQ; e += THR) sover[e] = 0.f;
  for (int kc = 0; kc < S; kc += CH) {
    const int nk = min(CH, S - kc);
    if constexpr (VISC) {
      pc_gradients<N, W>(kc, nk, first ? 1 : NT, kvs, first);
      __syncthreads();
    }
    pc_fluxes<N, W, VISC>(kc, nk, first);
    __syncthreads();
    pc_contract<N, W>(V.region, nk * 5, first);
    __syncthreads();
    // gather this chunk's entries, in list order
    pc_gather<N>(V, kc, nk, first, cur, cend, cstep, racc);
    for (int i = tid + THR; i < x.slots; i += THR) {
      int c1, e1, st1;
      slot_list(V.slist, x.Ni, x.nlong, i, c1, e1, st1);
      while (c1 < e1 && V.sinc[c1] < (kc << 6)) ++c1;  // entries of earlier chunks (these lists are short)
      if (c1 >= e1 || V.sinc[c1] >= (kc + nk) << 6) continue;
      float4* o = reinterpret_cast<float4*>(sover + (i - THR) * SQ);
      float a[5][NTP];
      load_sums(o, a);
      pc_gather<N>(V, kc, nk, first, c1, e1, 1, a);
      store_sums(o, a);
    }
    if (kc + CH < S) __syncthreads();  // the next chunk's items overwrite the results
  }
  if (warp < x.nlong) {  // the lanes' shares of a long list, in a fixed order
#pragma unroll
    for (int v = 0; v < 5; ++v)
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        if (first && t > 0) continue;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) racc[v][t] += __shfl_xor_sync(0xffffffffu, racc[v][t], o);
      }
  }
  // the right-hand side's power of two per variable, over the scaled rows.  The fragments overwrite the
  // region up to the sums of the third slots: those of the second slots are read before the barrier.
  float a[5][NTP];
#pragma unroll
  for (int v = 0; v < 5; ++v)
#pragma unroll
    for (int t = 0; t < NTP; ++t) a[v][t] = 0.f;
  float omax[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) omax[v] = 0.f;
  for (int i = tid + (x.slots - 1 - tid) / THR * THR; i >= THR; i -= THR) {  // the second slot last
    load_sums(reinterpret_cast<const float4*>(sover + (i - THR) * SQ), a);
    const float f = pow2f(-(int)V.sexp[V.slist[1 + 2 * (i - 31 * x.nlong)]]);
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      float mx = 0.f;
#pragma unroll
      for (int t = 0; t < NT; ++t) mx = fmaxf(mx, fabsf(a[v][t]));
      omax[v] = fmaxf(omax[v], mx * f);
    }
  }
  const float f0 = node0 >= 0 ? pow2f(-(int)V.sexp[node0]) : 0.f;
  int sc[5];  // biased exponents
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    float mx = 0.f;
#pragma unroll
    for (int t = 0; t < NT; ++t) mx = fmaxf(mx, fabsf(racc[v][t]));
    mx = fmaxf(omax[v], mx * f0);
    // non-negative floats order as integers
    mx = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(mx)));
    if (lane == 0) sred[v][warp] = mx;
  }
  __syncthreads();
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    float y = sred[v][0];
#pragma unroll
    for (int w = 1; w < W; ++w) y = fmaxf(y, sred[v][w]);
    sc[v] = f16_scale_exp(__float_as_uint(y));
    if (tid == 0) x.isv[v] = __uint_as_float((uint32_t)(254 - sc[v]) << 23);
  }
  // fragments: entry (row n, column col) at 16-row step n / 16, column tile col / 8, lane
  // (col & 7) 4 + ((n & 7) >> 1), words {b0 hi, b1 hi, b0 lo, b1 lo}, b = (n & 15) >> 3
  unsigned char* const frag = reinterpret_cast<unsigned char*>(V.region);
  const int fb = first ? 320 : FB;
  auto row = [&](int n) { return frag + (n >> 4) * fb + ((n & 7) >> 1) * 16 + ((n >> 3) & 1) * 4 + (n & 1) * 2; };
  auto put = [&](int n, const float (&a)[5][NTP]) {
    unsigned char* const b = row(n);
    const int p = V.sexp[n];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      // row and variable in one power of two (bounded: sums below 2^-112 of a cell's would need more)
      const float s = __uint_as_float((uint32_t)min(254, max(1, sc[v] - p)) << 23);
#pragma unroll
      for (int t = 0; t < NTP; ++t) {
        if (first && t > 0) continue;
        const int col = first ? v : v * NTP + t;
        const float y = a[v][t] * s;
        const __half hi = __float2half_rn(y);
        const __half lo = __float2half_rn(y - __half2float(hi));
        unsigned char* d = b + (col >> 3) * 512 + (col & 7) * 64;
        *reinterpret_cast<__half*>(d) = hi;
        *reinterpret_cast<__half*>(d + 8) = lo;
      }
    }
  };
  int n = warp >= x.nlong || lane == 0 ? node0 : -1;
#pragma unroll 1
  for (int i = tid;;) {  // first, second, later slots
    if (n >= 0) put(n, racc);
    i += THR;
    if (i >= x.slots) break;
    n = V.slist[1 + 2 * (i - 31 * x.nlong)];
    if (i >= 2 * THR) load_sums(reinterpret_cast<const float4*>(sover + (i - THR) * SQ), a);
#pragma unroll
    for (int v = 0; v < 5; ++v)
#pragma unroll
      for (int t = 0; t < NTP; ++t) racc[v][t] = a[v][t];
  }
  // rows past N_i: zero (the matrix is zero there, but not the memory)
  const int nc = first ? 5 : 5 * NTP;
  for (int e = tid; e < (16 * x.nks - x.Ni) * nc; e += THR) {
    const int col = e % nc;
    unsigned char* d = row(x.Ni + e / nc) + (col >> 3) * 512 + (col & 7) * 64;
    *reinterpret_cast<__half*>(d) = __half(0.f);
    *reinterpret_cast<__half*>(d + 8) = __half(0.f);
  }
}

// ---- 2. Y = M_i^-1 RHS and q^{r+1}: warp w takes the 16-row tiles w, w + W, ..., TP at a time.
// Returns this thread's max |q^{r+1} - q^r| and max |q^r|.
template <int N, int W, bool FIRST>
__device__ __forceinline__ float2 pc_apply() {
  using P = Pc<N>;
  constexpr int NT = P::NT, NTP = P::NTP, SQ = P::SQ;
  constexpr int NT1 = FIRST ? 1 : P::NNT;         // column tiles: 1 in the first iteration
  constexpr int fb = FIRST ? 320 : P::FB;
  constexpr int QL = FIRST ? 20 : 20 * NTP;       // fragment lanes in use over the column tiles
  constexpr int DP = N == 1 ? 2 : kPcDeep;
  const PcView<N> V;
  const PcCell& x = pc_shared().x;
  const PcRef& ref = pc_shared().ref;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int Ni = x.Ni, nks = x.nks;
  const unsigned char* const frag = reinterpret_cast<const unsigned char*>(V.region) + lane * 16;
  float res = 0.f, qmax = 0.f;
  // dt over the scaling of row n of the product
  auto unscale = [&](int n) { return pow2f(-(int)V.sexp[n] - 13) * x.dt; };
  // q^{r+1} of (node n, variable v) from its NT values of M_i^-1 RHS
  auto update = [&](int n, int v, float (&y)[NTP], float isc) {
    const float si = x.isv[v], uh = V.suh[n * 5 + v];
    float old[NTP], z[NTP];
    float* qp = V.sq + n * SQ + v * NTP;
    if constexpr (FIRST) {
#pragma unroll
      for (int t = 0; t < NTP; ++t) old[t] = uh;
    } else if constexpr (NTP == 4) {
      const float4 o = *reinterpret_cast<const float4*>(qp);
      old[0] = o.x, old[1] = o.y, old[2] = o.z, old[3] = o.w;
    } else {
      const float2 o = *reinterpret_cast<const float2*>(qp);
      old[0] = o.x, old[1] = o.y;
    }
#pragma unroll
    for (int t = 0; t < NTP; ++t)
      if (t == 0 || !FIRST) y[t] = (y[t] * isc) * si;
#pragma unroll
    for (int s = 0; s < NTP; ++s) {
      z[s] = 0.f;
      if (s >= NT) continue;
      float a = uh;
      if constexpr (FIRST) {
        a -= ref.kws[s] * y[0];
      } else {
#pragma unroll
        for (int t = 0; t < NT; ++t) a -= ref.kw[s][t] * y[t];
      }
      z[s] = a;
      res = fmaxf(res, fabsf(a - old[s]));
      qmax = fmaxf(qmax, fabsf(old[s]));
    }
    if constexpr (NTP == 4) *reinterpret_cast<float4*>(qp) = make_float4(z[0], z[1], z[2], z[3]);
    else *reinterpret_cast<float2*>(qp) = make_float2(z[0], z[1]);
  };
  for (int mt = warp; mt < nks; mt += W) {
    float acc[NT1][4];
#pragma unroll
    for (int nt = 0; nt < NT1; ++nt)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[nt][i] = 0.f;
    const uint32_t* const a0 = x.m16 + lane * 4;
    uint4 ah[DP], al[DP];  // tiles in flight
    // unconditional (past the end: the last tile again), so that the loads of DP steps stay in flight
    auto load = [&](int s, int ks) {
      const uint32_t* t = a0 + tri_tile(mt, min(ks, nks - 1)) * 256;
      ah[s] = ldg_stream(t);
      al[s] = ldg_stream(t + 128);
    };
    auto step = [&](int s, int ks) {
      uint4 b[NT1];
#pragma unroll
      for (int nt = 0; nt < NT1; ++nt) {
        const bool on = nt * 32 + lane < QL;
        b[nt] = on ? *reinterpret_cast<const uint4*>(frag + ks * fb + nt * 512) : make_uint4(0, 0, 0, 0);
      }
      uint4 h = ah[s], l = al[s];
      if (ks > mt) {  // above the diagonal: the mirrored tile
        h = transpose16(h);
        l = transpose16(l);
      }
#pragma unroll
      for (int nt = 0; nt < NT1; ++nt) mma_f16(acc[nt], l, b[nt].x, b[nt].y);
#pragma unroll
      for (int nt = 0; nt < NT1; ++nt) mma_f16(acc[nt], h, b[nt].z, b[nt].w);
#pragma unroll
      for (int nt = 0; nt < NT1; ++nt) mma_f16(acc[nt], h, b[nt].x, b[nt].y);
    };
#pragma unroll
    for (int s = 0; s < DP; ++s) load(s, s);
    int ks = 0;
    for (; ks + DP <= nks; ks += DP) {
#pragma unroll
      for (int s = 0; s < DP; ++s) {
        step(s, ks + s);
        load(s, ks + s + DP);
      }
    }
#pragma unroll
    for (int s = 0; s < DP - 1; ++s)
      if (ks + s < nks) step(s, ks + s);
    asm volatile("" ::: "memory");  // the update's constants are loaded behind the products, not held through them
    const int gq = lane >> 2, tq = lane & 3;
    const int row = mt * 16 + gq;
    const float is0 = unscale(row), is1 = unscale(row + 8);
      if constexpr (FIRST) {
        // columns 2 tq, 2 tq + 1 are variables
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int v = 2 * tq + (i & 1), n = row + (i >> 1) * 8;
          float y[NTP];
          y[0] = acc[0][i];
          if (v < 5 && n < Ni) update(n, v, y, i >> 1 ? is1 : is0);
        }
      } else if constexpr (NTP == 2) {
#pragma unroll
        for (int nt = 0; nt < NT1; ++nt)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int v = nt * 4 + tq, n = row + 8 * h;
            float y[2] = {acc[nt][2 * h], acc[nt][2 * h + 1]};
            if (v < 5 && n < Ni) update(n, v, y, h ? is1 : is0);
          }
      } else {
        // a lane pair holds the four time slices of rows g and g + 8: the even lane takes
        // row g, the odd lane row g + 8
#pragma unroll
        for (int nt = 0; nt < NT1; ++nt) {
          const float* d = acc[nt];
          const bool odd = tq & 1;
          const float s0 = odd ? d[0] : d[2], s1 = odd ? d[1] : d[3];
          const float r0 = __shfl_xor_sync(0xffffffffu, s0, 1), r1 = __shfl_xor_sync(0xffffffffu, s1, 1);
          const int v = nt * 2 + (tq >> 1), n = row + (odd ? 8 : 0);
          float y[4] = {odd ? r0 : d[0], odd ? r1 : d[1], odd ? d[2] : r0, odd ? d[3] : r1};
          if (v < 5 && n < Ni) update(n, v, y, odd ? is1 : is0);
        }
      }
  }
  return make_float2(res, qmax);
}

// B_bar[(k, v)][(d, j)] = dt adj(J_k)_d . sum_t w_t F(q_t) of a chunk.
template <int N, int W, bool VISC>
__device__ __forceinline__ void pc_mean_fluxes(int kc, int nk) {
  using P = Pc<N>;
  constexpr int NP = P::NP, NT = P::NT, NTP = P::NTP, KKS = P::KKS, KV = P::KV, K1 = P::K1;
  constexpr int kvs = VISC ? KV : K1;
  const PcView<N> V;
  const PcCell& x = pc_shared().x;
  const PcRef& ref = pc_shared().ref;
  const float gm1 = x.gm1, dt = x.dt;
  for (int e = threadIdx.x; e < nk * NP; e += 32 * W) {
    const int kl = e / NP, j = e - kl * NP;
    const float* gp = V.g(kc + kl);
    const int node = V.a(kc + kl)[j];
    float* dst = V.region + kl * 5 * kvs + j;
    float qv[5][NTP];
    load_q<NTP>(V.sq + node * P::SQ, qv);
    float out[3][5], g[9];
    if constexpr (VISC) {
#pragma unroll
      for (int i = 0; i < 9; ++i) g[i] = gp[i];
      float fb[3][5];
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int v = 0; v < 5; ++v) fb[d][v] = 0.f;
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        const float Q[5] = {qv[0][t], qv[1][t], qv[2][t], qv[3][t], qv[4][t]};
        float F[3][5];
        pc_flux_visc<N>(x, Q, g, 1.f / gp[9], dst + t * KKS, KV, F);
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
          for (int v = 0; v < 5; ++v) fb[d][v] += ref.w[t] * F[d][v];
      }
      f32_contract_adj(g, dt, fb, out);
    } else {
      // time integrals of m_a, m_a v_b (symmetric), p and (E + p) v_a, then adj(J) once
      float M[3] = {0.f, 0.f, 0.f}, T[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, pb = 0.f, E[3] = {0.f, 0.f, 0.f};
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        const float wt = ref.w[t], ir = 1.f / qv[0][t];
        const float m0 = qv[1][t], m1 = qv[2][t], m2 = qv[3][t];
        const float v0 = m0 * ir, v1 = m1 * ir, v2 = m2 * ir;
        const float pr = gm1 * (qv[4][t] - 0.5f * qv[0][t] * (v0 * v0 + v1 * v1 + v2 * v2));
        const float H = wt * (qv[4][t] + pr);
        const float w0 = wt * m0, w1 = wt * m1, w2 = wt * m2;
        M[0] += w0;
        M[1] += w1;
        M[2] += w2;
        T[0] += w0 * v0;
        T[1] += w0 * v1;
        T[2] += w0 * v2;
        T[3] += w1 * v1;
        T[4] += w1 * v2;
        T[5] += w2 * v2;
        pb += wt * pr;
        E[0] += H * v0;
        E[1] += H * v1;
        E[2] += H * v2;
      }
      const float fb[3][5] = {{M[0], T[0] + pb, T[1], T[2], E[0]},
                              {M[1], T[1], T[3] + pb, T[4], E[1]},
                              {M[2], T[2], T[4], T[5] + pb, E[2]}};
#pragma unroll
      for (int i = 0; i < 9; ++i) g[i] = gp[i];
      f32_contract_adj(g, dt, fb, out);
    }
#pragma unroll
    for (int v = 0; v < 5; ++v)
#pragma unroll
      for (int d = 0; d < 3; ++d) dst[v * kvs + d * NP] = out[d][v];
  }
}

// Volume term's contraction (S^ transposed), one column per thread, in place.
template <int N, int W>
__device__ __forceinline__ void pc_contract_t(int nkv, int kvs) {
  float* const region = PcView<N>().region;
  for (int col = threadIdx.x; col < nkv; col += 32 * W) {
    float acc[Pc<N>::NP];
#pragma unroll
    for (int i = 0; i < Pc<N>::NP; ++i) acc[i] = 0.f;
    float* dst = region + col * kvs;
    SrefFP32<N>::contract_t(dst, acc);
    asm volatile("" ::: "memory");  // the results replace the column
#pragma unroll
    for (int i = 0; i < Pc<N>::NP; ++i) dst[i] = acc[i];
  }
}

// ---- Epilogue: the volume term, q_bar and F_bar . n on the face slots.
template <int N, int W, bool VISC>
__device__ __forceinline__ void pc_epilogue() {
  using P = Pc<N>;
  constexpr int NP = P::NP, NT = P::NT, NF = P::NF, NTP = P::NTP, SQ = P::SQ, THR = 32 * W;
  const PcView<N> V;
  const PcCell& x = pc_shared().x;
  const PcRef& ref = pc_shared().ref;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const DevMesh& m = *x.m;
  const int S = x.S, ns = x.ns;
  const float* const sface = reinterpret_cast<const float*>(V.sinc + gat_up(2 * S * NP) / 2);
  const uint16_t* const sfinfo = reinterpret_cast<const uint16_t*>(sface + ns);
  const uint8_t* const sfloc = reinterpret_cast<const uint8_t*>(sfinfo + ns);
  float vacc[kPcOver + 1][5];
  int cur[kPcOver + 1], cend[kPcOver + 1], cstep[kPcOver + 1], node[kPcOver + 1];
#pragma unroll
  for (int r = 0; r <= kPcOver; ++r) {
#pragma unroll
    for (int v = 0; v < 5; ++v) vacc[r][v] = 0.f;
    node[r] = slot_list(V.slist, x.Ni, x.nlong, tid + r * THR, cur[r], cend[r], cstep[r]);
  }
  constexpr int kvs = VISC ? P::KV : P::K1;  // viscous cells hold the gradients of every time slice
  const int cap = x.room / (5 * kvs * 4);
  const int nch = (S + cap - 1) / cap, CH = (S + nch - 1) / nch;
  for (int kc = 0; kc < S; kc += CH) {
    const int nk = min(CH, S - kc);
    if (kc) __syncthreads();
    if constexpr (VISC) {
      pc_gradients<N, W>(kc, nk, NT, P::KV, false);
      __syncthreads();
    }
    pc_mean_fluxes<N, W, VISC>(kc, nk);
    __syncthreads();
    // face slots of the chunk's sub-tets: q_bar and F_bar . n.  2 area n = -adj(J)_d on the
    // face opposite vertex d + 1, and sum_d adj(J)_d on the face opposite vertex 0.
    float* const sqo = (float*)m.slot_q;
    float* const sfn = (float*)m.slot_fn;
    for (int e = tid; e < ns * NF; e += THR) {
      const int sl = e / NF;
      const int info = sfinfo[sl];
      const int kl = (info >> 2) - kc, o = info & 3;
      if (kl < 0 || kl >= nk) continue;
      const int j = sfloc[e];
      const int n = V.a(kc + kl)[j];
      const float s = sface[sl];
      const float* bp = V.region + kl * 5 * kvs + j;
      const int64_t at = (x.s0 * NF + e) * 5;
      float qv[5][NTP];
      load_q<NTP>(V.sq + n * SQ, qv);
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        float qb = 0.f;
#pragma unroll
        for (int t = 0; t < NT; ++t) qb += ref.w[t] * qv[v][t];
        const float f = o == 0 ? (bp[v * kvs] + bp[v * kvs + NP]) + bp[v * kvs + 2 * NP]
                               : -bp[v * kvs + (o - 1) * NP];
        sqo[at + v] = x.dt * qb;
        sfn[at + v] = s * f;
      }
    }
    __syncthreads();
    pc_contract_t<N, W>(nk * 5, kvs);
    __syncthreads();
#pragma unroll
    for (int r = 0; r <= kPcOver; ++r) {
      const int lim = (kc + nk) << 6;
      int w = cur[r] < cend[r] ? V.sinc[cur[r]] : lim;
      while (w < lim) {
        const float* src = V.region + ((w >> 6) - kc) * 5 * kvs + (w & 63);
        cur[r] += cstep[r];
        w = cur[r] < cend[r] ? V.sinc[cur[r]] : lim;
#pragma unroll
        for (int v = 0; v < 5; ++v) vacc[r][v] += src[v * kvs];
      }
    }
  }
  if (warp < x.nlong) {
#pragma unroll
    for (int v = 0; v < 5; ++v)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) vacc[0][v] += __shfl_xor_sync(0xffffffffu, vacc[0][v], o);
    if (lane) node[0] = -1;
  }
  float* const vol = (float*)m.vol;
#pragma unroll
  for (int r = 0; r <= kPcOver; ++r)
    if (node[r] >= 0)
#pragma unroll
      for (int v = 0; v < 5; ++v) vol[(x.n0 + node[r]) * 5 + v] = vacc[r][v];
}

// All cells of a kind from the queue: VISC = false the cells without viscosity and heat conduction, VISC =
// true the others; with both kinds present (`mixed`: the limiter's mu_i) each passes over the other's.
// One path for both would spill the viscous fluxes' registers in the inviscid cells too.  False when a
// bounded wait gave up.  Each kind has its own barrier and shared scalars: handed in by reference they
// cost the eight-warp kernels a third (8^3 P2 131 us per launch against 97, 4^3 P1 50 against 39).
template <int N, int W, bool VISC>
__device__ __forceinline__ bool predictor_cells(const Batch& bt, const PcRef& ref, int diag, int smem_bytes,
                                                bool mixed) {
  using P = Pc<N>;
  constexpr int NP = P::NP, NT = P::NT, NF = P::NF, NTP = P::NTP, SQ = P::SQ, THR = 32 * W;
  static_assert(P::FB == (P::NNT - 1) * 512 + (20 * NTP - (P::NNT - 1) * 32) * 16, "fragment bytes");
  PcCell& x = pc_shared().x;
  auto& sred = pc_shared().red;
  unsigned char* const srec = pc_smem + pc_up(sizeof(PcShared));
  __shared__ __align__(8) uint64_t sbar;
  __shared__ int sCell, sAbort;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    mbar_init(&sbar, 1);
    sAbort = 0;
    pc_shared().ref = ref;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  uint32_t phase = 0;
  // next cell of this kernel's kind from the queue (index order, or the schedule's cost order)
  int* const queue = bt.work + (VISC ? 1 : 0);
  auto take = [&]() {
    for (;;) {
      const int w = atomicAdd(queue, 1);
      if (w >= bt.cpre[bt.nh]) return w;
      const int g = bt.order != nullptr ? bt.order[w] : w;
      if (mixed) {
        const int hm = batch_find(bt.cpre, bt.nh, g);
        const DevMesh& m = bt.tab[hm];
        const double mu = m.mu[g - bt.cpre[hm]];
        if (((float)mu != 0.f || (float)cell_kappa(m, mu) != 0.f) != VISC) continue;
      }
      return g;
    }
  };
  int next = 0;
  if (tid == 0) next = take();

  for (;;) {
    if (tid == 0) sCell = next;
    __syncthreads();
    const int64_t gc = sCell;
    if (gc >= bt.cpre[bt.nh]) break;
    if (tid == 0) next = take();  // the next cell's index arrives while this one is computed
    {
      const int hm = batch_find(bt.cpre, bt.nh, gc);
      const DevMesh& m = bt.tab[hm];
      const int64_t c = gc - bt.cpre[hm];
      const int64_t n0 = m.node_ptr[c], kbase = m.sub_ptr[c], s0 = m.slot_ptr[c];
      const int Ni = (int)(m.node_ptr[c + 1] - n0), S = (int)(m.sub_ptr[c + 1] - kbase);
      const int ns = (int)(m.slot_ptr[c + 1] - s0);
      const uint32_t* const m16 = m16_block(m, c);
      const uint32_t gbytes = (uint32_t)gat_bytes(Ni, S, ns, NP, NF);
      const int head = minv_split_head(Ni);
      const uint32_t o_gat = (uint32_t)(pc_up(sizeof(PcShared)) + pc_up((size_t)S * P::REC)),
                     o_exp = o_gat + (uint32_t)pc_up(gbytes), o_uh = o_exp + head * 4,
                     o_q = o_uh + (uint32_t)pc_up((size_t)Ni * 20), o_region = o_q + (uint32_t)pc_up((size_t)Ni * SQ * 4);
      // records and gather block by two bulk copies; meanwhile u^, and M_i^-1 on its way into L2
      if (tid == 0) {
        // every thread's accesses to these bytes (generic proxy) precede the copies: each fenced
        // before the barrier above
        mbar_expect_tx(&sbar, (uint32_t)(S * P::REC) + gbytes);
        bulk_g2s(srec, m.sub32 + (size_t)kbase * P::REC, (uint32_t)(S * P::REC), &sbar);
        bulk_g2s(pc_smem + o_gat, m.gat + gat_start(n0, kbase, s0, c, NP, NF), gbytes, &sbar);
        const double mu = m.mu[c];
        x.m = &m;
        x.m16 = m16 + head;
        x.c = c;
        x.n0 = n0;
        x.s0 = s0;
        x.Ni = Ni;
        x.S = S;
        x.ns = ns;
        x.nks = (Ni + 15) / 16;
        x.room = smem_bytes - (int)o_region;
        x.o_gat = o_gat;
        x.o_inc = o_gat + (uint32_t)gat_up(2 * (size_t)(2 * Ni + 3));
        x.o_exp = o_exp;
        x.o_uh = o_uh;
        x.o_q = o_q;
        x.o_region = o_region;
        x.dt = (float)*m.dt;
        x.gam = (float)m.gamma;
        x.gm1 = x.gam - 1.f;
        x.mu = (float)mu;
        x.kap = (float)cell_kappa(m, mu);
      }
      if (warp == W - 1) {
        const uint32_t bytes = (uint32_t)(minv_split_words(Ni) - head) * 4u;
        for (uint32_t o = lane * 16384u; o < bytes; o += 32 * 16384u)
          asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(
                           reinterpret_cast<const unsigned char*>(m16 + head) + o),
                       "r"(min(16384u, bytes - o))
                       : "memory");
      }
      for (int e = tid; e < head; e += THR) reinterpret_cast<uint32_t*>(pc_smem + o_exp)[e] = m16[e];
      float* const suh = reinterpret_cast<float*>(pc_smem + o_uh);
      for (int e = tid; e < 5 * Ni; e += THR) suh[e] = (float)m.u[n0 * 5 + e];
      if (tid == 0) {
        if (!mbar_wait_bounded(&sbar, phase & 1u, m.first_wait_polls)) {
          atomicOr(&m.flags[F_TIMEOUT], 1);
          sAbort = 1;
        } else {
          x.nlong = min((int)*reinterpret_cast<const uint16_t*>(pc_smem + o_gat), W);
          x.slots = Ni + 31 * x.nlong;
        }
      }
    }
    __syncthreads();
    if (sAbort) {  // a copy that never completed: wait once more (bounded), then leave
      if (tid == 0) (void)mbar_wait_bounded(&sbar, phase & 1u);
      return false;
    }
    phase ^= 1u;

    int it = 0;
    bool conv = false;
    while (!conv && it < x.m->picard_max) {
      ++it;
      pc_rhs<N, W, VISC>(it == 1);
      __syncthreads();
      float2 rq = it == 1 ? pc_apply<N, W, true>() : pc_apply<N, W, false>();
      rq.x = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(rq.x)));
      rq.y = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(rq.y)));
      if (lane == 0) {
        sred[0][warp] = rq.x;
        sred[1][warp] = rq.y;
      }
      __syncthreads();  // q is complete, the fragments are free
#pragma unroll
      for (int w = 0; w < W; ++w) {
        rq.x = fmaxf(rq.x, sred[0][w]);
        rq.y = fmaxf(rq.y, sred[1][w]);
      }
      conv = rq.x <= (float)x.m->tol * fmaxf(1.f, rq.y);
    }
    if (tid == 0) {
      x.m->iters[x.c] = it;
      if (!conv) atomicAdd(&x.m->flags[F_NONCONV], 1);
    }
    pc_epilogue<N, W, VISC>();
    if (diag && x.m->qbar_diag) {
      const float* sq = reinterpret_cast<const float*>(pc_smem + x.o_q);
      for (int e = tid; e < x.Ni * 5; e += THR) {
        float acc = 0.f;
#pragma unroll
        for (int t = 0; t < NT; ++t) acc += pc_shared().ref.w[t] * sq[e * NTP + t];
        x.m->qbar_diag[x.n0 * 5 + e] = (double)x.dt * (double)acc;
      }
    }
    // the next cell's bulk copies (async proxy) overwrite memory read and written here
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  return true;
}

// W warps per block, at least MB blocks per SM (register limit).  KINDS: 1 inviscid cells, 2 viscous cells, 3
// both, the viscous ones, which take longer, first: in one launch the blocks go from one kind to the
// other without waiting for the slowest (us, two launches and one: four steps of a batch of
// P2 meshes of which some are limited 2,822 and 2,567, two of a limited 15^3 P3 mesh 2,982 and 2,848).
template <int N, int W, int MB, int KINDS>
__global__ void __launch_bounds__(32 * W, MB) predictor_cells_kernel(const __grid_constant__ Batch bt,
                                                                     const __grid_constant__ PcRef ref, int diag,
                                                                     int smem_bytes) {
  if constexpr (KINDS & 2)
    if (!predictor_cells<N, W, true>(bt, ref, diag, smem_bytes, KINDS == 3)) return;
  if constexpr (KINDS == 3) __syncthreads();  // the last cell of one kind is done with what the next sets up
  if constexpr (KINDS & 1) (void)predictor_cells<N, W, false>(bt, ref, diag, smem_bytes, KINDS == 3);
}

// ----------------------------------------------------------------------------------------
// FP32 corrector on the split M_i^-1 (Sec. 4.4), one block of W warps per cell.
//   f[slot][a] = 2 area sum_b Z^[a][b] G[b]     (a thread per slot and variable, once per slot)
//   r = vol - sum over the node's face incidences of f   (fixed order)
//   du = M_i^-1 r on the tensor cores: the tiles of the predictor's first iteration (5 columns), with the
//        leading products added up outside the tensor cores, which truncate, at N <= 2, where sums are
//        short, the product of the low parts, and at N = 1 r in three FP16 parts (all of its 24 bits): no
//        further off than FP32 multiply-adds over FP32 rows
//   u += du + (T - w_i . du) / |P_i|            (FP64: T = exact cell total of r, see
//                                                corrector_f32_kernel)
// What bounds it: M_i^-1 from HBM, once per step.  The lower triangle in 16-bit pairs is 53 % of the
// FP32 rows that corrector_f32_kernel streams (75 % of the copy rate there); each tile is read a
// second time for its mirror, from L2, which holds the cells in flight as long as few blocks
// share an SM (three: 2,210 us at 32^3 P3, two 2,841, before the sums outside the tensor cores).  FP64 work per node is kept to the update
// itself and conversions are integer instructions: with ten FP64 reductions per warp and FP64
// admissibility tests the launch took 3,017 us.
// us per launch, corrector_f32_kernel and here: 32^3 P3 3,155 and 2,264 (1,500 for the bytes at the copy
// rate), 16^3 P3 465 and 316, 21^3 P2 432 and 200, 24^3 P1 436 and 121, 8^3 P2 49 and 26.
__device__ __forceinline__ double f64_of(float x) {
  const unsigned b = __float_as_uint(x), e = b >> 23 & 255u;
  if (e - 1u >= 254u) return (double)x;  // zero, denormal, infinity, NaN
  return __hiloint2double((int)((b & 0x80000000u) | ((b & 0x7fffffffu) >> 3) + 0x38000000u), (int)(b << 29));
}

// Parts of the split right-hand side, and its bytes per 16 rows: two parts as the predictor's, behind them the
// third.  Relative L2 error of M_i^-1 r against 64 bits (random r, smooth du; FP32 multiply-adds), without the
// product of the low parts P3 1.2e-7, 3.4e-7 (3.2e-7, 5.2e-7), with it P2 1.0e-7, 3.2e-7 (1.9e-7, 3.4e-7), with
// the third part too P1 0.7e-7, 1.5e-7 (0.9e-7, 1.8e-7).
template <int N>
constexpr int corr_parts = N == 1 ? 3 : 2;
template <int N>
constexpr int corr_frag = 160 * corr_parts<N>;

template <int N, int W>
__global__ void __launch_bounds__(32 * W, N == 3 ? 3 : (N == 2 ? 8 : 24)) corrector_cells_kernel(
    const __grid_constant__ Batch bt, const __grid_constant__ CorrRef ref) {
  constexpr int NF = nf_of(N), THR = 32 * W, DP = N == 1 ? 2 : kPcDeep, FB = corr_frag<N>;
  constexpr bool three = corr_parts<N> == 3;
  extern __shared__ __align__(128) unsigned char pc_smem[];
  __shared__ double sred[10][W];
  __shared__ float smax[5][W];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t gc = blockIdx.x;
  const int h = batch_find(bt.cpre, bt.nh, gc);
  const DevMesh& m = bt.tab[h];
  const int64_t c = gc - bt.cpre[h];
  const int64_t n0 = m.node_ptr[c], s0 = m.slot_ptr[c];
  const int Ni = (int)(m.node_ptr[c + 1] - n0), ns = (int)(m.slot_ptr[c + 1] - s0), nks = (Ni + 15) / 16;
  const uint32_t* const m16 = m16_block(m, c);
  unsigned char* const frag = pc_smem;                                   // [nks][FB] split right-hand side
  float* const sr = reinterpret_cast<float*>(pc_smem + nks * FB);        // [N_i][5] r (rows scaled), then du
  float* const sf = sr + ((Ni * 5 + 3) & ~3);                            // [ns][NF][5] face integrals
  const float* const vol = (const float*)m.vol;
  const float* const sG = (const float*)m.slot_G;
  const int8_t* const ex = reinterpret_cast<const int8_t*>(m16);
  const uint32_t* const tiles = m16 + minv_split_head(Ni);
  if (warp == W - 1) {  // M_i^-1 on its way into L2
    const uint32_t bytes = (uint32_t)(minv_split_words(Ni) - minv_split_head(Ni)) * 4u;
    for (uint32_t o = lane * 8192u; o < bytes; o += 32 * 8192u)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(reinterpret_cast<const unsigned char*>(tiles) + o),
                   "r"(min(8192u, bytes - o))
                   : "memory");
  }
  // face integrals and the FP64 cell total of the update, item (slot, variable)
  double tot = 0.0;  // of variable tid % 5 (the stride keeps it)
  constexpr int FS = THR / 5 * 5;
  for (int e = tid; e < ns * 5 && tid < FS; e += FS) {
    const int sl = e / 5, v = e - sl * 5;
    const float* g = sG + (s0 + sl) * NF * 5 + v;
    const double twoA = 2.0 * m.slot_geo[(s0 + sl) * 4 + 3];
    const float tA = f32_of(twoA);
    float x[NF];
#pragma unroll
    for (int b = 0; b < NF; ++b) x[b] = g[b * 5];
    double z = 0.0;
#pragma unroll
    for (int b = 0; b < NF; ++b) z += ref.zs[b] * f64_of(x[b]);
    tot -= twoA * z;
#pragma unroll
    for (int a = 0; a < NF; ++a) {
      float f = 0.f;
#pragma unroll
      for (int b = 0; b < NF; ++b) f += ref.Z[a][b] * x[b];
      sf[(sl * NF + a) * 5 + v] = tA * f;
    }
  }
  __syncthreads();
  float mx[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
  for (int n = tid; n < Ni; n += THR) {
    float acc[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) acc[v] = vol[(n0 + n) * 5 + v];
    const float f0 = pow2f(-(int)ex[n]);
    const int64_t p1 = m.finc_ptr[n0 + n + 1];
    for (int64_t p = m.finc_ptr[n0 + n]; p < p1; ++p) {
      const uint32_t w = m.finc[p];
      const float* f = sf + ((w >> 4) * NF + (w & 15)) * 5;
#pragma unroll
      for (int v = 0; v < 5; ++v) acc[v] -= f[v];
    }
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      acc[v] *= f0;
      sr[n * 5 + v] = acc[v];
      mx[v] = fmaxf(mx[v], fabsf(acc[v]));
    }
  }
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    const float x = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(mx[v])));
    if (lane == 0) smax[v][warp] = x;
  }
  __syncthreads();
  // split right-hand side in fragment order, a power of two per variable
  float sc[5], isc[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    float x = smax[v][0];
#pragma unroll
    for (int w = 1; w < W; ++w) x = fmaxf(x, smax[v][w]);
    const int e = f16_scale_exp(__float_as_uint(x));
    sc[v] = __uint_as_float((uint32_t)e << 23);
    isc[v] = __uint_as_float((uint32_t)(254 - e) << 23);
  }
  for (int n = tid; n < 16 * nks; n += THR) {
    unsigned char* const rows = frag + (n >> 4) * FB;
    const int at = ((n >> 3) & 1) * 4 + (n & 1) * 2, ln = (n & 7) >> 1;
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      const float y = n < Ni ? sr[n * 5 + v] * sc[v] : 0.f;
      const __half hi = __float2half_rn(y);
      const float rest = y - __half2float(hi);
      const __half lo = __float2half_rn(rest);
      unsigned char* const b = rows + (v * 4 + ln) * 16 + at;
      *reinterpret_cast<__half*>(b) = hi;
      *reinterpret_cast<__half*>(b + 8) = lo;
      if constexpr (three)
        *reinterpret_cast<__half*>(rows + 320 + (v * 4 + ln) * 8 + at) = __float2half_rn(rest - __half2float(lo));
    }
  }
  __syncthreads();
  for (int mt = warp; mt < nks; mt += W) {
    float acc[4] = {0.f, 0.f, 0.f, 0.f}, low[4] = {0.f, 0.f, 0.f, 0.f};
    const uint32_t* const a0 = tiles + lane * 4;
    uint4 ah[DP], al[DP];
    auto load = [&](int s, int ks) {
      const uint32_t* t = a0 + tri_tile(mt, min(ks, nks - 1)) * 256;
      ah[s] = ldg_stream(t);
      al[s] = ldg_stream(t + 128);
    };
    auto step = [&](int s, int ks) {
      const unsigned char* const f = frag + ks * FB;
      const uint4 b = lane < 20 ? *reinterpret_cast<const uint4*>(f + lane * 16) : make_uint4(0, 0, 0, 0);
      uint4 x = ah[s], l = al[s];
      if (ks > mt) {  // above the diagonal: the mirrored tile
        x = transpose16(x);
        l = transpose16(l);
      }
      // A tensor-core accumulator is truncated after every product: sums of 20 steps would be off by
      // 1e-6 of themselves.  The leading products go to an accumulator of their own per step.
      float lead[4] = {0.f, 0.f, 0.f, 0.f};
      mma_f16(lead, x, b.x, b.y);
      if constexpr (three) {
        const uint2 b3 = lane < 20 ? *reinterpret_cast<const uint2*>(f + 320 + lane * 8) : make_uint2(0, 0);
        mma_f16(low, x, b3.x, b3.y);
      }
      if constexpr (N <= 2) mma_f16(low, l, b.z, b.w);
      mma_f16(low, l, b.x, b.y);
      mma_f16(low, x, b.z, b.w);
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[i] += lead[i];
    };
#pragma unroll
    for (int s = 0; s < DP; ++s) load(s, s);
    int ks = 0;
    for (; ks + DP <= nks; ks += DP) {
#pragma unroll
      for (int s = 0; s < DP; ++s) {
        step(s, ks + s);
        load(s, ks + s + DP);
      }
    }
#pragma unroll
    for (int s = 0; s < DP - 1; ++s)
      if (ks + s < nks) step(s, ks + s);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int v = 2 * (lane & 3) + (i & 1), n = mt * 16 + (lane >> 2) + (i >> 1) * 8;
      if (v < 5 && n < Ni) {
        float si = isc[0];
#pragma unroll
        for (int q = 1; q < 5; ++q)
          if (v == q) si = isc[q];
        sr[n * 5 + v] = ((acc[i] + low[i]) * pow2f(-(int)ex[n] - 13)) * si;
      }
    }
  }
  __syncthreads();
  // FP64 totals: target (per thread one variable) minus w . du, in a fixed order.  The FP64 pipe takes
  // 64 cycles per warp instruction and scheduler: the five sums share their shuffles (lanes 0-15
  // keep one sum, 16-31 another, and so on), one warp adds up the warps' parts.
  double d[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (int n = tid; n < Ni; n += THR) {
    const double w = -m.wvec[n0 + n];
#pragma unroll
    for (int v = 0; v < 5; ++v) d[v] += w * f64_of(sr[n * 5 + v]);
  }
  if (tid < FS && tid < ns * 5) {
    const int tv = tid % 5;
#pragma unroll
    for (int v = 0; v < 5; ++v)
      if (tv == v) d[v] += tot;
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {  // 8 sums over 32 lanes -> one sum per lane, over 4 lanes
    const int half = 4 >> k, o = 16 >> k;
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const double send = up ? d[i] : d[i + half], keep = up ? d[i + half] : d[i];
      d[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  d[0] += __shfl_xor_sync(0xffffffffu, d[0], 2);
  d[0] += __shfl_xor_sync(0xffffffffu, d[0], 1);
  if ((lane & 3) == 0 && lane < 20) sred[lane >> 2][warp] = d[0];  // lanes 4 v .. 4 v + 3 hold sum v
  __syncthreads();
  if (warp == 0) {
    double x = 0.0;
    if (lane < 5) {
#pragma unroll
      for (int w = 0; w < W; ++w) x += sred[lane][w];
      sred[5 + lane][0] = x / m.cell_vol[c];
    }
  }
  __syncthreads();
  double corr[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) corr[v] = sred[5 + v][0];
  for (int n = tid; n < Ni; n += THR) {
    double* un = m.u + (n0 + n) * 5;
    double x[5];
    bool ok = true;
    float xf[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      x[v] = un[v] + (f64_of(sr[n * 5 + v]) + corr[v]);
      un[v] = x[v];
      xf[v] = f32_head(x[v], ok);
    }
    // rho > 0 and p > 0, with p > 0 tested as rho E > |rho u|^2 / 2 (no division): in FP32 where the
    // margin is beyond its error, else in FP64, which also sees infinities and NaN
    const float a = xf[0] * xf[4], b = 0.5f * (xf[1] * xf[1] + xf[2] * xf[2] + xf[3] * xf[3]);
    if (ok && xf[0] > 0.f && xf[4] > 0.f && a > 1e-30f && a < 1e37f && a - b > 0x1p-18f * (a + b)) continue;
    bool bad = false;
#pragma unroll
    for (int v = 0; v < 5; ++v) bad |= !isfinite(x[v]);
    const double pr = x[0] * x[4] - 0.5 * (x[1] * x[1] + x[2] * x[2] + x[3] * x[3]);
    if (bad || !(x[0] > 0.0) || !(pr > 0.0)) atomicOr(&m.flags[F_NONFINITE], 8);
  }
}

}  // namespace afe
