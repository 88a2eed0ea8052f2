// FP64 space-time predictor (Sec. 4.3, Eqs. ADER-localCauchy, ader4, TAvectors) with the M_i^-1 product on
// the tensor cores.
//
// GB300 has few FP64 units: a warp's FP64 instruction takes 17 cycles of its SM (measured; 1.9
// multiply-adds per cycle and SM, the FP64 tensor instructions no more), so the time of this
// predictor is its count of FP64 instructions.  Against predictor_kernel:
//   - Y = M_i^-1 RHS (more than half of the arithmetic) is formed exactly in integers: both
//     factors as 62-bit fixed point in eight balanced digits of base 256, the products of digits
//     on mma.sync.m16n8k16 with FP16 operands (digits are exact in FP16) and FP32 accumulators,
//     which hold sums below 2^24 exactly: 112 terms of up to eight digit pairs.  The levels are
//     added up as integers and rounded once.  Digit pairs below 2^-64 of the largest product are left
//     out.  M_i^-1 is scaled by powers of two per row and column to a unit diagonal (|entries| <= 1
//     then, as it is positive definite) and the right-hand side per column, so that the error is
//     2^-58 of the scaled product's size, below FP64's own summation error.  36 tensor
//     instructions (77 cycles) replace 64 warp FMAs (1,088 cycles) per 16 x 16 x 8 block.
//   - The first iteration starts from q^0 = u^ at every time node: one time slice serves all.
//   - The flux goes straight to its contravariant form (half the arithmetic), with one
//     reciprocal refined by Newton steps.
//   - The stiffness contractions are digit products too, with the digits of S^ from a table.
// Error of the product against 64 bits on random rows of 320 entries: 1e-18 to 2e-16 of the sum of
// magnitudes, FP64 summation 6e-18 to 8e-16; of the whole step the same as before (3.3e-16 at 8^3 P3).
// us per launch, predictor_kernel and here: 8^3 P3 31,240 and 7,865 (11,430 with the contraction in FP64),
// 10^3 P2 12,740 and 5,390 (5,650), 6^3 P1 984 and 450.  What bounds it now, per cell-iteration at P3: the
// digit products' tensor instructions (160 k of 545 k cycles) and the integer work around them, the
// fluxes' FP64 instructions (100 k); at P2 the fluxes; at P1 the latency of an iteration's barriers.
// One block per cell, persistent; the cell's q, u^ and lists in shared memory; data flow, lists
// and gather order as in predictor_cells.cuh.
#pragma once

#include <cuda_fp16.h>

#include <cstring>

#define AFE_SREF_F64 1
#include "predictor_cells.cuh"
#include "predictor_f64.hpp"

namespace afe {

template <int N>
struct Pd {
  static constexpr int NP = np_of(N), NT = N + 1, NF = nf_of(N), NTP = f32_ntp(N);
  static constexpr int SQ = 5 * NT;              // doubles of q per node, time innermost
  static constexpr int KKS = (3 * NP) | 1;       // column of pre-contracted fluxes (odd: conflict-free)
  static constexpr int KST = (3 * NP + 15) / 16;  // its 16-row steps
  static constexpr int MT = (NP + 15) / 16;       // 16-row tiles of its contraction's result
  // bytes of a chunk per column: FP64 values, and their digits (1 KB per eight columns and step)
  static constexpr int CB = KKS * 8 + (N == 1 ? 0 : KST * 128);  // (P1 contracts in FP64)
  static constexpr int NNT = N == 1 ? 2 : 3;     // 8-column tiles of RHS / Y: column v NTP + t
  // bytes of the digit fragments per 16 rows: 32 per lane in use of every column tile
  static constexpr int FB = 20 * NTP * 32, FB1 = 20 * 32;
};

// At the start of dynamic shared memory.
struct PdShared {
  const DevMesh* m;
  const uint32_t* dig;
  int64_t c, n0, s0, k0;
  int Ni, S, ns, nks, nlong, slots, room;
  uint32_t o_inc, o_geo, o_A, o_exp, o_uh, o_q, o_region;
  double dt, mu, kap;
  int ev[5];        // exponent of the right-hand side's power of two, per variable
  int ired[5][16];
  long long red[2][16];
  PdRef ref;
  double dkw[4][4], dkws[4];  // dt times the time-basis constants
};
constexpr int kPdNone = 20000;  // exponent of a variable with an infinite or NaN entry
constexpr int kPdGat = (int)((sizeof(PdShared) + 127) / 128 * 128);  // the gather block follows
__device__ __forceinline__ PdShared& pd_shared() { return *reinterpret_cast<PdShared*>(pc_smem); }

template <int N>
__host__ __device__ constexpr size_t pd_fixed(int n, int s, int ns) {
  return kPdGat + pc_up(gat_bytes(n, s, ns, Pd<N>::NP, Pd<N>::NF)) + pc_up((size_t)s * 80) +
         pc_up((size_t)s * Pd<N>::NP * 2) + pc_up((size_t)n * 2) + pc_up((size_t)n * 40) + pc_up((size_t)n * Pd<N>::SQ * 8);
}
template <int N>
__host__ __device__ constexpr size_t pd_over(int slots, int thr) {
  return slots > thr ? (size_t)(slots - thr) * Pd<N>::SQ * 8 : 0;
}
template <int N>
__host__ __device__ constexpr size_t pd_need(int n, int s, int ns, int thr) {
  // the fragments beside the sums past the second slot; two sub-tets beside all sums
  const size_t frag = (size_t)((n + 15) / 16) * Pd<N>::FB + pd_over<N>(pc_slots(n, thr), 2 * thr);
  const size_t chunk = (size_t)(2 * 5 * Pd<N>::NT + 8) * (Pd<N>::CB + 4) + pd_over<N>(pc_slots(n, thr), thr);
  return pd_fixed<N>(n, s, ns) + (frag > chunk ? frag : chunk);
}

// 1 / x: the hardware's approximation (20 bits) and two Newton steps, y += y (1 - x y).
__device__ __forceinline__ double recip(double x) {
  if ((unsigned)((__double2hiint(x) >> 20 & 0x7ff) - 123) > 1800u) return 1.0 / x;
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  y = fma(y, fma(-x, y, 1.0), y);
  return fma(y, fma(-x, y, 1.0), y);
}

// x 2^(62 - e) to nearest as a 64-bit integer plus 128 in every byte, for |x| < 2^e: the bytes are the
// balanced base-256 digits plus 128.
__host__ __device__ __forceinline__ unsigned long long digits(double x, int e) {
#ifdef __CUDA_ARCH__
  const long long b = __double_as_longlong(x);
#else
  long long b;
  std::memcpy(&b, &x, 8);
#endif
  const int ex = (int)(b >> 52) & 0x7ff;
  unsigned long long m = ((unsigned long long)b & 0xfffffffffffffull) | (ex ? 1ull << 52 : 0ull);
  const int sh = (ex ? ex : 1) - 1075 + 62 - e;  // value = m 2^(ex - 1075)
  if (sh >= 0) m <<= sh < 10 ? sh : 10;
  else if (sh > -63) m = (m + (1ull << (-sh - 1))) >> -sh;
  else m = 0;
  const long long v = b < 0 ? -(long long)m : (long long)m;
  return (unsigned long long)v + 0x8080808080808080ull;
}
// Two biased digits (bytes) as the FP16 pair digit, digit: 1024 + byte has the byte as its last bits.
__device__ __forceinline__ uint32_t digit_pair(uint32_t w, uint32_t sel) {
  const uint32_t h = __byte_perm(w, 0x64646464u, sel);
  const __half2 r = __hsub2(*reinterpret_cast<const __half2*>(&h), __half2half2(__ushort_as_half(0x6480)));  // 1152
  return *reinterpret_cast<const uint32_t*>(&r);
}
// The exact product of digit tiles: a 16 x (16 steps) row of tiles at `at` (16-byte groups of this
// lane, 512 words per step) with an 8-column operand at `bt` (this lane's 32 bytes, `stride` bytes per
// step; the digit zero where !on).  The product is hi 2^32 + lo, times 2^56 of the factors' units.
__device__ __forceinline__ void digit_product(const uint32_t* at, const unsigned char* bt, int stride, bool on, int steps,
                                              long long (&hi)[4], long long (&lo)[4]) {
  uint4 nx[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) nx[q] = ldg_stream(at + q * 128);
#pragma unroll
  for (int i = 0; i < 4; ++i) hi[i] = lo[i] = 0;
  for (int k0 = 0; k0 < steps; k0 += 7) {  // 112 columns: what the FP32 accumulators hold exactly
    float acc[8][4];
#pragma unroll
    for (int l = 0; l < 8; ++l)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[l][i] = 0.f;
    const int k1 = min(k0 + 7, steps);
#pragma unroll 1
    for (int ks = k0; ks < k1; ++ks) {
      uint4 A[8];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t w[4] = {nx[q].x, nx[q].y, nx[q].z, nx[q].w};
#pragma unroll
        for (int s = 0; s < 2; ++s)
          A[2 * q + s] = make_uint4(digit_pair(w[2 * s], 0x4140), digit_pair(w[2 * s], 0x4342),
                                    digit_pair(w[2 * s + 1], 0x4140), digit_pair(w[2 * s + 1], 0x4342));
      }
      const uint32_t* t = at + (size_t)min(ks + 1, steps - 1) * 512;
#pragma unroll
      for (int q = 0; q < 4; ++q) nx[q] = ldg_stream(t + q * 128);
      const uint4 z4 = make_uint4(0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u);
      const uint4 b0 = on ? *reinterpret_cast<const uint4*>(bt + ks * stride) : z4;
      const uint4 b1 = on ? *reinterpret_cast<const uint4*>(bt + ks * stride + 16) : z4;
      const uint32_t b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const uint32_t c0 = digit_pair(b[u], 0x4140), c1 = digit_pair(b[u], 0x4342);
#pragma unroll
        for (int s = 0; s + u < 8; ++s) mma_f16(acc[s + u], A[s], c0, c1);
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      int a[8];
#pragma unroll
      for (int l = 0; l < 8; ++l) a[l] = __float2int_rn(acc[l][i]);
      hi[i] += ((long long)a[0] << 24) + ((long long)a[1] << 16) + ((long long)a[2] << 8) + a[3];
      lo[i] += ((long long)a[4] << 24) + ((long long)a[5] << 16) + ((long long)a[6] << 8) + a[7];
    }
  }
}
// (hi 2^32 + lo) 2^k, rounded once, for |hi|, |lo| < 2^51; none: a factor was infinite or NaN.  The integers
// enter as the last bits of 1.5 2^52 + integer, because the conversion instructions go through
// the FP64 pipe too.
__device__ __forceinline__ double digit_value(long long hi, long long lo, int k, bool none) {
  const double h = fma(__longlong_as_double(hi + 0x4338000000000000ll), 0x1p32, -0x1.8p84);  // hi 2^32, exact
  const double s = h + (__longlong_as_double(lo + 0x4338000000000000ll) - 0x1.8p52);
  if (none) return __hiloint2double(0x7ff80000, 0);
  if ((unsigned)(k + 900) <= 1800u) return s * __hiloint2double((1023 + k) << 20, 0);
  k = max(-2000, min(2000, k));
  const int k2 = k / 2;
  return s * __hiloint2double((1023 + k2) << 20, 0) * __hiloint2double((1023 + k - k2) << 20, 0);
}

__device__ __forceinline__ void contravariant_flux(const double (&Q)[5], const double (&g)[9], double gm1,
                                                   double out[3][5]) {
  const double ir = recip(Q[0]);
  const double v0 = Q[1] * ir, v1 = Q[2] * ir, v2 = Q[3] * ir;
  const double p = gm1 * (Q[4] - 0.5 * (Q[1] * v0 + Q[2] * v1 + Q[3] * v2));
  const double H = Q[4] + p;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double U = g[3 * d] * v0 + g[3 * d + 1] * v1 + g[3 * d + 2] * v2;
    out[d][0] = Q[0] * U;
#pragma unroll
    for (int a = 0; a < 3; ++a) out[d][1 + a] = Q[1 + a] * U + p * g[3 * d + a];
    out[d][4] = H * U;
  }
}

template <int N>
struct PdView {
  const uint16_t *slist, *sinc;
  const int16_t* sexp;
  const uint16_t* sA;             // [S][Np] node ids
  const double *sgeo, *suh;       // [S][10] adj(J), det J; u^
  double *sq, *region;
  __device__ __forceinline__ PdView()
      : slist(reinterpret_cast<const uint16_t*>(pc_smem + kPdGat)),
        sinc(reinterpret_cast<const uint16_t*>(pc_smem + pd_shared().o_inc)),
        sexp(reinterpret_cast<const int16_t*>(pc_smem + pd_shared().o_exp)),
        sA(reinterpret_cast<const uint16_t*>(pc_smem + pd_shared().o_A)),
        sgeo(reinterpret_cast<const double*>(pc_smem + pd_shared().o_geo)),
        suh(reinterpret_cast<const double*>(pc_smem + pd_shared().o_uh)),
        sq(reinterpret_cast<double*>(pc_smem + pd_shared().o_q)),
        region(reinterpret_cast<double*>(pc_smem + pd_shared().o_region)) {}
};

// Gradient columns of a chunk (viscous cells), as pc_gradients.
template <int N, int THR>
__device__ __forceinline__ void pd_gradients(int kc, int nk, int nte, bool first) {
  using P = Pd<N>;
  const PdView<N> V;
  for (int col = threadIdx.x; col < nk * 5 * nte; col += THR) {
    const int kv = col / nte, t = col - kv * nte, kl = kv / 5, v = kv - kl * 5;
    const uint16_t* Ak = V.sA + (kc + kl) * P::NP;
    double q[P::NP];
#pragma unroll
    for (int l = 0; l < P::NP; ++l) q[l] = first ? V.suh[Ak[l] * 5 + v] : V.sq[Ak[l] * P::SQ + v * P::NT + t];
    SrefFP64<N>::gradient(q, V.region + col * P::KKS);
  }
}

// Physical flux of a viscous cell at a node whose reference gradients sit in the buffer columns
// (vstride between variables).
template <int N>
__device__ __forceinline__ void pd_flux_visc(const PdShared& x, const double (&Q)[5], const double (&g)[9], double idet,
                                             const double* gcol, int vstride, double F[3][5]) {
  double gq[3][5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    const double x0 = gcol[v * vstride], x1 = gcol[v * vstride + Pd<N>::NP], x2 = gcol[v * vstride + 2 * Pd<N>::NP];
#pragma unroll
    for (int e = 0; e < 3; ++e) gq[e][v] = (g[e] * x0 + g[3 + e] * x1 + g[6 + e] * x2) * idet;
  }
  phys_flux<double>(Q, gq, true, x.mu, x.kap, x.m->gamma, x.m->Rgas, F);
}

__device__ __forceinline__ void contract_adj(const double (&g)[9], double scale, const double (&F)[3][5],
                                             double out[3][5]) {
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int v = 0; v < 5; ++v)
      out[d][v] = scale * (g[d * 3] * F[0][v] + g[d * 3 + 1] * F[1][v] + g[d * 3 + 2] * F[2][v]);
}

// Contraction of `cols` columns (`cstride` doubles apart) with S^ or its transpose, in place:
// four lanes per column find its power of two and write its digits as fragments behind the columns
// and their exponents behind those, then (row tile, 8 columns) pairs go over the warps.  A column's
// 882 FP64 multiply-adds at N = 3 would take 15 k cycles per warp of columns, this 2.5 k.
template <int N, int W>
__device__ __forceinline__ void pd_contract(const PdRef& ref, bool transposed, int cols, int cstride) {
  using P = Pd<N>;
  constexpr int NP = P::NP, KK = 3 * NP, KST = P::KST, THR = 32 * W, QN = KST * 4;  // values per lane
  double* const col0 = PdView<N>().region;
  if constexpr (N == 1) {  // 12 values per column: 24 multiply-adds are less than the digits' own work
    for (int c = threadIdx.x; c < cols; c += THR) {
      double acc[NP];
#pragma unroll
      for (int i = 0; i < NP; ++i) acc[i] = 0.0;
      double* b = col0 + (size_t)c * cstride;
      if (transposed) SrefFP64<N>::contract_t(b, acc);
      else SrefFP64<N>::contract(b, acc);
      asm volatile("" ::: "memory");  // the results replace the column
#pragma unroll
      for (int i = 0; i < NP; ++i) b[i] = acc[i];
    }
    return;
  }
  unsigned char* const dig = reinterpret_cast<unsigned char*>(col0) + pc_up((size_t)cols * cstride * 8);
  const int tiles = (cols + 7) / 8;
  int* const dex = reinterpret_cast<int*>(dig + (size_t)tiles * KST * 1024);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // digits: lane quarter u of a column takes rows 16 ks + 2 u, + 1, + 8, + 9 of every step, the two 16-bit
  // halves of a fragment word
  for (int e = tid; e < tiles * 32; e += THR) {
    const int c = e >> 2, u = e & 3;
    const double* b = col0 + (size_t)c * cstride;
    double val[QN];
    int ex = 1;
#pragma unroll
    for (int q = 0; q < QN; ++q) {
      const int kk = (q >> 2) * 16 + 2 * u + (q & 1) + 8 * ((q >> 1) & 1);
      val[q] = c < cols && kk < KK ? b[kk] : 0.0;
      ex = max(ex, __double2hiint(val[q]) >> 20 & 0x7ff);
    }
    ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, 1));
    ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, 2));
    if (u == 0) dex[c] = ex == 0x7ff ? kPdNone : ex - 1022;
#pragma unroll
    for (int ks = 0; ks < KST; ++ks) {
      unsigned long long d[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) d[i] = digits(val[ks * 4 + i], ex - 1022);
      uint32_t w[8];
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        w[s] = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) w[s] |= (uint32_t)(d[i] >> (56 - 8 * s) & 255u) << (8 * i);
      }
      uint4* o = reinterpret_cast<uint4*>(dig + ((size_t)(c >> 3) * KST + ks) * 1024 + ((c & 7) * 4 + u) * 32);
      o[0] = make_uint4(w[0], w[1], w[2], w[3]);
      o[1] = make_uint4(w[4], w[5], w[6], w[7]);
    }
  }
  __syncthreads();
  for (int job = warp; job < tiles * P::MT; job += W) {
    const int ct = job / P::MT, mt = job - ct * P::MT;
    long long hi[4], lo[4];
    digit_product((transposed ? ref.sdig_t : ref.sdig) + (size_t)mt * KST * 512 + lane * 4, dig + (size_t)ct * KST * 1024 + lane * 32, 1024, true, KST, hi, lo);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int c = ct * 8 + 2 * (lane & 3) + (i & 1), row = mt * 16 + (lane >> 2) + 8 * (i >> 1);
      if (c < cols && row < NP) {
        const int ec = dex[c];
        col0[(size_t)c * cstride + row] = digit_value(hi[i], lo[i], 56 - 124 + ref.sexp + ec, ec >= kPdNone);
      }
    }
  }
}

// Sums of V values over the lanes of a warp, in a fixed order, to lane 0: every step halves the values
// a lane holds (V - 1 + a few additions per lane instead of 5 V), then the lanes hand theirs over.
template <int V>
__device__ __forceinline__ void lane_sums(double* r, int lane) {
  double d[V + 1];
#pragma unroll
  for (int i = 0; i < V; ++i) d[i] = r[i];
  d[V] = 0.0;
  constexpr int n1 = (V + 1) / 2, n2 = (n1 + 1) / 2, n3 = (n2 + 1) / 2, n4 = (n3 + 1) / 2, n5 = (n4 + 1) / 2;
  static_assert(n5 == 1, "up to 32 values");
  auto fold = [&](auto have, auto half, int o) {
    constexpr int n = decltype(have)::value, h = decltype(half)::value;
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const double hi = i + h < n ? d[i + h] : 0.0;
      const double send = up ? d[i] : hi, keep = up ? hi : d[i];
      d[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  };
  fold(std::integral_constant<int, V>{}, std::integral_constant<int, n1>{}, 16);
  fold(std::integral_constant<int, n1>{}, std::integral_constant<int, n2>{}, 8);
  fold(std::integral_constant<int, n2>{}, std::integral_constant<int, n3>{}, 4);
  fold(std::integral_constant<int, n3>{}, std::integral_constant<int, n4>{}, 2);
  if constexpr (n4 > 1) fold(std::integral_constant<int, n4>{}, std::integral_constant<int, n5>{}, 1);
  else d[0] += __shfl_xor_sync(0xffffffffu, d[0], 1);
#pragma unroll
  for (int i = 0; i < V; ++i) {  // value i sits in the lane its halves lead to
    int k = i, src = 0;
    if (k >= n1) k -= n1, src |= 16;
    if (k >= n2) k -= n2, src |= 8;
    if (k >= n3) k -= n3, src |= 4;
    if (k >= n4) k -= n4, src |= 2;
    if (k >= n5) k -= n5, src |= 1;
    r[i] = __shfl_sync(0xffffffffu, d[0], src);
  }
}

// ---- 1. Right-hand side, left in the region as digit fragments.
template <int N, int W, bool VISC>
__device__ __forceinline__ void pd_rhs(bool first) {
  using P = Pd<N>;
  constexpr int NP = P::NP, NT = P::NT, SQ = P::SQ, THR = 32 * W, KKS = P::KKS;
  const PdView<N> V;
  PdShared& x = pd_shared();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int S = x.S, over = max(x.slots - THR, 0);
  double* const sover = V.region + x.room / 8 - over * SQ;
  const int nte = first ? 1 : NT;
  // (the columns' tiles of eight and their exponents take part of a tile more)
  const int cap = (x.room - over * SQ * 8 - 8 * P::CB) / (5 * nte * (P::CB + 4));
  const int nch = (S + cap - 1) / cap, CH = (S + nch - 1) / nch;
  double racc[5][NT];
  int cur, cend, cstep;
  const int node0 = slot_list(V.slist, x.Ni, x.nlong, tid, cur, cend, cstep);
#pragma unroll
  for (int v = 0; v < 5; ++v)
#pragma unroll
    for (int t = 0; t < NT; ++t) racc[v][t] = 0.0;
  for (int e = tid; e < over * SQ; e += THR) sover[e] = 0.0;
  const double gm1 = x.m->gamma - 1.0;
  for (int kc = 0; kc < S; kc += CH) {
    const int nk = min(CH, S - kc);
    if constexpr (VISC) {
      pd_gradients<N, THR>(kc, nk, nte, first);
      __syncthreads();
    }
    // fluxes, items (sub-tet, node, time slice): columns (k, v, t)
    for (int e = tid; e < nk * NP * nte; e += THR) {
      const int kj = first ? e : e / NT, t = first ? 0 : e - kj * NT, kl = kj / NP, j = kj - kl * NP;
      const double* gp = V.sgeo + (kc + kl) * 10;
      double g[9], Q[5], out[3][5];
#pragma unroll
      for (int i = 0; i < 9; ++i) g[i] = gp[i];
      const int node = V.sA[(kc + kl) * NP + j];
#pragma unroll
      for (int v = 0; v < 5; ++v) Q[v] = first ? V.suh[node * 5 + v] : V.sq[node * SQ + v * NT + t];
      double* dst = V.region + (kl * 5 * nte + t) * KKS + j;
      const int vs = nte * KKS;
      if constexpr (VISC) {
        double F[3][5];
        pd_flux_visc<N>(x, Q, g, 1.0 / gp[9], dst, vs, F);
        contract_adj(g, 1.0, F, out);
      } else {
        contravariant_flux(Q, g, gm1, out);
      }
#pragma unroll
      for (int v = 0; v < 5; ++v)
#pragma unroll
        for (int d = 0; d < 3; ++d) dst[v * vs + d * NP] = out[d][v];
    }
    __syncthreads();
    pd_contract<N, W>(x.ref, false, nk * 5 * nte, KKS);
    __syncthreads();
    auto gather = [&](int& c1, int end, int step, double (&acc)[5][NT]) {
      const int lim = (kc + nk) << 6;
      int w = c1 < end ? V.sinc[c1] : lim;
      while (w < lim) {
        const double* src = V.region + ((w >> 6) - kc) * 5 * nte * KKS + (w & 63);
        c1 += step;
        w = c1 < end ? V.sinc[c1] : lim;
#pragma unroll
        for (int v = 0; v < 5; ++v)
#pragma unroll
          for (int t = 0; t < NT; ++t)
            if (t == 0 || !first) acc[v][t] += src[(v * nte + t) * KKS];
      }
    };
    gather(cur, cend, cstep, racc);
    for (int i = tid + THR; i < x.slots; i += THR) {
      int c1, e1, st1;
      slot_list(V.slist, x.Ni, x.nlong, i, c1, e1, st1);
      while (c1 < e1 && V.sinc[c1] < (kc << 6)) ++c1;
      if (c1 >= e1 || V.sinc[c1] >= (kc + nk) << 6) continue;
      double* o = sover + (i - THR) * SQ;
      double a[5][NT];
#pragma unroll
      for (int q = 0; q < SQ; ++q) a[q / NT][q % NT] = o[q];
      gather(c1, e1, 1, a);
#pragma unroll
      for (int q = 0; q < SQ; ++q) o[q] = a[q / NT][q % NT];
    }
    if (kc + CH < S) __syncthreads();
  }
  if (warp < x.nlong) lane_sums<SQ>(&racc[0][0], lane);  // the lanes' shares of a long list
  // per variable the exponent e with |r 2^-p| < 2^e over the nodes (p: the row's exponent)
  // (infinities and NaN: kPdNone, the product is NaN then)
  auto expo = [&](double r, int p) {
    const int ex = __double2hiint(r) >> 20 & 0x7ff;
    return ex == 0x7ff ? kPdNone : max(ex, 1) - 1022 - p;
  };
  const bool own0 = node0 >= 0 && (warp >= x.nlong || lane == 0);
  const int p0 = own0 ? V.sexp[node0] : 0;
  double a[5][NT];
#pragma unroll
  for (int v = 0; v < 5; ++v)
#pragma unroll
    for (int t = 0; t < NT; ++t) a[v][t] = 0.0;
  int mx[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    mx[v] = -20000;
#pragma unroll
    for (int t = 0; t < NT; ++t)
      if (own0 && (t == 0 || !first)) mx[v] = max(mx[v], expo(racc[v][t], p0));
  }
  for (int i = tid + (x.slots - 1 - tid) / THR * THR; i >= THR; i -= THR) {  // the second slot last
    const double* o = sover + (i - THR) * SQ;
    const int p = V.sexp[V.slist[1 + 2 * (i - 31 * x.nlong)]];
#pragma unroll
    for (int q = 0; q < SQ; ++q) {
      a[q / NT][q % NT] = o[q];
      if (q % NT == 0 || !first) mx[q / NT] = max(mx[q / NT], expo(o[q], p));
    }
  }
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    const int r = __reduce_max_sync(0xffffffffu, mx[v]);
    if (lane == 0) x.ired[v][warp] = r;
  }
  __syncthreads();
  int ev[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    ev[v] = x.ired[v][0];
#pragma unroll
    for (int w = 1; w < W; ++w) ev[v] = max(ev[v], x.ired[v][w]);
    if (tid == 0) x.ev[v] = ev[v];
  }
  // digit fragments: value (row n, column col) at step n / 16, column tile col / 8, lane (col & 7) 4 +
  // ((n & 7) >> 1): 32 bytes, digit s (0: the highest) in word s at byte 2 (n >> 3 & 1) + (n & 1)
  unsigned char* const frag = reinterpret_cast<unsigned char*>(V.region);
  const int fb = first ? P::FB1 : P::FB;
  auto at = [&](int n, int col) {
    return frag + (n >> 4) * fb + (col >> 3) * 1024 + ((col & 7) * 4 + ((n & 7) >> 1)) * 32 + ((n >> 3) & 1) * 2 + (n & 1);
  };
  auto put = [&](int n, const double (&r)[5][NT]) {
    const int p = V.sexp[n];
#pragma unroll
    for (int v = 0; v < 5; ++v)
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        if (first && t > 0) continue;
        const unsigned long long d = digits(r[v][t], ev[v] + p);
        unsigned char* o = at(n, first ? v : v * P::NTP + t);
#pragma unroll
        for (int s = 0; s < 8; ++s) o[4 * s] = (unsigned char)(d >> (56 - 8 * s));
      }
  };
  int n = own0 ? node0 : -1;
#pragma unroll 1
  for (int i = tid;;) {  // first, second, later slots
    if (n >= 0) put(n, racc);
    i += THR;
    if (i >= x.slots) break;
    n = V.slist[1 + 2 * (i - 31 * x.nlong)];
#pragma unroll
    for (int q = 0; q < SQ; ++q) racc[q / NT][q % NT] = i >= 2 * THR ? sover[(i - THR) * SQ + q] : a[q / NT][q % NT];
  }
  // rows past N_i and padded time slices: the digit zero
  const int nc = first ? 5 : 5 * P::NTP;
  for (int e = tid; e < (16 * x.nks - x.Ni) * nc; e += THR) {
    unsigned char* o = at(x.Ni + e / nc, e % nc);
#pragma unroll
    for (int s = 0; s < 8; ++s) o[4 * s] = 128;
  }
  if (NT < P::NTP && !first)
    for (int e = tid; e < 5 * x.Ni; e += THR) {
      unsigned char* o = at(e / 5, e % 5 * P::NTP + NT);
#pragma unroll
      for (int s = 0; s < 8; ++s) o[4 * s] = 128;
    }
}

// ---- 2. Y = M_i^-1 RHS and q^{r+1}; (16-row tile, 8-column tile) pairs over the warps.  Returns this
// thread's max |q^{r+1} - q^r| and max |q^r|.
template <int N, int W, bool FIRST>
__device__ __forceinline__ longlong2 pd_apply() {
  using P = Pd<N>;
  constexpr int NT = P::NT, NTP = P::NTP, SQ = P::SQ, fb = FIRST ? P::FB1 : P::FB;
  constexpr int NT1 = FIRST ? 1 : P::NNT, QL = FIRST ? 20 : 20 * NTP;
  const PdView<N> V;
  const PdShared& x = pd_shared();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, gq = lane >> 2, tq = lane & 3;
  const int Ni = x.Ni, nks = x.nks;
  long long res = 0, qmax = 0;
  auto update = [&](int n, int v, const double (&y)[NT]) {
    const double uh = V.suh[n * 5 + v];
    double* qp = V.sq + n * SQ + v * NT;
#pragma unroll
    for (int s = 0; s < NT; ++s) {
      double z = uh;
      if constexpr (FIRST) {
        z -= x.dkws[s] * y[0];
      } else {
#pragma unroll
        for (int t = 0; t < NT; ++t) z -= x.dkw[s][t] * y[t];
      }
      const double old = FIRST ? uh : qp[s];
      // maxima of magnitudes as integers: non-negative doubles order as their bits
      // (NaN passed over, as fmax does)
      const long long dz = __double_as_longlong(z - old) & 0x7fffffffffffffffll;
      const long long ob = __double_as_longlong(old) & 0x7fffffffffffffffll;
      if (dz <= 0x7ff0000000000000ll) res = max(res, dz);
      if (ob <= 0x7ff0000000000000ll) qmax = max(qmax, ob);
      qp[s] = z;
    }
  };
  for (int job = warp; job < nks * NT1; job += W) {
    const int mt = job / NT1, nt = job - mt * NT1;
    long long hi[4], lo[4];
    digit_product(x.dig + (size_t)mt * nks * 512 + lane * 4,
                  reinterpret_cast<const unsigned char*>(V.region) + nt * 1024 + lane * 32, fb, nt * 32 + lane < QL, nks, hi,
                  lo);
    // digit s of one factor weighs 2^(56 - 8 s): level l 2^(112 - 8 l); the factors are scaled by 2^62
    // (over the row's, column's and right-hand side's powers)
    auto value = [&](int i, int n, int v) {
      return digit_value(hi[i], lo[i], 56 - 124 + x.ev[v] - V.sexp[n], x.ev[v] >= kPdNone);
    };
    if constexpr (FIRST) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int v = 2 * tq + (i & 1), n = mt * 16 + gq + (i >> 1) * 8;
        if (v < 5 && n < Ni) {
          const double y[NT] = {value(i, n, v)};
          update(n, v, y);
        }
      }
    } else if constexpr (NTP == 2) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int v = nt * 4 + tq, n = mt * 16 + gq + 8 * h;
        if (v < 5 && n < Ni) {
          const double y[2] = {value(2 * h, n, v), value(2 * h + 1, n, v)};
          update(n, v, y);
        }
      }
    } else {
      // a lane pair holds the time slices of rows g and g + 8: the even lane takes row g
      const bool odd = tq & 1;
      const int v = nt * 2 + (tq >> 1), n = mt * 16 + gq + (odd ? 8 : 0);
      long long h0 = odd ? hi[0] : hi[2], h1 = odd ? hi[1] : hi[3], l0 = odd ? lo[0] : lo[2], l1 = odd ? lo[1] : lo[3];
      h0 = __shfl_xor_sync(0xffffffffu, h0, 1);
      h1 = __shfl_xor_sync(0xffffffffu, h1, 1);
      l0 = __shfl_xor_sync(0xffffffffu, l0, 1);
      l1 = __shfl_xor_sync(0xffffffffu, l1, 1);
      if (odd) {
        hi[0] = h0, hi[1] = h1, lo[0] = l0, lo[1] = l1;
      } else {
        hi[2] = h0, hi[3] = h1, lo[2] = l0, lo[3] = l1;
      }
      if (v < 5 && n < Ni) {
        double y[NT];
#pragma unroll
        for (int t = 0; t < NT; ++t) y[t] = value(t, n, v);
        update(n, v, y);
      }
    }
  }
  return make_longlong2(res, qmax);
}

// ---- Epilogue: volume term, q_bar and F_bar . n on the face slots, as pc_epilogue.
template <int N, int W, bool VISC>
__device__ __forceinline__ void pd_epilogue() {
  using P = Pd<N>;
  constexpr int NP = P::NP, NT = P::NT, NF = P::NF, SQ = P::SQ, THR = 32 * W, KKS = P::KKS;
  constexpr int cv = VISC ? NT * KKS : KKS;  // per (k, v): viscous cells hold the gradients of every time slice
  const PdView<N> V;
  const PdShared& x = pd_shared();
  const PdRef& ref = x.ref;
  const DevMesh& m = *x.m;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, S = x.S, ns = x.ns;
  const uint16_t* const sfinfo = reinterpret_cast<const uint16_t*>(
      reinterpret_cast<const float*>(V.sinc + gat_up(2 * (size_t)S * NP) / 2) + ns);
  const uint8_t* const sfloc = reinterpret_cast<const uint8_t*>(sfinfo + ns);
  double vacc[kPcOver + 1][5];
  int cur[kPcOver + 1], cend[kPcOver + 1], cstep[kPcOver + 1], node[kPcOver + 1];
#pragma unroll
  for (int r = 0; r <= kPcOver; ++r) {
#pragma unroll
    for (int v = 0; v < 5; ++v) vacc[r][v] = 0.0;
    node[r] = slot_list(V.slist, x.Ni, x.nlong, tid + r * THR, cur[r], cend[r], cstep[r]);
  }
  const int cap = (x.room - 8 * P::CB) / (5 * (cv * 8 + P::CB - KKS * 8 + 4)), nch = (S + cap - 1) / cap, CH = (S + nch - 1) / nch;
  const double gm1 = m.gamma - 1.0, dt = x.dt;
  for (int kc = 0; kc < S; kc += CH) {
    const int nk = min(CH, S - kc);
    if (kc) __syncthreads();
    if constexpr (VISC) {
      pd_gradients<N, THR>(kc, nk, NT, false);
      __syncthreads();
    }
    for (int e = tid; e < nk * NP; e += THR) {
      const int kl = e / NP, j = e - kl * NP;
      const double* gp = V.sgeo + (kc + kl) * 10;
      const double* qn = V.sq + V.sA[(kc + kl) * NP + j] * SQ;
      double* dst = V.region + kl * 5 * cv + j;
      double fb[3][5];
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int v = 0; v < 5; ++v) fb[d][v] = 0.0;
      double g[9];
      if constexpr (VISC) {
#pragma unroll
        for (int i = 0; i < 9; ++i) g[i] = gp[i];
      }
#pragma unroll 1
      for (int t = 0; t < NT; ++t) {
        const double Q[5] = {qn[t], qn[NT + t], qn[2 * NT + t], qn[3 * NT + t], qn[4 * NT + t]};
        const double wt = ref.w[t];
        if constexpr (VISC) {
          double F[3][5];
          pd_flux_visc<N>(x, Q, g, 1.0 / gp[9], dst + t * KKS, cv, F);
#pragma unroll
          for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int v = 0; v < 5; ++v) fb[d][v] += wt * F[d][v];
        } else {
          const double ir = recip(Q[0]);
          const double vel[3] = {Q[1] * ir, Q[2] * ir, Q[3] * ir};
          const double p = gm1 * (Q[4] - 0.5 * (Q[1] * vel[0] + Q[2] * vel[1] + Q[3] * vel[2]));
          const double H = wt * (Q[4] + p), wp = wt * p;
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const double wm = wt * Q[1 + d];
            fb[d][0] += wm;
#pragma unroll
            for (int a = 0; a <= d; ++a) fb[d][1 + a] += wm * vel[a];
            fb[d][1 + d] += wp;
            fb[d][4] += H * vel[d];
          }
        }
      }
      if constexpr (!VISC) {  // m_a v_b is symmetric
        fb[0][2] = fb[1][1];
        fb[0][3] = fb[2][1];
        fb[1][3] = fb[2][2];
#pragma unroll
        for (int i = 0; i < 9; ++i) g[i] = gp[i];
      }
      double out[3][5];
      contract_adj(g, dt, fb, out);
#pragma unroll
      for (int v = 0; v < 5; ++v)
#pragma unroll
        for (int d = 0; d < 3; ++d) dst[v * cv + d * NP] = out[d][v];
    }
    __syncthreads();
    double* const sqo = (double*)m.slot_q;
    double* const sfn = (double*)m.slot_fn;
    for (int e = tid; e < ns * NF; e += THR) {
      const int sl = e / NF, info = sfinfo[sl], kl = (info >> 2) - kc, o = info & 3;
      if (kl < 0 || kl >= nk) continue;
      const int j = sfloc[e];
      const double* qn = V.sq + V.sA[(kc + kl) * NP + j] * SQ;
      const double s = 0.5 / m.slot_geo[(x.s0 + sl) * 4 + 3];
      const double* bp = V.region + kl * 5 * cv + j;
      const int64_t at = (x.s0 * NF + e) * 5;
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        double qb = 0.0;
#pragma unroll
        for (int t = 0; t < NT; ++t) qb += ref.w[t] * qn[v * NT + t];
        const double f = o == 0 ? (bp[v * cv] + bp[v * cv + NP]) + bp[v * cv + 2 * NP] : -bp[v * cv + (o - 1) * NP];
        sqo[at + v] = dt * qb;
        sfn[at + v] = s * f;
      }
    }
    __syncthreads();
    pd_contract<N, W>(ref, true, nk * 5, cv);
    __syncthreads();
#pragma unroll
    for (int r = 0; r <= kPcOver; ++r) {
      const int lim = (kc + nk) << 6;
      int w = cur[r] < cend[r] ? V.sinc[cur[r]] : lim;
      while (w < lim) {
        const double* src = V.region + ((w >> 6) - kc) * 5 * cv + (w & 63);
        cur[r] += cstep[r];
        w = cur[r] < cend[r] ? V.sinc[cur[r]] : lim;
#pragma unroll
        for (int v = 0; v < 5; ++v) vacc[r][v] += src[v * cv];
      }
    }
  }
  if (warp < x.nlong) {
    lane_sums<5>(vacc[0], lane);
    if (lane) node[0] = -1;
  }
  double* const vol = (double*)m.vol;
#pragma unroll
  for (int r = 0; r <= kPcOver; ++r)
    if (node[r] >= 0)
#pragma unroll
      for (int v = 0; v < 5; ++v) vol[(x.n0 + node[r]) * 5 + v] = vacc[r][v];
}

template <int N, int W, int MB, bool VISC>
__global__ void __launch_bounds__(32 * W, MB) predictor_f64_kernel(const __grid_constant__ Batch bt,
                                                                   const __grid_constant__ PdRef ref, int diag,
                                                                   int smem_bytes, int mixed) {
  using P = Pd<N>;
  constexpr int NP = P::NP, NT = P::NT, NF = P::NF, SQ = P::SQ, THR = 32 * W;
  PdShared& x = pd_shared();
  __shared__ int sCell;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) x.ref = ref;
  int* const queue = bt.work + (VISC ? 1 : 0);
  const DevMesh& m = bt.tab[0];
  auto take = [&]() {  // next cell of this kernel's kind
    for (;;) {
      const int w = atomicAdd(queue, 1);
      if (w >= bt.cpre[1]) return w;
      const int g = bt.order != nullptr ? bt.order[w] : w;
      if (mixed) {
        const double mu = m.mu[g];
        if ((mu != 0.0 || cell_kappa(m, mu) != 0.0) != VISC) continue;
      }
      return g;
    }
  };
  int next = 0;
  if (tid == 0) next = take();
  for (;;) {
    if (tid == 0) sCell = next;
    __syncthreads();
    const int64_t c = sCell;
    if (c >= bt.cpre[1]) break;
    if (tid == 0) next = take();
    const int64_t n0 = m.node_ptr[c], k0 = m.sub_ptr[c], s0 = m.slot_ptr[c];
    const int Ni = (int)(m.node_ptr[c + 1] - n0), S = (int)(m.sub_ptr[c + 1] - k0), ns = (int)(m.slot_ptr[c + 1] - s0);
    const uint32_t gbytes = (uint32_t)gat_bytes(Ni, S, ns, NP, NF);
    const uint32_t o_geo = kPdGat + (uint32_t)pc_up(gbytes), o_A = o_geo + (uint32_t)pc_up((size_t)S * 80),
                   o_exp = o_A + (uint32_t)pc_up((size_t)S * NP * 2), o_uh = o_exp + (uint32_t)pc_up((size_t)Ni * 2),
                   o_q = o_uh + (uint32_t)pc_up((size_t)Ni * 40), o_region = o_q + (uint32_t)pc_up((size_t)Ni * SQ * 8);
    const int nks = (Ni + 15) / 16;
    const uint32_t* const dig = m16_block(m, c);
    {
      const uint4* src = reinterpret_cast<const uint4*>(m.gat + gat_start(n0, k0, s0, c, NP, NF));
      uint4* dst = reinterpret_cast<uint4*>(pc_smem + kPdGat);
      for (int e = tid; e < (int)(gbytes / 16); e += THR) dst[e] = src[e];
      const int16_t* ex = reinterpret_cast<const int16_t*>(dig + (size_t)nks * nks * 512);
      int16_t* se = reinterpret_cast<int16_t*>(pc_smem + o_exp);
      for (int e = tid; e < Ni; e += THR) se[e] = ex[e];
      double* sg = reinterpret_cast<double*>(pc_smem + o_geo);
      for (int e = tid; e < S * 10; e += THR) sg[e] = m.geo[k0 * 10 + e];
      uint16_t* sa = reinterpret_cast<uint16_t*>(pc_smem + o_A);
      for (int e = tid; e < S * NP; e += THR) sa[e] = m.A[k0 * NP + e];
      double* su = reinterpret_cast<double*>(pc_smem + o_uh);
      for (int e = tid; e < 5 * Ni; e += THR) su[e] = m.u[n0 * 5 + e];
    }
    if (tid == 0) {
      x.m = &m;
      x.dig = dig;
      x.c = c;
      x.n0 = n0;
      x.s0 = s0;
      x.k0 = k0;
      x.Ni = Ni;
      x.S = S;
      x.ns = ns;
      x.nks = nks;
      x.room = smem_bytes - (int)o_region;
      x.o_inc = kPdGat + (uint32_t)gat_up(2 * (size_t)(2 * Ni + 3));
      x.o_geo = o_geo;
      x.o_A = o_A;
      x.o_exp = o_exp;
      x.o_uh = o_uh;
      x.o_q = o_q;
      x.o_region = o_region;
      x.dt = *m.dt;
      for (int s = 0; s < NT; ++s) {
        x.dkws[s] = x.dt * ref.kws[s];
        for (int t = 0; t < NT; ++t) x.dkw[s][t] = x.dt * ref.kw[s][t];
      }
      x.mu = m.mu[c];
      x.kap = cell_kappa(m, x.mu);
      x.nlong = min((int)*reinterpret_cast<const uint16_t*>(m.gat + gat_start(n0, k0, s0, c, NP, NF)), W);
      x.slots = Ni + 31 * x.nlong;
    }
    __syncthreads();
    int it = 0;
    bool conv = false;
    while (!conv && it < m.picard_max) {
      ++it;
      pd_rhs<N, W, VISC>(it == 1);
      __syncthreads();
      longlong2 rq = it == 1 ? pd_apply<N, W, true>() : pd_apply<N, W, false>();
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        rq.x = max(rq.x, __shfl_xor_sync(0xffffffffu, rq.x, o));
        rq.y = max(rq.y, __shfl_xor_sync(0xffffffffu, rq.y, o));
      }
      if (lane == 0) {
        x.red[0][warp] = rq.x;
        x.red[1][warp] = rq.y;
      }
      __syncthreads();
#pragma unroll
      for (int w = 0; w < W; ++w) {
        rq.x = max(rq.x, x.red[0][w]);
        rq.y = max(rq.y, x.red[1][w]);
      }
      conv = __longlong_as_double(rq.x) <= m.tol * fmax(1.0, __longlong_as_double(rq.y));
    }
    if (tid == 0) {
      m.iters[c] = it;
      if (!conv) atomicAdd(&m.flags[F_NONCONV], 1);
    }
    pd_epilogue<N, W, VISC>();
    if (diag && m.qbar_diag) {
      const double* sq = reinterpret_cast<const double*>(pc_smem + o_q);
      for (int e = tid; e < Ni * 5; e += THR) {
        double acc = 0.0;
#pragma unroll
        for (int t = 0; t < NT; ++t) acc += x.ref.w[t] * sq[e * NT + t];
        m.qbar_diag[n0 * 5 + e] = x.dt * acc;
      }
    }
    __syncthreads();
  }
}

// ----------------------------------------------------------------------------------------
// FP64 corrector on the digits of M_i^-1 (Sec. 4.4), one block per cell: r as corrector_kernel forms it, du = M_i^-1 r
// by the digit products of the predictor's first iteration (5 columns), u += du.  With the FP64 rows read
// here a handle would hold M_i^-1 twice.  us per launch, corrector_kernel on the rows and here: 8^3 P3 816 and 220,
// 10^3 P2 254 and 112, 6^3 P1 18 and 18.
template <int N>
__host__ __device__ constexpr size_t pd_corr_smem(int n) {
  return (size_t)(n + 15) / 16 * Pd<N>::FB1 + (size_t)n * 40;
}
template <int N, int W, int MB>
__global__ void __launch_bounds__(32 * W, MB) corrector_f64_kernel(const __grid_constant__ Batch bt,
                                                                   const RefData* __restrict__ ref) {
  using P = Pd<N>;
  constexpr int NF = P::NF, THR = 32 * W;
  const DevMesh& m = bt.tab[0];
  const int64_t c = blockIdx.x, n0 = m.node_ptr[c], s0 = m.slot_ptr[c];
  const int Ni = (int)(m.node_ptr[c + 1] - n0), nks = (Ni + 15) / 16;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __shared__ double sZ[NF][NF];
  __shared__ int ired[5][W];
  unsigned char* const frag = pc_smem;                                        // digits of r (rows scaled)
  double* const r = reinterpret_cast<double*>(pc_smem + (size_t)nks * P::FB1);  // [N_i][5] r, then du
  const uint32_t* const dig = m16_block(m, c);
  const int16_t* const sexp = reinterpret_cast<const int16_t*>(dig + (size_t)nks * nks * 512);
  const double* const vol = (const double*)m.vol;
  const double* const sG = (const double*)m.slot_G;
  for (int e = tid; e < NF * NF; e += THR) sZ[e / NF][e % NF] = ref->Z[e / NF][e % NF];
  __syncthreads();
  // a thread's items are of one variable (its stride is a multiple of 5)
  constexpr int FS = THR / 5 * 5;
  int mx = -20000;
  for (int e = tid; e < Ni * 5 && tid < FS; e += FS) {
    const int n = e / 5, v = e - n * 5;
    double acc = vol[(n0 + n) * 5 + v];
    for (int64_t p = m.finc_ptr[n0 + n]; p < m.finc_ptr[n0 + n + 1]; ++p) {
      const uint32_t w = m.finc[p];
      const int64_t s = s0 + (w >> 4);
      const double* z = sZ[w & 15];
      double f = 0;
#pragma unroll
      for (int b = 0; b < NF; ++b) f += z[b] * sG[(s * NF + b) * 5 + v];
      acc -= 2.0 * m.slot_geo[s * 4 + 3] * f;
    }
    r[e] = acc;
    const int ex = __double2hiint(acc) >> 20 & 0x7ff;
    mx = max(mx, ex == 0x7ff ? kPdNone : max(ex, 1) - 1022 - sexp[n]);
  }
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    const int x = __reduce_max_sync(0xffffffffu, tid % 5 == v ? mx : -20000);
    if (lane == 0) ired[v][warp] = x;
  }
  __syncthreads();
  int ev[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    ev[v] = ired[v][0];
#pragma unroll
    for (int w = 1; w < W; ++w) ev[v] = max(ev[v], ired[v][w]);
  }
  // fragments as pd_rhs writes them; rows past N_i: the digit zero
  for (int n = tid; n < 16 * nks; n += THR) {
    unsigned char* const row = frag + (n >> 4) * P::FB1 + ((n & 7) >> 1) * 32 + ((n >> 3) & 1) * 2 + (n & 1);
    const int p = n < Ni ? sexp[n] : 0;
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      const unsigned long long d = n < Ni ? digits(r[n * 5 + v], ev[v] + p) : 0x8080808080808080ull;
#pragma unroll
      for (int s = 0; s < 8; ++s) row[v * 128 + 4 * s] = (unsigned char)(d >> (56 - 8 * s));
    }
  }
  __syncthreads();
  for (int mt = warp; mt < nks; mt += W) {
    long long hi[4], lo[4];
    digit_product(dig + (size_t)mt * nks * 512 + lane * 4, frag + lane * 32, P::FB1, lane < 20, nks, hi, lo);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int v = 2 * (lane & 3) + (i & 1), n = mt * 16 + (lane >> 2) + (i >> 1) * 8;
      if (v < 5 && n < Ni) {
        int e = ev[0];
#pragma unroll
        for (int q = 1; q < 5; ++q)
          if (v == q) e = ev[q];
        r[n * 5 + v] = digit_value(hi[i], lo[i], 56 - 124 + e - sexp[n], e >= kPdNone);
      }
    }
  }
  __syncthreads();
  for (int n = tid; n < Ni; n += THR) {
    bool bad = false;
    double* un = m.u + (n0 + n) * 5;
    double x[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      x[v] = un[v] + r[n * 5 + v];
      un[v] = x[v];
      bad |= !isfinite(x[v]);
    }
    const double p = (m.gamma - 1.0) * (x[4] - 0.5 * (x[1] * x[1] + x[2] * x[2] + x[3] * x[3]) / x[0]);
    if (bad || !(x[0] > 0.0) || !(p > 0.0)) atomicOr(&m.flags[F_NONFINITE], 8);
  }
}

}  // namespace afe
