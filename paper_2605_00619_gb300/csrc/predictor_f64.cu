// Kernels, plans and launches of predictor_f64.cuh for one order (AFE_ORDER), and, with the first, the
// set-up of the digits of M_i^-1.
#include "predictor_f64.cuh"

#include <algorithm>
#include <cmath>

namespace afe {
namespace {

// Warps per block and blocks per SM at most: FP64 instructions set the time, so a few warps per
// scheduler suffice; at P1 and P2 several cells per SM fill each other's barriers.
template <int N>
struct PdShape {
  static constexpr int W = N == 3 ? 16 : 8, MB = N == 3 ? 1 : 2;
};
template <int N, bool VISC>
constexpr auto pd_kernel = predictor_f64_kernel<N, PdShape<N>::W, PdShape<N>::MB, VISC>;

// Warps per block of the corrector, and blocks per SM (register limit).
template <int N>
constexpr int pd_corr_warps = N == 3 ? 8 : 4;
template <int N>
constexpr auto pd_corr_kernel = corrector_f64_kernel<N, pd_corr_warps<N>, 16 / pd_corr_warps<N>>;

}  // namespace

template <int N>
cudaError_t pd_plan(int device, int Nmax, int Smax, int Fmax, PdPlan* out) {
  constexpr int THR = 32 * PdShape<N>::W;
  *out = PdPlan{};
  if (pc_slots(Nmax, THR) > (kPcOver + 1) * THR || Smax > kPcMaxSub) return cudaSuccess;
  cudaFuncAttributes fa, fv;
  cudaError_t e = cudaFuncGetAttributes(&fa, pd_kernel<N, false>);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fv, pd_kernel<N, true>);
  int per_sm = 0, optin = 0;
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
  if (e != cudaSuccess) return e;
  const int stat = (int)std::max(fa.sharedSizeBytes, fv.sharedSizeBytes);
  cudaFuncAttributes fc;
  e = cudaFuncGetAttributes(&fc, pd_corr_kernel<N>);
  if (e != cudaSuccess) return e;
  const size_t corr = (size_t)optin - fc.sharedSizeBytes;
  if (pd_corr_smem<N>(Nmax) > corr) return cudaSuccess;
  e = cudaFuncSetAttribute(pd_corr_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)corr);
  if (e != cudaSuccess) return e;
  for (int nb = PdShape<N>::MB; nb >= 1; --nb) {
    const int64_t share = std::min<int64_t>(per_sm / nb - 1024, optin) - stat;
    const size_t smem = share > 0 ? (size_t)share / 128 * 128 : 0;
    if (pd_need<N>(Nmax, Smax, Fmax, THR) > smem) continue;
    e = cudaFuncSetAttribute(pd_kernel<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - stat);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(pd_kernel<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - stat);
    out->blocks = nb;
    out->smem = smem;
    return e;
  }
  return cudaSuccess;
}

template <int N>
void pd_launch(const PdPlan& p, const Batch& b, const PdRef& ref, bool inviscid, bool viscous, int diag, int n_sm,
               cudaStream_t st) {
  constexpr int THR = 32 * PdShape<N>::W;
  const int grid = (int)std::min<int64_t>(b.cpre[b.nh], (int64_t)n_sm * p.blocks);
  const int smem = (int)p.smem, mixed = inviscid && viscous;
  if (inviscid) pd_kernel<N, false><<<grid, THR, smem, st>>>(b, ref, diag, smem, mixed);
  if (viscous) pd_kernel<N, true><<<grid, THR, smem, st>>>(b, ref, diag, smem, mixed);
}

template <int N>
void pd_correct(const Batch& b, const RefData* ref, int Nmax, cudaStream_t st) {
  pd_corr_kernel<N><<<(unsigned)b.cpre[1], 32 * pd_corr_warps<N>, pd_corr_smem<N>(Nmax), st>>>(b, ref);
}

template void pd_correct<AFE_ORDER>(const Batch&, const RefData*, int, cudaStream_t);
template cudaError_t pd_plan<AFE_ORDER>(int, int, int, int, PdPlan*);
template void pd_launch<AFE_ORDER>(const PdPlan&, const Batch&, const PdRef&, bool, bool, int, int, cudaStream_t);

#if AFE_ORDER == 1
// Digits of the scaled M_i^-1 in fragment order (see predictor_f64.cuh), one block per cell at a time.
// Row exponent p_i: M_ii 2^(2 p_i) in [1/4, 1) or [1/8, 1/2).
static __global__ void __launch_bounds__(256) digits_kernel(DevMesh m) {
  for (int64_t c = blockIdx.x; c < m.C; c += gridDim.x) {
    const int64_t n0 = m.node_ptr[c];
    const int n = (int)(m.node_ptr[c + 1] - n0), LD = minv_ld(n), nks = (n + 15) / 16;
    const double* A = m.minv64 + m.minv_ptr[c];
    uint32_t* out = m16_block(m, c);
    int16_t* ex = reinterpret_cast<int16_t*>(out + (size_t)nks * nks * 512);
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const int e = (__double2hiint(A[(int64_t)i * LD + i]) >> 20 & 0x7ff) - 1022;  // M_ii < 2^e
      ex[i] = (int16_t)(-((e + 1) >> 1));
    }
    __syncthreads();
    // 16-byte group (tile, q, lane): digits 2 q and 2 q + 1 of the lane's eight entries, a word of four
    // entries for columns 2 t, 2 t + 1 (rows g, g + 8) and one for columns 2 t + 8, 2 t + 9
    for (int w = threadIdx.x; w < nks * nks * 64; w += blockDim.x) {
      const int half = w & 1, lane = (w >> 1) & 31, tile = w >> 6, ti = tile / nks, tj = tile - ti * nks;
      unsigned long long d[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int row = 16 * ti + (lane >> 2) + 8 * (i >> 1), col = 16 * tj + 2 * (lane & 3) + 8 * half + (i & 1);
        d[i] = row < n && col < n ? digits(A[(int64_t)row * LD + col], -(int)ex[row] - (int)ex[col]) : 0x8080808080808080ull;
      }
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        uint32_t v = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) v |= (uint32_t)(d[i] >> (56 - 8 * s) & 255u) << (8 * i);
        out[(size_t)tile * 512 + (s >> 1) * 128 + lane * 4 + (s & 1) * 2 + half] = v;
      }
    }
    __syncthreads();
  }
}

int pd_stiffness_words(int N) { return (np_of(N) + 15) / 16 * ((3 * np_of(N) + 15) / 16) * 512; }

int pd_stiffness_digits(const RefData& r, bool transposed, uint32_t* out) {
  const int np = r.Np, kst = (3 * np + 15) / 16, mts = (np + 15) / 16;
  double smax = 0.0;
  for (int d = 0; d < 3; ++d)
    for (int m = 0; m < np; ++m)
      for (int j = 0; j < np; ++j) smax = std::max(smax, std::fabs(r.S[d][m][j]));
  int e = 0;
  (void)std::frexp(smax, &e);
  for (int mt = 0; mt < mts; ++mt)
    for (int ks = 0; ks < kst; ++ks)
      for (int lane = 0; lane < 32; ++lane)
        for (int half = 0; half < 2; ++half)
          for (int s = 0; s < 8; ++s) {
            uint32_t v = 0;
            for (int i = 0; i < 4; ++i) {
              const int row = 16 * mt + (lane >> 2) + 8 * (i >> 1), kk = 16 * ks + 2 * (lane & 3) + 8 * half + (i & 1);
              double x = 0.0;
              if (row < np && kk < 3 * np) x = transposed ? r.S[kk / np][kk % np][row] : r.S[kk / np][row][kk % np];
              if (std::fabs(x) < 1e-13 * smax) x = 0.0;  // zeros of the exact matrix
              v |= (uint32_t)(digits(x, e) >> (56 - 8 * s) & 255u) << (8 * i);
            }
            out[(size_t)(mt * kst + ks) * 512 + (s >> 1) * 128 + lane * 4 + (s & 1) * 2 + half] = v;
          }
  return e;
}

void pd_set_up(const DevMesh& m, int grid, cudaStream_t st) { digits_kernel<<<grid, 256, 0, st>>>(m); }
#endif

}  // namespace afe
