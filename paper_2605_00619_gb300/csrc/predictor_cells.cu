// Kernels, plans and launches of predictor_cells.cuh for one order (AFE_ORDER), and, with the
// first, the set-up of the data they read.
#include "predictor_cells.cuh"

#include <algorithm>

namespace afe {
namespace {

// Block shapes by order: warps per block and blocks per SM at most.  Shape 1 serves meshes with
// many cells (us per step of the predictor, 24^3 P1 / 8^3 P2 / 32^3 P3 meshes), shape 0 those whose
// cells all run at once with more warps each, where the slowest cell's latency is the time
// (4^3 P1: 41 us with 8 warps, 58 with 2).
template <int N, int SHAPE>
struct PcShape;
template <> struct PcShape<1, 0> { static constexpr int W = 8, MB = 2; };
template <> struct PcShape<1, 1> { static constexpr int W = 2, MB = 10; };
template <> struct PcShape<2, 0> { static constexpr int W = 8, MB = 2; };
template <> struct PcShape<2, 1> { static constexpr int W = 4, MB = 4; };
template <> struct PcShape<3, 0> { static constexpr int W = 16, MB = 1; };
template <> struct PcShape<3, 1> { static constexpr int W = 8, MB = 2; };

template <int N, int SHAPE, int KINDS>
constexpr auto pc_kernel = predictor_cells_kernel<N, PcShape<N, SHAPE>::W, PcShape<N, SHAPE>::MB, KINDS>;

// Warps per block of the corrector.
template <int N>
constexpr int corr_warps = N == 3 ? 8 : (N == 2 ? 4 : 1);

template <int N>
size_t corr_smem(int n, int ns) {
  return (size_t)(n + 15) / 16 * corr_frag<N> + (size_t)((n * 5 + 3) & ~3) * 4 + (size_t)ns * nf_of(N) * 20;
}

template <int N, int SHAPE>
cudaError_t plan_shape(int device, const PcCells& q, PcPlan* out) {
  const int Nmax = q.Nmax, Smax = q.Smax, Fmax = q.Fmax;
  constexpr int W = PcShape<N, SHAPE>::W, MB = PcShape<N, SHAPE>::MB, THR = 32 * W;
  *out = PcPlan{};
  if (pc_slots(Nmax, THR) > (kPcOver + 1) * THR || Smax > kPcMaxSub) return cudaSuccess;
  int per_sm = 0, optin = 0, stat = 0;
  cudaError_t e = cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
  void (*const kernels[3])(const Batch, const PcRef, int, int) = {pc_kernel<N, SHAPE, 1>, pc_kernel<N, SHAPE, 2>,
                                                                  pc_kernel<N, SHAPE, 3>};
  for (auto* k : kernels) {
    cudaFuncAttributes fa;
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k);
    if (e == cudaSuccess) stat = std::max(stat, (int)fa.sharedSizeBytes);
  }
  if (e != cudaSuccess) return e;
  for (int nb = MB; nb >= std::min(MB, 2); --nb) {
    // 1 KB of every block's share is the system's
    const int64_t share = std::min<int64_t>(per_sm / nb - 1024, optin) - stat;
    const size_t smem = share > 0 ? (size_t)share / 128 * 128 : 0;
    if (q.need[SHAPE] > smem) continue;
    // the limit is the function's, shared by every handle: the most any plan may ask for
    for (auto* k : kernels)
      if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - stat);
    auto* corr = corrector_cells_kernel<N, corr_warps<N>>;
    cudaFuncAttributes fc;
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fc, corr);
    if (e != cudaSuccess) return e;
    if (corr_smem<N>(Nmax, Fmax) > optin - fc.sharedSizeBytes) return cudaSuccess;
    e = cudaFuncSetAttribute(corr, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fc.sharedSizeBytes);
    out->Fmax = Fmax;
    out->shape = SHAPE;
    out->blocks = nb;
    out->smem = smem;
    return e;
  }
  return cudaSuccess;
}

template <int N, int SHAPE>
void launch_shape(const PcPlan& p, const Batch& b, const PcRef& ref, bool inviscid, bool viscous, int diag, int n_sm,
                  cudaStream_t st) {
  constexpr int THR = 32 * PcShape<N, SHAPE>::W;
  const int grid = (int)std::min<int64_t>(b.cpre[b.nh], (int64_t)n_sm * p.blocks), smem = (int)p.smem;
  if (inviscid && viscous) pc_kernel<N, SHAPE, 3><<<grid, THR, smem, st>>>(b, ref, diag, smem);
  else if (viscous) pc_kernel<N, SHAPE, 2><<<grid, THR, smem, st>>>(b, ref, diag, smem);
  else pc_kernel<N, SHAPE, 1><<<grid, THR, smem, st>>>(b, ref, diag, smem);
}

}  // namespace

template <int N>
void pc_add_cell(int n, int s, int ns, PcCells* q) {
  q->Nmax = std::max(q->Nmax, n);
  q->Smax = std::max(q->Smax, s);
  q->Fmax = std::max(q->Fmax, ns);
  q->need[0] = std::max(q->need[0], pc_need<N>(n, s, ns, 32 * PcShape<N, 0>::W));
  q->need[1] = std::max(q->need[1], pc_need<N>(n, s, ns, 32 * PcShape<N, 1>::W));
}

template <int N>
cudaError_t pc_plan(int device, int n_sm, int64_t cells, bool viscous, const PcCells& q, PcPlan* out) {
  // P3 meshes whose largest cell leaves no room for two blocks of shape 1 take shape 0, which gives a cell the
  // whole SM: 32^3 mesh with cells of up to 539 nodes, step 18.1 ms in the one-block form, 12.6 ms here (a mesh
  // that fits both shapes is 25 % slower in this one, so a batch with one such member still gains over
  // the one-block form, but less).  P1 and P2 meshes that do not fit shape 1 (three gather slots per
  // thread: cells of up to 130 and 322 nodes) keep the one-block form: shape 0 has not been timed on them.
  PcPlan many;
  cudaError_t e = plan_shape<N, 1>(device, q, &many);
  *out = many;
  // at P2 the viscous fluxes' registers make eight warps per cell the better shape for any number of
  // cells (21^3 Navier-Stokes: 1,345 us per launch against 1,565)
  const bool wide = cells <= (int64_t)n_sm * PcShape<N, 0>::MB || (N == 2 && viscous) ||
                    (N == 3 && !many.blocks);
  if (e != cudaSuccess || !(many.blocks || N == 3) || !wide) return e;
  PcPlan few;
  e = plan_shape<N, 0>(device, q, &few);
  if (few.blocks) *out = few;
  return e;
}

template <int N>
void pc_launch(const PcPlan& p, const Batch& b, const PcRef& ref, bool inviscid, bool viscous, int diag, int n_sm,
               cudaStream_t st) {
  if (p.shape) launch_shape<N, 1>(p, b, ref, inviscid, viscous, diag, n_sm, st);
  else launch_shape<N, 0>(p, b, ref, inviscid, viscous, diag, n_sm, st);
}

template <int N>
void pc_correct(const Batch& b, const CorrRef& ref, int Nmax, int Fmax, cudaStream_t st) {
  corrector_cells_kernel<N, corr_warps<N>>
      <<<(unsigned)b.cpre[b.nh], 32 * corr_warps<N>, corr_smem<N>(Nmax, Fmax), st>>>(b, ref);
}

template void pc_correct<AFE_ORDER>(const Batch&, const CorrRef&, int, int, cudaStream_t);
template cudaError_t pc_plan<AFE_ORDER>(int, int, int64_t, bool, const PcCells&, PcPlan*);
template void pc_add_cell<AFE_ORDER>(int, int, int, PcCells*);
template void pc_launch<AFE_ORDER>(const PcPlan&, const Batch&, const PcRef&, bool, bool, int, int, cudaStream_t);

#if AFE_ORDER == 1
// The split copy of M_i^-1 (see minv_split_words); one block per cell at a time.  Row exponent p_i:
// M_ii 2^(2 p_i) in [1/4, 1) (bounded where M_ii is far outside FP32's range); entry (i, j) is kept as
// 2^(13 + p_i + p_j) M_ij, below 2^13 in magnitude because the matrix is positive definite.  One power of two
// for the whole cell would leave the rows of its large sub-tets the bits that FP16's range has left
// below those of its smallest one.  Both parts come from the FP64 inverses.
static __global__ void __launch_bounds__(256) split_minv_kernel(DevMesh m) {
  for (int64_t c = blockIdx.x; c < m.C; c += gridDim.x) {
    const int n = (int)(m.node_ptr[c + 1] - m.node_ptr[c]), LD = minv_ld(n);
    const double* A = m.minv64 + m.minv_ptr[c];
    uint32_t* out = m16_block(m, c);
    auto expo = [&](int i) {
      const int e = (__double2hiint(A[(int64_t)i * LD + i]) >> 20 & 0x7ff) - 1022;  // M_ii < 2^e
      return max(-100, min(100, -((e + 1) >> 1)));
    };
    for (int i = threadIdx.x; i < 4 * minv_split_head(n); i += blockDim.x)
      reinterpret_cast<int8_t*>(out)[i] = (int8_t)(i < n ? expo(i) : 0);
    const int nt = (n + 15) / 16;
    // word (tile, part, lane, i): entries (row, col), (row, col + 1) with row = 16 ti + lane / 4 + 8 (i & 1),
    // col = 16 tj + 2 (lane & 3) + 8 (i >> 1)
    for (int w = threadIdx.x; w < nt * nt * 128; w += blockDim.x) {
      const int i = w & 3, lane = (w >> 2) & 31, blk = w >> 7, ti = blk / nt, tj = blk - ti * nt;
      if (tj > ti) continue;
      const int row = 16 * ti + (lane >> 2) + 8 * (i & 1), col = 16 * tj + 2 * (lane & 3) + 8 * (i >> 1);
      uint32_t hi = 0, lo = 0;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const double x = (row < n && col + q < n)
                             ? A[(int64_t)row * LD + col + q] *
                                   __hiloint2double((1023 + 13 + expo(row) + expo(col + q)) << 20, 0)
                             : 0.0;
        const __half h = __double2half(x), l = __double2half(x - (double)__half2float(h));
        hi |= (uint32_t)__half_as_ushort(h) << (16 * q);
        lo |= (uint32_t)__half_as_ushort(l) << (16 * q);
      }
      uint32_t* o = out + minv_split_head(n) + tri_tile(ti, tj) * 256 + lane * 4 + i;
      o[0] = hi;
      o[128] = lo;
    }
  }
}

// The gather blocks (see gat_bytes), one block per cell at a time.
static __global__ void __launch_bounds__(256) gather_lists_kernel(DevMesh m, int np, int nf) {
  for (int64_t c = blockIdx.x; c < m.C; c += gridDim.x) {
    const int64_t n0 = m.node_ptr[c], k0 = m.sub_ptr[c], s0 = m.slot_ptr[c];
    const int n = (int)(m.node_ptr[c + 1] - n0), S = (int)(m.sub_ptr[c + 1] - k0), ns = (int)(m.slot_ptr[c + 1] - s0);
    unsigned char* blk = m.gat + gat_start(n0, k0, s0, c, np, nf);
    uint16_t* list = reinterpret_cast<uint16_t*>(blk);
    uint16_t* inc = reinterpret_cast<uint16_t*>(blk + gat_up(2 * (size_t)(2 * n + 3)));
    float* face = reinterpret_cast<float*>(blk + gat_up(2 * (size_t)(2 * n + 3)) + gat_up(2 * (size_t)S * np));
    uint16_t* info = reinterpret_cast<uint16_t*>(face + ns);
    uint8_t* loc = reinterpret_cast<uint8_t*>(info + ns);
    // nodes by decreasing list length (equal lengths in node order): a node's place and the
    // offset of its list are sums over the nodes ahead of it
    auto len = [&](int i) { return (int)(m.inc_ptr[n0 + i + 1] - m.inc_ptr[n0 + i]); };
    int longs = 0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const int li = len(i);
      int place = 0, off = 0;
      for (int q = 0; q < n; ++q) {
        const int lq = len(q);
        if (lq > li || (lq == li && q < i)) {
          ++place;
          off += lq;
        }
      }
      list[1 + 2 * place] = (uint16_t)i;
      list[2 + 2 * place] = (uint16_t)off;
      for (int e = 0; e < li; ++e) inc[off + e] = (uint16_t)m.inc[m.inc_ptr[n0 + i] + e];
    }
    if (threadIdx.x == 0) {
      for (int i = 0; i < n; ++i) longs += len(i) > kLongList;
      list[0] = (uint16_t)min(longs, kMaxLong);
        list[2 + 2 * n] = (uint16_t)(S * np);
    }
    for (int s = threadIdx.x; s < ns; s += blockDim.x) {
      int o = 6;  // local nodes 0 .. 3 are the sub-tet's vertices: the one missing lies opposite
      for (int a = 0; a < nf; ++a) {
        const int j = m.slot_loc[(s0 + s) * nf + a];
        loc[s * nf + a] = (uint8_t)j;
        if (j < 4) o -= j;
      }
      face[s] = (float)(0.5 / m.slot_geo[(s0 + s) * 4 + 3]);
      info[s] = (uint16_t)(m.slot_sub[s0 + s] << 2 | o);
    }
  }
}

size_t pc_gather_bytes(const DevMesh& m, int64_t n_subtets, int np, int nf) {
  return gat_start(m.n_nodes, n_subtets, m.n_slots, m.C, np, nf);
}

void pc_set_up(const DevMesh& m, int np, int nf, int grid, cudaStream_t st) {
  split_minv_kernel<<<grid, 256, 0, st>>>(m);
  pc_gather_set_up(m, np, nf, grid, st);
}

void pc_gather_set_up(const DevMesh& m, int np, int nf, int grid, cudaStream_t st) {
  gather_lists_kernel<<<grid, 256, 0, st>>>(m, np, nf);
}
#endif

}  // namespace afe
