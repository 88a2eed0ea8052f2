// du = M_i^-1 r by the FP32 corrector's kernel for given inverses and right-hand sides: cells without
// faces, whose volume term is r, from a zero state (tests/test_corrector_product_gpu.py).
#include <cstdint>
#include <vector>

#include "predictor_cells.hpp"
#include "topology.hpp"

namespace {
template <typename T>
T* device(const std::vector<T>& v, std::vector<void*>* keep) {
  void* p = nullptr;
  if (cudaMalloc(&p, v.size() * sizeof(T) + 16) != cudaSuccess) return nullptr;
  keep->push_back(p);
  if (!v.empty()) cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice);
  return (T*)p;
}
}  // namespace

// minv: the cells' rows, minv_ld(n) apart, cell c at minv_ptr[c].  0 on success.
extern "C" int corrector_product(int N, int64_t C, const int64_t* node_ptr, const int64_t* minv_ptr, const double* minv,
                                 const float* r, double* du) {
  const int64_t nodes = node_ptr[C];
  std::vector<int64_t> np(node_ptr, node_ptr + C + 1), none(C + 1, 0), lists(nodes + 1, 0);
  int nmax = 0;
  for (int64_t c = 0; c < C; ++c) nmax = np[c + 1] - np[c] > nmax ? (int)(np[c + 1] - np[c]) : nmax;
  const int Np = (N + 1) * (N + 2) * (N + 3) / 6, Nf = (N + 1) * (N + 2) / 2;
  std::vector<void*> keep;
  afe::Batch b{};
  afe::DevMesh& m = b.tab[0];
  m.N = N;
  m.C = C;
  m.n_nodes = nodes;
  m.gamma = 1.4;
  m.node_ptr = device(np, &keep);
  m.sub_ptr = m.slot_ptr = device(none, &keep);
  m.inc_ptr = m.finc_ptr = device(lists, &keep);
  m.minv_ptr = device(std::vector<int64_t>(minv_ptr, minv_ptr + C + 1), &keep);
  m.minv64 = device(std::vector<double>(minv, minv + minv_ptr[C]), &keep);
  m.vol = device(std::vector<float>(r, r + nodes * 5), &keep);
  m.u = device(std::vector<double>(nodes * 5, 0.0), &keep);
  m.wvec = device(std::vector<double>(nodes, 0.0), &keep);  // no correction of the cell's total
  m.cell_vol = device(std::vector<double>(C, 1.0), &keep);
  m.flags = device(std::vector<int>(64, 0), &keep);
  const afe::BlockLayout L = afe::block_layout(np, afe::minv_split_words, 0, afe::pc_gather_bytes(m, 0, Np, Nf));
  unsigned char* p = device(std::vector<unsigned char>(L.bytes, 0), &keep);
  int rc = 1;
  if (p && m.flags && m.u) {
    cudaMemcpy(p, L.ptr.data(), L.ptr.size() * 8, cudaMemcpyHostToDevice);
    m.m16 = (uint32_t*)p;
    m.gat = p + L.gather;
    b.nh = 1;
    b.Nmax = nmax;
    b.cpre[1] = C;
    afe::pc_set_up(m, Np, Nf, (int)C, nullptr);
    afe::CorrRef ref{};
    if (N == 1) afe::pc_correct<1>(b, ref, nmax, 0, nullptr);
    else if (N == 2) afe::pc_correct<2>(b, ref, nmax, 0, nullptr);
    else afe::pc_correct<3>(b, ref, nmax, 0, nullptr);
    if (cudaDeviceSynchronize() == cudaSuccess && cudaGetLastError() == cudaSuccess)
      rc = cudaMemcpy(du, m.u, nodes * 5 * sizeof(double), cudaMemcpyDeviceToHost) == cudaSuccess ? 0 : 1;
  }
  for (void* q : keep) cudaFree(q);
  return rc;
}
