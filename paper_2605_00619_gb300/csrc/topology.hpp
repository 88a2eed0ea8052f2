// Host-side mesh topology of the AFE scheme (Sec. 4.1, 4.4): cell nodes, sub-tet gather
// maps, per-sub-tet affine geometry, cell-boundary sub-triangles ("face slots") and their
// matching across cells.  Everything here is integer bookkeeping plus FP64 geometry; the
// mass matrices are assembled and inverted on the GPU.
#pragma once

#include <cstdint>
#include <string>
#include <vector>

#include "refelem.hpp"

namespace afe {

// Leading dimension of a cell's M_i^-1 block: N_i rounded up to a multiple of 16, plus 8.
// Rows start on 16-byte boundaries (bulk copies of whole rows), every 16-row tile of the
// tensor-core apply stays inside a row, and LD = 8 (mod 16) makes the fragment loads of
// four consecutive rows hit 32 different shared-memory banks.
inline constexpr int minv_ld(int n) { return (n + 15) / 16 * 16 + 8; }

// Words (32 bits) of a cell's block of split M_i^-1 (pairs of 16-bit values): the row exponents (8 bits
// each, padded to 128), then the 16 x 16 tiles (i, j), j <= i, of the lower triangle at i (i + 1) / 2 + j,
// 128 words of hi and 128 of lo each.
inline constexpr int minv_split_head(int n) { return (n + 127) / 128 * 32; }
inline constexpr int64_t minv_split_words(int n) {
  return minv_split_head(n) + (int64_t)((n + 15) / 16) * ((n + 15) / 16 + 1) / 2 * 256;
}
// The same of a cell's digit block (the FP64 form): 16 x 16 tiles of 512 words, then the row exponents.
inline constexpr int64_t pd_words(int n) {
  return (int64_t)((n + 15) / 16) * ((n + 15) / 16) * 512 + (n + 63) / 64 * 32;
}

// What the tensor-core forms keep of a mesh, in one allocation: the word offsets of the cells' blocks from
// its start, the blocks (words(n) for a cell of n nodes), `tail` further words and gather blocks of
// `gather` bytes.  Parts start at multiples of 128 bytes, of which the blocks and the tail are whole
// multiples.  One allocation, because a device with room for a part only would keep that part for
// nothing while the handle lives.
struct BlockLayout {
  std::vector<int64_t> ptr;      // [C+1]
  size_t tail = 0, gather = 0;   // byte offsets
  size_t bytes = 0;
};
template <typename Words>
BlockLayout block_layout(const std::vector<int64_t>& node_ptr, Words words, size_t tail, size_t gather) {
  BlockLayout L;
  L.ptr.assign(node_ptr.size(), (int64_t)(node_ptr.size() + 15) / 16 * 32);
  for (size_t c = 0; c + 1 < node_ptr.size(); ++c)
    L.ptr[c + 1] = L.ptr[c] + words((int)(node_ptr[c + 1] - node_ptr[c]));
  L.tail = (size_t)L.ptr.back() * 4;
  L.gather = L.tail + tail * 4;
  L.bytes = L.gather + gather;
  return L;
}

struct Topology {
  int N = 0, Np = 0, Nt = 0, Nf = 0;
  int64_t C = 0, T = 0, n_nodes = 0, n_slots = 0, n_groups = 0;
  int Nmax = 0, Smax = 0, slots_max = 0;

  std::vector<int64_t> node_ptr;   // [C+1] global node offset of each cell
  std::vector<int64_t> sub_ptr;    // [C+1] sub-tet offset of each cell
  std::vector<int64_t> slot_ptr;   // [C+1] face-slot offset of each cell
  std::vector<int64_t> minv_ptr;   // [C+1] offset of the dense N_i x minv_ld(N_i) block of each cell

  std::vector<uint16_t> A;         // [T*Np] cell-local node of sub-tet node j
  std::vector<double> geo;         // [T*10] adj(J) row-major (adj = det(J) J^-1), det(J)
  std::vector<double> node_xyz;    // [n_nodes*3]

  // node -> (sub-tet, local node) incidences, cell-local sub-tet index, fixed order
  std::vector<int64_t> inc_ptr;    // [n_nodes+1]
  std::vector<uint32_t> inc;       // (k_local << 6) | j

  // face slots: one per cell-boundary sub-triangle, grouped by cell
  std::vector<int32_t> slot_cell;  // [n_slots]
  std::vector<uint16_t> slot_sub;  // [n_slots] cell-local sub-tet owning the triangle
  std::vector<uint8_t> slot_loc;   // [n_slots*Nf] sub-tet-local node of each face node
  std::vector<uint16_t> slot_node; // [n_slots*Nf] cell-local node of each face node
  std::vector<double> slot_geo;    // [n_slots*4] outward unit normal (3), area
  std::vector<int64_t> slot_partner; // [n_slots] matched slot of the neighbour, or -1
  std::vector<int32_t> slot_nbr;   // [n_slots] neighbour cell, or -1 on the domain boundary

  // node -> (slot, face node) incidences for the corrector's face term
  std::vector<int64_t> finc_ptr;   // [n_nodes+1]
  std::vector<uint32_t> finc;      // (slot_local << 4) | a

  // polygonal faces: slots of one cell shared with one neighbour image, listed once per pair
  std::vector<int64_t> group_ptr;  // [n_groups+1]
  std::vector<int64_t> group_slot; // own-side slots

  std::vector<double> cell_vol;    // |P_i|
  std::vector<double> cell_h;      // 6 |P_i| / |dP_i|
  std::vector<double> cell_hsub;   // min over the cell's sub-tets of 6 |T_k| / |dT_k|
  std::vector<double> cell_diam;   // largest distance between two vertices of the cell
  double h_min = 0;
};

// Builds the topology; returns 0 on success, 2 (AFE_EMESH) or 1 (AFE_EINVAL) with a message.
int build_topology(const RefData& ref, int64_t n_vertices, const double* xyz, int64_t n_cells,
                   const int64_t* cell_subtet_ptr, const int64_t* subtet_vtx,
                   const int8_t* subtet_shift, const double period[3], bool periodic,
                   Topology* out, std::string* err);

}  // namespace afe
