// Host tables of deferred products (see NodeGather in gather.hpp).
#pragma once
#include <cstddef>
#include <cstdint>
#include <vector>

namespace mfns {

// The node of every place of the contribution buffer.  cell_nodes: nb nodes per cell of the forest's order;
// perm: the forest's cell at every position of the colour order.  Place of slot b of a cell: position *
// nb + b, or with by_slot b * cells + cell.
inline std::vector<int32_t> nodes_by_place(const std::vector<int32_t>& cell_nodes, int nb,
                                           const std::vector<int32_t>& perm, bool by_slot) {
  const size_t nc = perm.size();
  std::vector<int32_t> v(nc * nb);
  for (size_t i = 0; i < nc; ++i)
    for (int b = 0; b < nb; ++b) {
      if (by_slot) v[b * nc + i] = cell_nodes[i * nb + b];
      else v[i * nb + b] = cell_nodes[(size_t)perm[i] * nb + b];
    }
  return v;
}

// The places of every node, ascending: idx[ptr[g]] to idx[ptr[g + 1] - 1] for node g of n.
inline void gather_table(const std::vector<int32_t>& node_of_place, int64_t n, std::vector<int32_t>& ptr,
                         std::vector<int32_t>& idx) {
  ptr.assign((size_t)n + 1, 0);
  for (int32_t g : node_of_place) ++ptr[(size_t)g + 1];
  for (int64_t g = 0; g < n; ++g) ptr[g + 1] += ptr[g];
  idx.resize(node_of_place.size());
  std::vector<int32_t> at(ptr.begin(), ptr.end() - 1);
  for (size_t e = 0; e < node_of_place.size(); ++e) idx[at[node_of_place[e]]++] = (int32_t)e;
}

}  // namespace mfns
