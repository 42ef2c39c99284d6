// Node pass of deferred products: a cell launch writes every cell's contributions, and one thread per
// node adds those of its cells in the fixed order of the table and applies what follows.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "common.hpp"
#include "ns_lines.hpp"

namespace mfns {

// Contributions of a level's nodes: entry e of node g (ptr[g] <= e < ptr[g + 1]) is slot idx[e] =
// (cell position) * slots + slot, ascending, so a node's cells are added in colour order.
struct NodeGather {
  DevBuf ptr, idx;      // main nodes
  DevBuf ptr_p, idx_p;  // Taylor--Hood pressure nodes
  DevBuf mask;          // per node (main, then pressure): bit f set where entry f is an identity row
  int64_t n_main = 0, n_p = 0, slots = 0, slots_p = 0;  // nodes; contributions of all cells
  int nu = 1;
  DevBuf buf[2];        // the contributions per precision: main, then pressure
  size_t bytes() const { return ptr.bytes() + idx.bytes() + ptr_p.bytes() + idx_p.bytes() + mask.bytes() + buf[0].bytes() + buf[1].bytes(); }
  int64_t main_values() const;  // values of the main part of buf
};

// after: 0, 1, 2 as NsAfterArgs; 3: dst = the sum, 0 on identity rows (a restriction)
void gather_nodes(const NodeGather& g, int prec, const NsAfterArgs& a, cudaStream_t s);

}  // namespace mfns
