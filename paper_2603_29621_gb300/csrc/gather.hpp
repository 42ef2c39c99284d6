// Node pass of deferred products: a cell launch writes every cell's contributions, and one thread per
// node adds those of its cells in the fixed order of the table and applies what follows.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <memory>
#include <vector>

#include "common.hpp"
#include "ns_lines.hpp"

namespace mfns {

// What lies between the two launches of a product: one buffer for all levels and both precisions of a problem,
// whose products run one at a time.  Levels without one (null) run colour by colour, and so does a
// problem that fits its context's budget only then.
struct ProductScratch {
  Budget* bud = nullptr;
  size_t need = 0;    // largest request
  size_t tables = 0;  // bytes of the levels' tables and layouts that only products through this buffer use
  explicit ProductScratch(Budget* b) : bud(b) {}
  void reserve(size_t bytes) {  // while levels are laid out (the contents are dropped)
    need = std::max(need, bytes);
    if (buf_.bytes() < need) buf_.alloc(bud, need);
  }
  void* get() const { return buf_.get(); }

 private:
  DevBuf buf_;
};
using ScratchPtr = std::shared_ptr<ProductScratch>;

// build(scratch), and build(null) if the budget or the device's memory does not hold the first by no more
// than what the scratch and its tables take
template <typename F>
void build_within_budget(Budget* bud, F build) {
  ScratchPtr scratch = std::make_shared<ProductScratch>(bud);
  try {
    return build(scratch);
  } catch (const BudgetError& e) {
    if (e.over > scratch->need + scratch->tables) throw;
  } catch (const Error& e) {
    if (e.code != kErrOom || !scratch->need) throw;
    (void)cudaGetLastError();
  }
  scratch.reset();
  build(nullptr);
}

// Contributions of a level's nodes: entries e of node g (ptr[g] <= e < ptr[g + 1]) are the places idx[e]
// in the buffer, ascending.  Place of (cell, slot): position * slots + slot with cells in colour order,
// so that a node's cells are added in that order; with tensor-product cells (`tensor`) slot * cells +
// cell in the forest's order, so that neighbouring cells lie next to each other.
struct NodeGather {
  bool tensor = false;
  int64_t cell_stride = 0, slot_stride = 0, cell_stride_p = 0, slot_stride_p = 0;
  DevBuf pos;           // position of every cell of the colour order (transfers), or null: the same
  // tensor-product cells: node per (slot, cell) with bit 31 on Dirichlet nodes, masks, edge lengths
  DevBuf cell_u, cell_p, cell_mask, cell_h[2];
  DevBuf ptr, idx;      // main nodes
  DevBuf ptr_p, idx_p;  // Taylor--Hood pressure nodes
  DevBuf mask;          // per node (main, then pressure): bit f set where entry f is an identity row
  int64_t n_main = 0, n_p = 0, slots = 0, slots_p = 0;  // nodes; contributions of all cells
  int nu = 1;
  ScratchPtr scratch;   // holds the contributions: main, then pressure
  size_t bytes() const {
    return ptr.bytes() + idx.bytes() + ptr_p.bytes() + idx_p.bytes() + mask.bytes() + pos.bytes() + cell_u.bytes() + cell_p.bytes() +
           cell_mask.bytes() + cell_h[0].bytes() + cell_h[1].bytes();
  }
  int64_t main_values() const;  // values of the main part of buf
};

// after: 0, 1, 2 as NsAfterArgs; 3: dst = the sum, 0 on identity rows (a restriction)
void gather_nodes(const NodeGather& g, int prec, const NsAfterArgs& a, cudaStream_t s);

}  // namespace mfns
