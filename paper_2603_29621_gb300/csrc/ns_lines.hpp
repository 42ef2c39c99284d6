// Stabilised operator on uniform 3D levels (ns_lines.cu): a product is a cell launch that writes rows
// of node values and a node pass that adds them and applies what follows the product.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "op_launch.hpp"

namespace mfns {

// whether L's products take this path once its point values are laid out (L.lq, L.lc)
bool ns_lines(const OpLaunch& L);
int ns_cells_per_block(int k, int prec, int64_t cells);
// bytes of the level's point values and of a product's rows (needs L.lc)
size_t ns_fq_bytes(const OpLaunch& L, int prec);
size_t ns_rows_bytes(const OpLaunch& L, int prec);

// the level's cell kernel (0, 1 or 2); they round differently, and a multi-problem launch is of one kind
int ns_kernel(const OpLaunch& L, int prec);
// blocks of a cell launch
int64_t ns_blocks(const OpLaunch& L, int prec);
// appends the descriptor of L's product to those of a multi-problem launch
void ns_descriptor(const OpLaunch& L, int prec, const void* src, void* rows, int32_t first_block,
                   std::vector<char>& out);

// cells of one problem: rows <- contributions of A src
void ns_cells(const OpLaunch& L, int prec, const void* src, void* rows, cudaStream_t s);
// cells of several problems (descriptors on the device; every block names its problem)
struct NsMulti {
  const void* probs = nullptr;
  const int32_t* block_pid = nullptr;
  int64_t blocks = 0;
  int cmax = 0;  // largest cells per block of the members
};
void ns_cells_multi(const OpLaunch& L, int prec, const NsMulti& m, cudaStream_t s);

// node pass.  after 0: dst = A src; 1: d = c1 d + c2 dinv (b - A x), x += d (dst = src = x); 2: dst = b - A src.
// Identity rows (velocity of boundary nodes) of A src are src.
struct NsAfterArgs {
  int after = 0;
  void* dst = nullptr;
  const void* src = nullptr;
  const void* b = nullptr;
  const void* dinv = nullptr;
  void* d = nullptr;
  double c1 = 0.0, c2 = 0.0;
};
void ns_nodes(const OpLaunch& L, int prec, const NsAfterArgs& a, void* rows, cudaStream_t s);

// diagonal with 1 on the identity rows; rows: the buffer of a product's rows (scratch)
void ns_diagonal(const OpLaunch& L, int prec, void* diag, void* rows, cudaStream_t s);

}  // namespace mfns
