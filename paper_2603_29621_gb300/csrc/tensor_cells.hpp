// Vector Laplacian, Taylor--Hood Stokes and pressure mass in 3D: every cell is an
// axis-aligned cube, so its matrix is a sum of tensor products of 1D mass, stiffness and mixed
// matrices (tensor_cells.cu).
#pragma once
#include <cuda_runtime.h>

#include "gather.hpp"
#include "op_launch.hpp"

namespace mfns {

bool tensor_cells(const OpLaunch& L);

// contributions of A src to g.buf (slot-major, cells in the forest's order); g.cell_* must be laid out
void tensor_product(const OpLaunch& L, const NodeGather& g, int prec, const void* src, cudaStream_t s);

}  // namespace mfns
