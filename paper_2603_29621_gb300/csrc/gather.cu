// Node pass of deferred products (see gather.hpp).
#include "common.hpp"
#include "gather.hpp"
#include "op_kernel.cuh"
#include "smoother.cuh"

namespace mfns {

int64_t NodeGather::main_values() const { return slots * defer_stride(nu); }

// a + b rounded as the L2's FP32 reduction rounds it (subnormal inputs and result flushed to
// zero), so that a gathered sum equals the colour-ordered reductions bit for bit; the FP64
// reduction does not flush
__device__ __forceinline__ float add_as_reduction(float a, float b) {
  float r;
  asm("add.rn.ftz.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ double add_as_reduction(double a, double b) { return a + b; }

template <typename T>
struct GatherArgs {
  T* dst;
  const T *src, *b, *dinv;
  T* d;
  const T *buf, *buf_p;
  const int32_t *ptr, *idx, *ptr_p, *idx_p;
  const uint8_t* mask;
  uint32_t n_main, n_p;
  T c1, c2;
};

template <typename T, int NU>
__device__ __forceinline__ void load_slot(const T* buf, int64_t e, T (&v)[NU]) {
  const T* p = buf + e * defer_stride(NU);
  if constexpr (NU >= 3 && sizeof(T) == 4) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z;
    if (NU == 4) v[NU - 1] = q.w;
  } else if constexpr (NU >= 3) {
    const double2 q0 = *reinterpret_cast<const double2*>(p), q1 = *reinterpret_cast<const double2*>(p + 2);
    v[0] = q0.x; v[1] = q0.y; v[2] = q1.x;
    if (NU == 4) v[NU - 1] = q1.y;
  } else {
#pragma unroll
    for (int f = 0; f < NU; ++f) v[f] = p[f];
  }
}

// Entries loaded together: their indices, then their values; the first indices are loaded before the wait
// for the cell launch.  Eight cover the nodes of a uniform mesh, which is what counts on a level of few
// blocks (26,000 nodes of a refined Q1 level 6.2 -> 5.1 us, the whole V-cycle on 16^3 with two
// refinements 505 -> 438 us); on large levels their registers cost more than the second round of loads
// (Stokes Q2/Q1 on 24^3 with two refinements, 600,000 nodes: 31 us with four, 33 us with eight).
constexpr uint32_t kLargeNodes = 152 * 1024;

template <int kBatch>
__device__ __forceinline__ void load_indices(const int32_t* idx, int32_t lo, int32_t hi, int32_t (&id)[kBatch]) {
#pragma unroll
  for (int j = 0; j < kBatch; ++j) id[j] = lo + j < hi ? idx[lo + j] : -1;
}

// The sum of one node and what follows it; id: its first indices.
template <typename T, int NU, int AFTER, int kBatch>
__device__ __forceinline__ void gather_one(const GatherArgs<T>& a, const T* buf, const int32_t* idx, int32_t lo,
                                           int32_t hi, int32_t (&id)[kBatch], uint32_t m, int64_t dof) {
  T x[NU], bb[NU], qq[NU], dd[NU];
#pragma unroll
  for (int f = 0; f < NU; ++f) {
    if (AFTER == 1 || (AFTER != 3 && ((m >> f) & 1u))) x[f] = a.src[dof + f];  // the iterate, or identity rows
    if (AFTER == 1 || AFTER == 2) bb[f] = a.b[dof + f];
    if (AFTER == 1) {
      qq[f] = a.dinv[dof + f];
      dd[f] = a.c1 != T(0) ? a.d[dof + f] : T(0);
    }
  }
  T acc[NU];
#pragma unroll
  for (int f = 0; f < NU; ++f) acc[f] = T(0);
  for (int32_t e = lo; e < hi; e += kBatch) {
    if (e != lo) load_indices(idx, e, hi, id);
    T v[kBatch][NU];
#pragma unroll
    for (int j = 0; j < kBatch; ++j)
      if (id[j] >= 0) load_slot<T, NU>(buf, id[j], v[j]);
#pragma unroll
    for (int j = 0; j < kBatch; ++j)
      if (id[j] >= 0)
#pragma unroll
        for (int f = 0; f < NU; ++f) acc[f] = add_as_reduction(acc[f], v[j][f]);
  }
#pragma unroll
  for (int f = 0; f < NU; ++f) {
    const bool fixed = (m >> f) & 1u;
    if constexpr (AFTER == 3) {
      a.dst[dof + f] = fixed ? T(0) : acc[f];
    } else {
      const T ax = fixed ? x[f] : acc[f];
      if constexpr (AFTER == 0) {
        a.dst[dof + f] = ax;
      } else if constexpr (AFTER == 2) {
        a.dst[dof + f] = bb[f] - ax;
      } else {
        const T dn = smoother_direction(a.c1, a.c2, dd[f], qq[f], bb[f] - ax);
        a.d[dof + f] = dn;
        a.dst[dof + f] = x[f] + dn;
      }
    }
  }
}

// Bound by the contributions' reads (written just before, L2-resident on all but the largest levels) and
// on small levels by the latency of three dependent loads: 7.6 us at 193,000 nodes of three FP32
// components, 3.8 us on the smallest levels (launch included; the pass it replaces, which derived the
// cells from the node's index, took 8 us there).
template <typename T, int NU, int AFTER, int kBatch>
__global__ void __launch_bounds__(256) k_gather_nodes(const GatherArgs<T> a) {
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const uint32_t i = blockIdx.x * 256u + threadIdx.x;
  const bool main = i < a.n_main, in = i < a.n_main + a.n_p;
  int32_t lo = 0, hi = 0;
  uint32_t m = 0;
  int32_t id[kBatch];
  if (in) {  // the table is constant data
    const int32_t* p = main ? a.ptr + i : a.ptr_p + (i - a.n_main);
    lo = p[0];
    hi = p[1];
    m = a.mask[i];
    load_indices(main ? a.idx : a.idx_p, lo, hi, id);
  }
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  if (!in) return;
  if (main)
    gather_one<T, NU, AFTER, kBatch>(a, a.buf, a.idx, lo, hi, id, m, (int64_t)i * NU);
  else
    gather_one<T, 1, AFTER, kBatch>(a, a.buf_p, a.idx_p, lo, hi, id, m, (int64_t)a.n_main * NU + (i - a.n_main));
}

template <typename T, int NU>
static void launch(const NodeGather& g, int prec, const NsAfterArgs& f, cudaStream_t s) {
  GatherArgs<T> a{};
  a.dst = static_cast<T*>(f.dst);
  a.src = static_cast<const T*>(f.src);
  a.b = static_cast<const T*>(f.b);
  a.dinv = static_cast<const T*>(f.dinv);
  a.d = static_cast<T*>(f.d);
  a.buf = static_cast<const T*>(g.scratch->get());
  a.buf_p = a.buf + g.main_values();
  a.ptr = g.ptr.as<int32_t>();
  a.idx = g.idx.as<int32_t>();
  a.ptr_p = g.ptr_p.as<int32_t>();
  a.idx_p = g.idx_p.as<int32_t>();
  a.mask = g.mask.as<uint8_t>();
  a.n_main = (uint32_t)g.n_main;
  a.n_p = (uint32_t)g.n_p;
  a.c1 = (T)f.c1;
  a.c2 = (T)f.c2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((g.n_main + g.n_p + 255) / 256));
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const bool large = a.n_main + a.n_p > kLargeNodes;
#define GO(AFTER)                                                                         \
  MFNS_CUDA(large ? cudaLaunchKernelEx(&cfg, k_gather_nodes<T, NU, AFTER, 4>, a)          \
                  : cudaLaunchKernelEx(&cfg, k_gather_nodes<T, NU, AFTER, 8>, a));        \
  return
  switch (f.after) {
    case 0: GO(0);
    case 1: GO(1);
    case 2: GO(2);
    default: GO(3);
  }
#undef GO
}

void gather_nodes(const NodeGather& g, int prec, const NsAfterArgs& a, cudaStream_t s) {
  switch (g.nu * 2 + (prec == 0 ? 0 : 1)) {
    case 2: return launch<double, 1>(g, prec, a, s);
    case 3: return launch<float, 1>(g, prec, a, s);
    case 4: return launch<double, 2>(g, prec, a, s);
    case 5: return launch<float, 2>(g, prec, a, s);
    case 6: return launch<double, 3>(g, prec, a, s);
    case 7: return launch<float, 3>(g, prec, a, s);
    case 8: return launch<double, 4>(g, prec, a, s);
    case 9: return launch<float, 4>(g, prec, a, s);
  }
  throw Error(kErrArg, "node pass: components per node");
}

}  // namespace mfns
