// Cell kernel of the stabilised Navier--Stokes Jacobian on uniform 3D levels, and the node pass that
// completes its product.
//
// Mapping.  A block works on C consecutive cells (lexicographic, x fastest) with Q^2 lines of Q points
// each per cell (Q = k + 1): a thread owns one line of one cell -- an x-line, then a y-line, then a
// z-line, as the contraction needs -- with the four fields of the equal-order system in one 16-byte
// (FP32) access.  The line index is the slow thread index, so the lanes of a warp are cells: every
// lane works (the warp-per-three-cells mapping of op_kernel keeps 27 of 32), shared-memory accesses
// are consecutive 16-byte words without bank conflicts, neighbouring cells' nodes are consecutive in
// memory, and the 1D tables are uniform operands instead of per-lane reads.
//
// Arithmetic.  Contractions along an owned line use the symmetry of the tables about the element
// centre (even-odd form; for Q = 3 the centre Gauss point is a node and the second derivative is
// constant along a line).  Weights and cell size are folded into the test-side tables, 1/h, the
// linearisation factors and tau into the stored point values, so a point costs 66 operations
// instead of 108 and a Q2 cell 4,600 instead of 7,500.
//
// Scatter.  No colours: the block adds the face between x-neighbours of the block in registers and
// writes its rows of node values to `rows` (one x-row of nodes per cell row, line and block; the face
// between two blocks of a cell row goes to `tails`); k_ns_nodes adds the at most four rows that
// share a node in a fixed order and applies what follows the product (store, smoother update,
// residual) while the sum is in registers.  Results are deterministic and the same for one problem
// and for several in a launch.
//
// Measured against eight colour launches of the warp-per-three-cells kernel (whole product, GB300): Q2
// 64^3 FP32 176 -> 119 us, 48^3 FP64 1849 -> 1116 us (FP64 pipe 87 % busy), Q3 31^3 FP32 61.8 -> 51 us,
// five Q1 45^3 FP32 smoothing sweeps 116 -> 50 us.  The FP32 cell launch (95 us at 64^3) is bound by
// the DRAM stream of the point values (5.7 TB/s), the node pass (about 25 us) by its rows.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "smoother.cuh"

namespace mfns {

// 1D tables of a level: symmetric (value) and antisymmetric (derivative) about the element centre.
template <typename T, int Q>
struct NsTab {
  T S[Q][Q];    // trial values at the Gauss points
  T Sp[Q][Q];   // the same / h (pressure; last trial stage applied)
  T D[Q][Q];    // collocation derivative
  T D2[Q][Q];   // second derivative times -nu / h^2 (0 without the strong viscous term)
  T St[Q][Q];   // test values, weighted: St[a][l] = S[l][a] w_l (Q = 3: / w_1)
  T Dw[Q][Q];   // W^-1 D^T W
  T Sf[Q][Q];   // last test stage: St with the remaining factors (h^3)
  T DS[Q][Q];   // derivative at the Gauss points from nodal values
  T D2S[Q][Q];  // second derivative from nodal values, scaled as D2
  T Sfp[Q][Q];  // last test stage of the pressure (h^2 times the sign of the continuity row)
  // Q = 3: half the sum and half the difference of the first row's outer entries, of S, Sp, D, St, Dw, Sf, Sfp
  T hS[2], hSp[2], hD[2], hSt[2], hDw[2], hSf[2], hSfp[2];
};

template <typename T>
struct NsProb {
  const T* src;
  const T* fq;         // point values, see ns_fq_at
  T* rows;             // [cell row][line][node along x][4]
  T* tails;            // [block][line][4]
  int32_t first_block; // multi-problem launches: first block of this problem
  int32_t n;           // cells per direction
  int32_t C;           // cells per block
  uint32_t cells;      // n^3
  T cmm, nuh2;         // factor of the mass term, nu / h^2
  T cfc, cfs, cfp;     // convection, SUPG, PSPG / continuity sign
  int32_t gen;         // 0: the three factors above are 1
};

// Offset, in units of one value, of the quad `quad` (4 values) of point l on z-line w of the cell in
// slot `lane` of block `blk`: [block][line][point][quad][(FP64: half)][slot], 16 bytes per slot.
template <typename T, int Q>
__host__ __device__ inline int64_t ns_fq_at(int64_t blk, int w, int l, int quad, int half, int lane, int C) {
  constexpr int H = sizeof(T) / 4, V = 16 / sizeof(T);
  return (((((blk * (Q * Q) + w) * Q + l) * 4 + quad) * H + half) * C + lane) * V;
}

template <typename T> struct NsVec;
template <> struct NsVec<float> {
  static constexpr int H = 1;
  using V = float4;
};
template <> struct NsVec<double> {
  static constexpr int H = 2;
  using V = double2;
};

// four values of one slot: ls slots per (entry, half)
template <typename T>
__device__ __forceinline__ void ns_ld(const T* buf, int e, int lane, int ls, T (&v)[4]) {
  const typename NsVec<T>::V* b = reinterpret_cast<const typename NsVec<T>::V*>(buf);
  if constexpr (sizeof(T) == 4) {
    const float4 q = b[e * ls + lane];
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  } else {
    const double2 q0 = b[(2 * e) * ls + lane], q1 = b[(2 * e + 1) * ls + lane];
    v[0] = q0.x; v[1] = q0.y; v[2] = q1.x; v[3] = q1.y;
  }
}
template <typename T>
__device__ __forceinline__ void ns_st(T* buf, int e, int lane, int ls, T v0, T v1, T v2, T v3) {
  typename NsVec<T>::V* b = reinterpret_cast<typename NsVec<T>::V*>(buf);
  if constexpr (sizeof(T) == 4) {
    b[e * ls + lane] = make_float4(v0, v1, v2, v3);
  } else {
    b[(2 * e) * ls + lane] = make_double2(v0, v1);
    b[(2 * e + 1) * ls + lane] = make_double2(v2, v3);
  }
}

// ---- rows in the L2: written to stay while the point values stream past, read back to be dropped
// (Q2 64^3 FP32 product 125 -> 123 us, 48^3 V-cycle 1057 -> 1026 us)
__device__ __forceinline__ void st_keep(float4* p, float a, float b, float c, float d) {
  uint64_t keep;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;\n" : "=l"(keep));
  asm volatile("st.global.L2::cache_hint.v4.f32 [%0], {%1, %2, %3, %4}, %5;\n" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d),
               "l"(keep)
               : "memory");
}
__device__ __forceinline__ void ld_last(const float* p, float (&v)[4]) {
  uint64_t once;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;\n" : "=l"(once));
  asm volatile("ld.global.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;\n"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
               : "l"(p), "l"(once)
               : "memory");
}

// ---- contractions along a line (u -> o); every product is rounded where it stands or explicitly fused,
// so that the kernel's instantiations (one problem, several) round alike
enum NsRow { kDense, kTrial, kTest };
// symmetric table; for Q = 3: kTrial: the centre row is a multiple of (0, 1, 0); kTest: the centre
// column is, and unless SCALED its entry is 1
template <int Q, NsRow R, bool SCALED, typename T>
__device__ __forceinline__ void line_sym(const T (&M)[Q][Q], const T (&h)[2], const T (&u)[Q], T (&o)[Q]) {
  if constexpr (Q == 3 && R != kDense) {
    const T e = u[0] + u[2], d = u[0] - u[2];
    const T pe = h[0], po = h[1];
    if constexpr (R == kTrial) {
      const T E = fma(pe, e, M[0][1] * u[1]);
      o[0] = fma(po, d, E);
      o[2] = fma(-po, d, E);
      o[1] = SCALED ? mul_rn(M[1][1], u[1]) : u[1];
    } else {
      const T E = pe * e;
      o[0] = fma(po, d, E);
      o[2] = fma(-po, d, E);
      o[1] = fma(M[1][0], e, SCALED ? M[1][1] * u[1] : u[1]);
    }
  } else {
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      T s = mul_rn(M[i][0], u[0]);
#pragma unroll
      for (int a = 1; a < Q; ++a) s = fma(M[i][a], u[a], s);
      o[i] = s;
    }
  }
}
// derivative at the Gauss points and, with SECOND, the scaled second derivative (Q = 3: one value)
template <int Q, bool SECOND, typename T>
__device__ __forceinline__ void line_deriv(const T (&D)[Q][Q], const T (&h)[2], const T (&D2)[Q][Q], const T (&u)[Q],
                                           T (&o)[Q], T (&x)[Q]) {
  if constexpr (Q == 3) {
    // rows (a, b, c), (-d, 0, d), (-c, -b, -a) with a + b + c = 0; D2 rows q (1, -2, 1)
    const T e = u[0] + u[2], d = u[0] - u[2];
    const T t = fma(T(-0.5), e, u[1]);
    const T m = mul_rn(h[1], d);
    o[0] = fma(D[0][1], t, m);
    o[2] = fma(-D[0][1], t, m);
    o[1] = mul_rn(D[1][0], d);
    if (SECOND) x[0] = x[1] = x[2] = mul_rn(D2[0][1], t);
  } else if constexpr (Q == 2) {
    o[0] = o[1] = mul_rn(D[0][1], u[1] - u[0]);
    if (SECOND) x[0] = x[1] = T(0);
  } else {
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      T s = mul_rn(D[i][0], u[0]), s2 = mul_rn(D2[i][0], u[0]);
#pragma unroll
      for (int a = 1; a < Q; ++a) {
        s = fma(D[i][a], u[a], s);
        s2 = fma(D2[i][a], u[a], s2);
      }
      o[i] = s;
      if (SECOND) x[i] = s2;
    }
  }
}
// o = Dw u, or with ADD o += Dw u
template <int Q, bool ADD, typename T>
__device__ __forceinline__ void line_dwt(const T (&Dw)[Q][Q], const T (&h)[2], const T (&u)[Q], T (&o)[Q]) {
  if constexpr (Q == 3) {
    const T e = u[0] + u[2], d = u[0] - u[2];
    const T m = h[0], k = h[1];
    const T X = fma(m, e, Dw[0][1] * u[1]);
    o[0] = fma(k, d, ADD ? o[0] + X : X);
    o[2] = fma(k, d, ADD ? o[2] - X : -X);
    o[1] = ADD ? fma(Dw[1][0], d, o[1]) : mul_rn(Dw[1][0], d);
  } else {
#pragma unroll
    for (int i = 0; i < Q; ++i)
#pragma unroll
      for (int a = 0; a < Q; ++a) o[i] = ADD || a ? fma(Dw[i][a], u[a], o[i]) : mul_rn(Dw[i][a], u[a]);
  }
}

// The pointwise Jacobian at one Gauss point.  v: velocity and p/h; gx, gy, gz: reference derivatives of
// the velocity and (entry 3) grad p; lap: -nu lap u; F: quads (U/h, tau), (G_i, Rb_i).  Out: value
// and gradient coefficients of the test functions (weights and cell size left to the test tables).
template <typename T>
__device__ __forceinline__ void ns_point(const T (&v)[4], const T (&gx)[4], const T (&gy)[4], const T (&gz)[4],
                                         const T (&lap)[3], const T (&F)[4][4], const NsProb<T>& P, T (&c0)[4],
                                         T (&cx)[4], T (&cy)[4], T (&cz)[4]) {
  T r[3];
  const T gp[3] = {gx[3], gy[3], gz[3]};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    T c = F[0][0] * gx[i];
    c = fma(F[0][1], gy[i], c);
    c = fma(F[0][2], gz[i], c);
    if (P.gen) c = mul_rn(c, P.cfc);
    c = fma(P.cmm, v[i], c);
    c = fma(F[1 + i][0], v[0], c);
    c = fma(F[1 + i][1], v[1], c);
    c = fma(F[1 + i][2], v[2], c);
    c0[i] = c;
    r[i] = mul_rn(F[0][3], c + (gp[i] + lap[i]));
  }
  c0[3] = gx[0] + gy[1] + gz[2];
  T s[3] = {r[0], r[1], r[2]}, q[3] = {r[0], r[1], r[2]};
  if (P.gen) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      s[i] = mul_rn(s[i], P.cfs);
      q[i] = mul_rn(q[i], P.cfp);
    }
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const T a = F[1 + i][3];
    cx[i] = fma(s[i], F[0][0], fma(a, v[0], i == 0 ? fma(P.nuh2, gx[0], -v[3]) : P.nuh2 * gx[i]));
    cy[i] = fma(s[i], F[0][1], fma(a, v[1], i == 1 ? fma(P.nuh2, gy[1], -v[3]) : P.nuh2 * gy[i]));
    cz[i] = fma(s[i], F[0][2], fma(a, v[2], i == 2 ? fma(P.nuh2, gz[2], -v[3]) : P.nuh2 * gz[i]));
  }
  cx[3] = q[0];
  cy[3] = q[1];
  cz[3] = q[2];
}

// Block shapes.  FP32: one warp per line, up to 32 cells; the point values of the block come in with
// one TMA bulk copy (Q < 4).  FP64: threads packed over (line, cell), 128 threads at most -- with
// 2 DFMA per SM and cycle only the number of operations counts, and a single warp's operations
// take 64 cycles each, so blocks are small and idle lanes are avoided.
template <int K, typename T>
struct NsShape {
  static constexpr int Q = K + 1, NL = Q * Q;
  static constexpr bool UNI = sizeof(T) == 4;     // lanes of a warp share the line
  static constexpr bool LINES = sizeof(T) == 8;   // x / y derivatives by the owners of the lines
  static constexpr bool STAGE = sizeof(T) == 4 && Q < 4;
  static constexpr int CMAX = UNI ? 32 : 128 / NL;
  static constexpr int THREADS = UNI ? NL * 32 : 128;
  // FP64: five blocks' worth of registers (spilling a little); with four, the 1,323 blocks of a 21^3 level
  // need a second round (V-cycle 1863 -> 1795 us)
  static constexpr int MINB = UNI ? (Q == 2 ? 6 : Q == 3 ? 2 : 1) : (Q == 4 ? 3 : 5);
  static constexpr int NXX = !LINES || Q == 2 ? 0 : Q == 3 ? NL : NL * Q;  // second-derivative entries per cell
  __host__ __device__ static constexpr int slots(int C) { return UNI ? 32 : C; }
  __host__ __device__ static constexpr size_t buf_values(int C) { return (size_t)NL * Q * 4 * slots(C); }
  __host__ __device__ static constexpr size_t stage_bytes(int C) {
    return STAGE ? (size_t)NL * Q * 16 * sizeof(T) * C : 0;
  }
  __host__ __device__ static constexpr size_t smem(int C) {
    return stage_bytes(C) + (3 * buf_values(C) + 2 * (size_t)NXX * 2 * slots(C)) * sizeof(T) + 16;
  }
  __host__ __device__ static constexpr int threads(int C) { return UNI ? THREADS : (C * NL + 31) / 32 * 32; }
};

template <typename T, int Q>
struct NsDesc {
  NsTab<T, Q> tab;
  NsProb<T> p;
};

template <typename T, int Q>
struct NsArgs {
  NsDesc<T, Q> one;
  const NsDesc<T, Q>* probs;  // multi-problem launches: one descriptor per problem (device)
  const int32_t* block_pid;   // ... and the problem of every block
  int* err;
};

__device__ __forceinline__ bool ns_mbar_try(unsigned addr) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(addr)
      : "memory");
  return ok != 0;
}

template <int K, typename T, bool MULTI>
__global__ void __launch_bounds__(NsShape<K, T>::THREADS, NsShape<K, T>::MINB)
k_ns_cells(const __grid_constant__ NsArgs<T, K + 1> args) {
  using Sh = NsShape<K, T>;
  constexpr int Q = K + 1, NL = Q * Q;
  extern __shared__ __align__(128) unsigned char ns_smem[];
  const NsDesc<T, Q>& desc = MULTI ? args.probs[args.block_pid[blockIdx.x]] : args.one;
  const NsTab<T, Q>& tab = desc.tab;
  const NsProb<T>& P = desc.p;
  const int blk = (int)blockIdx.x - (MULTI ? P.first_block : 0);
  const int C = P.C, n = P.n, ls = Sh::UNI ? 32 : C;
  int w, lane;
  if constexpr (Sh::UNI) {
    w = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    lane = threadIdx.x & 31;
  } else {
    w = (int)threadIdx.x / C;
    lane = (int)threadIdx.x - w * C;
  }
  const bool work = Sh::UNI || w < NL;  // packed blocks: threads beyond the last line only synchronise
  if (!work) w = 0;
  T* stage = reinterpret_cast<T*>(ns_smem);
  T* A = reinterpret_cast<T*>(ns_smem + Sh::stage_bytes(C));
  T* B = A + Sh::buf_values(C);
  T* G = B + Sh::buf_values(C);
  T* XX = G + Sh::buf_values(C);
  T* YY = XX + (size_t)Sh::NXX * 2 * ls;
  const unsigned mbar = (unsigned)__cvta_generic_to_shared(ns_smem + Sh::smem(C) - 16);
  // the next kernel of the stream may be scheduled; it waits for this grid before it reads `rows`
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  if constexpr (Sh::STAGE) {
    // the block's point values: constant data, so the copy need not wait for the previous kernel
    if (threadIdx.x == 0) {
      const unsigned bytes = (unsigned)Sh::stage_bytes(C);
      const unsigned sdst = (unsigned)__cvta_generic_to_shared(stage);
      const T* g = P.fq + ns_fq_at<T, Q>(blk, 0, 0, 0, 0, 0, C);
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(mbar) : "memory");
      asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(mbar), "r"(bytes) : "memory");
      asm volatile(
          "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(sdst),
          "l"(g), "r"(bytes), "r"(mbar)
          : "memory");
    }
  }
  // the slot's cell (spare slots repeat the last cell and write nothing)
  const uint32_t t = (uint32_t)blk * (uint32_t)C + (uint32_t)lane;
  const bool valid = work && lane < C && t < P.cells;
  const uint32_t tt = t < P.cells ? t : P.cells - 1;
  const int cx = (int)(tt % (uint32_t)n), row = (int)(tt / (uint32_t)n);
  const int cy = row % n, cz = row / n;
  const int M = K * n + 1;
  const int l0 = w % Q, l1 = w / Q;
  // lines of this thread: x-line (l0, l1) along x, y-line (l0, ., l1), z-line (l0, l1, .)
  const int px = Q * (l0 + Q * l1), py = l0 + Q * Q * l1, pz = l0 + Q * l1;
  const int slot = lane < ls ? lane : 0;

  // ---- trial side: values at the Gauss points, one direction after the other (src may have been written
  // by a kernel that this one overlapped until here: ordinary loads, not read-only ones)
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  const int iy = K * cy + l0, iz = K * cz + l1;
  const bool bnd_line = iy == 0 || iy == M - 1 || iz == 0 || iz == M - 1;
  {
    T u[4][Q];
    const T* s = P.src + ((int64_t)(K * cx) + (int64_t)M * ((int64_t)iy + (int64_t)M * iz)) * 4;
#pragma unroll
    for (int a = 0; a < Q; ++a) {
      const bool bnd = bnd_line || (a == 0 && cx == 0) || (a == K && cx == n - 1);
      if constexpr (sizeof(T) == 4) {
        const float4 q = reinterpret_cast<const float4*>(s)[a];
        u[0][a] = q.x; u[1][a] = q.y; u[2][a] = q.z; u[3][a] = q.w;
      } else {
        const double2 q0 = reinterpret_cast<const double2*>(s)[2 * a];
        const double2 q1 = reinterpret_cast<const double2*>(s)[2 * a + 1];
        u[0][a] = q0.x; u[1][a] = q0.y; u[2][a] = q1.x; u[3][a] = q1.y;
      }
#pragma unroll
      for (int f = 0; f < 3; ++f) u[f][a] = bnd ? T(0) : u[f][a];
    }
    T o[4][Q];
#pragma unroll
    for (int f = 0; f < 3; ++f) line_sym<Q, kTrial, false>(tab.S, tab.hS, u[f], o[f]);
    line_sym<Q, kTrial, true>(tab.Sp, tab.hSp, u[3], o[3]);
    if (work)
#pragma unroll
      for (int a = 0; a < Q; ++a) ns_st(A, px + a, slot, ls, o[0][a], o[1][a], o[2][a], o[3][a]);
  }
  auto load_line = [&](const T* buf, int p0, int st, T (&u)[4][Q]) {
#pragma unroll
    for (int a = 0; a < Q; ++a) {
      T q[4];
      ns_ld(buf, p0 + st * a, slot, ls, q);
#pragma unroll
      for (int f = 0; f < 4; ++f) u[f][a] = q[f];
    }
  };
  auto store_line = [&](T* buf, int p0, int st, const T (&u)[4][Q]) {
    if (work)
#pragma unroll
      for (int a = 0; a < Q; ++a) ns_st(buf, p0 + st * a, slot, ls, u[0][a], u[1][a], u[2][a], u[3][a]);
  };
  __syncthreads();
  {
    T u[4][Q], o[4][Q];
    load_line(A, py, Q, u);
#pragma unroll
    for (int f = 0; f < 4; ++f) line_sym<Q, kTrial, false>(tab.S, tab.hS, u[f], o[f]);
    store_line(A, py, Q, o);  // a thread's own entries: in place
  }
  __syncthreads();
  T val[4][Q], dz[4][Q], lz[3][Q];
  {
    T u[4][Q];
    load_line(A, pz, Q * Q, u);
#pragma unroll
    for (int f = 0; f < 4; ++f) line_sym<Q, kTrial, false>(tab.S, tab.hS, u[f], val[f]);
    store_line(A, pz, Q * Q, val);
    T dummy[Q];
#pragma unroll
    for (int f = 0; f < 3; ++f) line_deriv<Q, true>(tab.D, tab.hD, tab.D2, val[f], dz[f], lz[f]);
    line_deriv<Q, false>(tab.D, tab.hD, tab.D2, val[3], dz[3], dummy);
  }
  __syncthreads();
  if constexpr (Sh::LINES) {
    // derivatives along the owned x- and y-lines; the second derivative of the component along the
    // line's direction rides in the pressure derivative's place (they are only needed as a sum)
    T u[4][Q], o[4][Q], x2[3][Q], dummy[Q];
    load_line(A, px, 1, u);
#pragma unroll
    for (int f = 0; f < 3; ++f) line_deriv<Q, true>(tab.D, tab.hD, tab.D2, u[f], o[f], x2[f]);
    line_deriv<Q, false>(tab.D, tab.hD, tab.D2, u[3], o[3], dummy);
#pragma unroll
    for (int a = 0; a < Q; ++a)
      if (Q > 2) o[3][a] += x2[0][a];
    store_line(B, px, 1, o);
    if (Q > 2 && work) {
      double2* x = reinterpret_cast<double2*>(XX);
      if (Q == 3) x[w * ls + slot] = make_double2(x2[1][0], x2[2][0]);
      else
#pragma unroll
        for (int a = 0; a < Q; ++a) x[(px + a) * ls + slot] = make_double2(x2[1][a], x2[2][a]);
    }
    load_line(A, py, Q, u);
#pragma unroll
    for (int f = 0; f < 3; ++f) line_deriv<Q, true>(tab.D, tab.hD, tab.D2, u[f], o[f], x2[f]);
    line_deriv<Q, false>(tab.D, tab.hD, tab.D2, u[3], o[3], dummy);
#pragma unroll
    for (int a = 0; a < Q; ++a)
      if (Q > 2) o[3][a] += x2[1][a];
    store_line(G, py, Q, o);
    if (Q > 2 && work) {
      double2* y = reinterpret_cast<double2*>(YY);
      if (Q == 3) y[w * ls + slot] = make_double2(x2[0][0], x2[2][0]);
      else
#pragma unroll
        for (int a = 0; a < Q; ++a) y[(py + Q * a) * ls + slot] = make_double2(x2[0][a], x2[2][a]);
    }
    __syncthreads();
  }

  // ---- pointwise terms along the z-line
  if constexpr (Sh::STAGE) {
    constexpr uint32_t kLimit = 1u << 22;
    bool done = false;
    for (uint32_t it = 0; it < kLimit && !done; ++it) done = ns_mbar_try(mbar);
    if (!done) {  // report, and give the copy a last chance to end before the block does
      if (args.err) atomicOr(args.err, 1);
      for (uint32_t it = 0; it < kLimit && !done; ++it) done = ns_mbar_try(mbar);
    }
  }
  T acc[4][Q], cz4[4][Q];
#pragma unroll
  for (int l = 0; l < Q; ++l) {
    T F[4][4];
    const int fl = lane < C ? lane : C - 1;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if constexpr (Sh::STAGE) {
        const float4 f4 = reinterpret_cast<const float4*>(stage)[((w * Q + l) * 4 + q) * C + fl];
        F[q][0] = f4.x; F[q][1] = f4.y; F[q][2] = f4.z; F[q][3] = f4.w;
      } else if constexpr (sizeof(T) == 4) {
        const float4 f4 = __ldg(reinterpret_cast<const float4*>(P.fq + ns_fq_at<T, Q>(blk, w, l, q, 0, fl, C)));
        F[q][0] = f4.x; F[q][1] = f4.y; F[q][2] = f4.z; F[q][3] = f4.w;
      } else {
        const double2 a = __ldg(reinterpret_cast<const double2*>(P.fq + ns_fq_at<T, Q>(blk, w, l, q, 0, fl, C)));
        const double2 b = __ldg(reinterpret_cast<const double2*>(P.fq + ns_fq_at<T, Q>(blk, w, l, q, 1, fl, C)));
        F[q][0] = a.x; F[q][1] = a.y; F[q][2] = b.x; F[q][3] = b.y;
      }
    }
    T gx[4], gy[4], gz[4], v[4], lap[3], c0[4], cxp[4], cyp[4], czp[4];
    const int p = pz + Q * Q * l;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      v[f] = val[f][l];
      gz[f] = dz[f][l];
    }
    if constexpr (Sh::LINES) {
      ns_ld(B, p, slot, ls, gx);
      ns_ld(G, p, slot, ls, gy);
      lap[0] = lap[1] = lap[2] = T(0);
      if (Q > 2) {
        const double2 x = reinterpret_cast<const double2*>(XX)[(Q == 3 ? l1 + Q * l : p) * ls + slot];
        const double2 y = reinterpret_cast<const double2*>(YY)[(Q == 3 ? l0 + Q * l : p) * ls + slot];
        lap[0] = y.x + lz[0][l];
        lap[1] = x.x + lz[1][l];
        lap[2] = (x.y + y.y) + lz[2][l];
      }
    } else {
      // the z-line's owner forms its own x and y derivatives from the neighbours in the plane
      T x[4], y[4];
#pragma unroll
      for (int f = 0; f < 4; ++f) gx[f] = gy[f] = T(0);
#pragma unroll
      for (int f = 0; f < 3; ++f) lap[f] = Q > 2 ? lz[f][l] : T(0);
#pragma unroll
      for (int a = 0; a < Q; ++a) {
        ns_ld(A, a + Q * (l1 + Q * l), slot, ls, x);
        ns_ld(A, l0 + Q * (a + Q * l), slot, ls, y);
        const T dx = tab.D[l0][a], dy = tab.D[l1][a];
#pragma unroll
        for (int f = 0; f < 4; ++f) {
          gx[f] = a ? fma(dx, x[f], gx[f]) : dx * x[f];
          gy[f] = a ? fma(dy, y[f], gy[f]) : dy * y[f];
        }
        if (Q > 2) {
          const T dx2 = tab.D2[l0][a], dy2 = tab.D2[l1][a];
#pragma unroll
          for (int f = 0; f < 3; ++f) lap[f] = fma(dx2, x[f], fma(dy2, y[f], lap[f]));
        }
      }
    }
    ns_point<T>(v, gx, gy, gz, lap, F, P, c0, cxp, cyp, czp);
    if (work) {
      ns_st(B, p, slot, ls, cxp[0], cxp[1], cxp[2], cxp[3]);
      ns_st(G, p, slot, ls, cyp[0], cyp[1], cyp[2], cyp[3]);
    }
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      acc[f][l] = c0[f];
      cz4[f][l] = czp[f];
    }
  }
#pragma unroll
  for (int f = 0; f < 4; ++f) line_dwt<Q, true>(tab.Dw, tab.hDw, cz4[f], acc[f]);
  __syncthreads();
  // ---- test side: transposed derivatives, then the transposed values z, y, x
  if constexpr (Sh::LINES) {
    T u[4][Q], o[4][Q];
    load_line(B, px, 1, u);
#pragma unroll
    for (int f = 0; f < 4; ++f) line_dwt<Q, false>(tab.Dw, tab.hDw, u[f], o[f]);
    store_line(B, px, 1, o);
    load_line(G, py, Q, u);
#pragma unroll
    for (int f = 0; f < 4; ++f) line_dwt<Q, false>(tab.Dw, tab.hDw, u[f], o[f]);
    store_line(G, py, Q, o);
    __syncthreads();
#pragma unroll
    for (int l = 0; l < Q; ++l) {
      T x[4], y[4];
      ns_ld(B, pz + Q * Q * l, slot, ls, x);
      ns_ld(G, pz + Q * Q * l, slot, ls, y);
#pragma unroll
      for (int f = 0; f < 4; ++f) acc[f][l] += x[f] + y[f];
    }
  } else {
#pragma unroll
    for (int l = 0; l < Q; ++l)
#pragma unroll
      for (int a = 0; a < Q; ++a) {
        T x[4], y[4];
        ns_ld(B, a + Q * (l1 + Q * l), slot, ls, x);
        ns_ld(G, l0 + Q * (a + Q * l), slot, ls, y);
        const T dx = tab.Dw[l0][a], dy = tab.Dw[l1][a];
#pragma unroll
        for (int f = 0; f < 4; ++f) acc[f][l] = fma(dx, x[f], fma(dy, y[f], acc[f][l]));
      }
  }
  {
    T o[4][Q];
#pragma unroll
    for (int f = 0; f < 4; ++f) line_sym<Q, kTest, false>(tab.St, tab.hSt, acc[f], o[f]);
    store_line(A, pz, Q * Q, o);
  }
  __syncthreads();
  {
    T u[4][Q], o[4][Q];
    load_line(A, py, Q, u);
#pragma unroll
    for (int f = 0; f < 4; ++f) line_sym<Q, kTest, false>(tab.St, tab.hSt, u[f], o[f]);
    store_line(A, py, Q, o);
  }
  __syncthreads();
  T r[4][Q];
  {
    T u[4][Q];
    load_line(A, px, 1, u);
#pragma unroll
    for (int f = 0; f < 3; ++f) line_sym<Q, kTest, true>(tab.Sf, tab.hSf, u[f], r[f]);
    line_sym<Q, kTest, true>(tab.Sfp, tab.hSfp, u[3], r[3]);
  }
  // ---- the face between x-neighbours of the block, then the node values of the row
  T left[4];
  if constexpr (Sh::UNI) {
#pragma unroll
    for (int f = 0; f < 4; ++f) left[f] = __shfl_up_sync(0xffffffffu, r[f][K], 1);
  } else {
    // (every thread has read its x-line; entries are a thread's own until the barrier)
    if (work) ns_st(A, px, slot, ls, r[0][K], r[1][K], r[2][K], r[3][K]);
    __syncthreads();
    ns_ld(A, px, slot > 0 ? slot - 1 : 0, ls, left);
  }
  const bool joined = lane > 0 && cx > 0;
  if (valid) {
#pragma unroll
    for (int f = 0; f < 4; ++f) r[f][0] += joined ? left[f] : T(0);
    T* out = P.rows + (((int64_t)row * NL + w) * M + K * cx) * 4;
    auto put = [](T* d, T a, T b, T c, T e) {
      if constexpr (sizeof(T) == 4) {
        *reinterpret_cast<float4*>(d) = make_float4(a, b, c, e);
      } else {
        *reinterpret_cast<double2*>(d) = make_double2(a, b);
        *reinterpret_cast<double2*>(d + 2) = make_double2(c, e);
      }
    };
#pragma unroll
    for (int a = 0; a < K; ++a) put(out + 4 * a, r[0][a], r[1][a], r[2][a], r[3][a]);
    if (cx == n - 1) put(out + 4 * K, r[0][K], r[1][K], r[2][K], r[3][K]);
    else if (lane == C - 1)
      put(P.tails + ((int64_t)blk * NL + w) * 4, r[0][K], r[1][K], r[2][K], r[3][K]);
  }
}

// ------------------------------------------------------------------------------------ small FP64 levels: items
// FP64 levels that do not fill the chip: a block of 128 threads works on C cells, and every stage splits its
// work into items of one field of one line, or one point, over all threads; the fields live in shared
// memory between the stages.  A thread then does a quarter of the operations that a line's owner does,
// which is the time of a small FP64 level: one warp's FP64 operations take 64 cycles each.  Warps are
// rotated by the block index, because a stage with few items would otherwise always load the same
// quarter of the SM.
template <int K>
struct NsItems {
  static constexpr int Q = K + 1, NL = Q * Q, NP = NL * Q, THREADS = 128;
  static constexpr int NX = Q == 2 ? 0 : Q == 3 ? NL : NP;  // second derivatives per direction and field
  static constexpr int CELL = 16 * NP + 9 * NX;              // values of a cell
  __host__ __device__ static constexpr size_t smem(int C) { return (size_t)CELL * C * 8; }
};

template <int K, bool MULTI>
__global__ void __launch_bounds__(128) k_ns_items(const __grid_constant__ NsArgs<double, K + 1> args) {
  using T = double;
  using It = NsItems<K>;
  constexpr int Q = K + 1, NL = Q * Q, NP = NL * Q, NX = It::NX;
  extern __shared__ __align__(128) unsigned char ns_smem[];
  const NsDesc<T, Q>& desc = MULTI ? args.probs[args.block_pid[blockIdx.x]] : args.one;
  const NsTab<T, Q>& tab = desc.tab;
  const NsProb<T>& P = desc.p;
  const int blk = (int)blockIdx.x - (MULTI ? P.first_block : 0);
  const int C = P.C, n = P.n, M = K * n + 1;
  const int tid = (int)((threadIdx.x + 32u * (blockIdx.x & 3u)) & 127u);
  T* mem = reinterpret_cast<T*>(ns_smem);
  // per cell: U[4][NP] (values, then sums), G[3][4][NP] (derivatives, then their coefficients), X[3][3][NX]
  auto U = [&](int c, int f) { return mem + c * It::CELL + f * NP; };
  auto G = [&](int c, int d, int f) { return mem + c * It::CELL + (4 + 4 * d + f) * NP; };
  auto X = [&](int c, int d, int f) { return mem + c * It::CELL + 16 * NP + (3 * d + f) * NX; };
  const uint32_t t0 = (uint32_t)blk * (uint32_t)C;
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  auto line = [](int dir, int w, int& p0, int& st) {  // entries of line w along dir
    p0 = dir == 0 ? Q * w : dir == 1 ? w % Q + Q * Q * (w / Q) : w;
    st = dir == 0 ? 1 : dir == 1 ? Q : Q * Q;
  };
  // ---- trial values: x (from the nodal values), y, z
  for (int it = tid; it < C * 4 * NL; it += 128) {
    const int c = it / (4 * NL), f = it / NL % 4, w = it % NL;
    const uint32_t t = min(t0 + (uint32_t)c, P.cells - 1);
    const int cx = (int)(t % (uint32_t)n), row = (int)(t / (uint32_t)n), cy = row % n, cz = row / n;
    const int iy = K * cy + w % Q, iz = K * cz + w / Q;
    const bool bl = iy == 0 || iy == M - 1 || iz == 0 || iz == M - 1;
    const T* s = P.src + ((int64_t)(K * cx) + (int64_t)M * ((int64_t)iy + (int64_t)M * iz)) * 4 + f;
    T u[Q], o[Q];
#pragma unroll
    for (int a = 0; a < Q; ++a) {
      u[a] = s[4 * a];
      if (f < 3 && (bl || (a == 0 && cx == 0) || (a == K && cx == n - 1))) u[a] = T(0);
    }
    if (f < 3) line_sym<Q, kTrial, false>(tab.S, tab.hS, u, o);
    else line_sym<Q, kTrial, true>(tab.Sp, tab.hSp, u, o);
#pragma unroll
    for (int a = 0; a < Q; ++a) U(c, f)[Q * w + a] = o[a];
  }
#pragma unroll
  for (int dir = 1; dir < 3; ++dir) {
    __syncthreads();
    for (int it = tid; it < C * 4 * NL; it += 128) {
      const int c = it / (4 * NL), f = it / NL % 4, w = it % NL;
      int p0, st;
      line(dir, w, p0, st);
      T u[Q], o[Q];
#pragma unroll
      for (int a = 0; a < Q; ++a) u[a] = U(c, f)[p0 + st * a];
      line_sym<Q, kTrial, false>(tab.S, tab.hS, u, o);
#pragma unroll
      for (int a = 0; a < Q; ++a) U(c, f)[p0 + st * a] = o[a];
    }
  }
  __syncthreads();
  // ---- derivatives along every line
  for (int it = tid; it < C * 12 * NL; it += 128) {
    const int c = it / (12 * NL), d = it / (4 * NL) % 3, f = it / NL % 4, w = it % NL;
    int p0, st;
    line(d, w, p0, st);
    T u[Q], o[Q], x2[Q];
#pragma unroll
    for (int a = 0; a < Q; ++a) u[a] = U(c, f)[p0 + st * a];
    line_deriv<Q, true>(tab.D, tab.hD, tab.D2, u, o, x2);
#pragma unroll
    for (int a = 0; a < Q; ++a) G(c, d, f)[p0 + st * a] = o[a];
    if (f < 3) {
      if (Q == 3) X(c, d, f)[w] = x2[0];
      else if (Q > 3)
#pragma unroll
        for (int a = 0; a < Q; ++a) X(c, d, f)[p0 + st * a] = x2[a];
    }
  }
  __syncthreads();
  // ---- pointwise terms
  for (int it = tid; it < C * NP; it += 128) {
    const int c = it / NP, p = it % NP, i = p % Q, j = p / Q % Q, l = p / NL;
    T F[4][4], v[4], gx[4], gy[4], gz[4], lap[3], c0[4], cxp[4], cyp[4], czp[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double2 a = __ldg(reinterpret_cast<const double2*>(P.fq + ns_fq_at<T, Q>(blk, p % NL, l, q, 0, c, C)));
      const double2 b = __ldg(reinterpret_cast<const double2*>(P.fq + ns_fq_at<T, Q>(blk, p % NL, l, q, 1, c, C)));
      F[q][0] = a.x; F[q][1] = a.y; F[q][2] = b.x; F[q][3] = b.y;
    }
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      v[f] = U(c, f)[p];
      gx[f] = G(c, 0, f)[p];
      gy[f] = G(c, 1, f)[p];
      gz[f] = G(c, 2, f)[p];
    }
#pragma unroll
    for (int f = 0; f < 3; ++f)
      lap[f] = Q == 2 ? T(0)
                      : (X(c, 0, f)[Q == 3 ? j + Q * l : p] + X(c, 1, f)[Q == 3 ? i + Q * l : p]) +
                            X(c, 2, f)[Q == 3 ? i + Q * j : p];
    ns_point<T>(v, gx, gy, gz, lap, F, P, c0, cxp, cyp, czp);
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      U(c, f)[p] = c0[f];
      G(c, 0, f)[p] = cxp[f];
      G(c, 1, f)[p] = cyp[f];
      G(c, 2, f)[p] = czp[f];
    }
  }
  __syncthreads();
  // ---- test side: transposed derivatives, then z, y, x
  for (int it = tid; it < C * 12 * NL; it += 128) {
    const int c = it / (12 * NL), d = it / (4 * NL) % 3, f = it / NL % 4, w = it % NL;
    int p0, st;
    line(d, w, p0, st);
    T u[Q], o[Q];
#pragma unroll
    for (int a = 0; a < Q; ++a) u[a] = G(c, d, f)[p0 + st * a];
    line_dwt<Q, false>(tab.Dw, tab.hDw, u, o);
#pragma unroll
    for (int a = 0; a < Q; ++a) G(c, d, f)[p0 + st * a] = o[a];
  }
#pragma unroll
  for (int dir = 2; dir >= 0; --dir) {
    __syncthreads();
    for (int it = tid; it < C * 4 * NL; it += 128) {
      const int c = it / (4 * NL), f = it / NL % 4, w = it % NL;
      int p0, st;
      line(dir, w, p0, st);
      T u[Q], o[Q];
#pragma unroll
      for (int a = 0; a < Q; ++a) {
        const int p = p0 + st * a;
        u[a] = U(c, f)[p];
        if (dir == 2) u[a] = (u[a] + G(c, 0, f)[p]) + (G(c, 1, f)[p] + G(c, 2, f)[p]);
      }
      if (dir > 0) line_sym<Q, kTest, false>(tab.St, tab.hSt, u, o);
      else if (f < 3) line_sym<Q, kTest, true>(tab.Sf, tab.hSf, u, o);
      else line_sym<Q, kTest, true>(tab.Sfp, tab.hSfp, u, o);
#pragma unroll
      for (int a = 0; a < Q; ++a) U(c, f)[p0 + st * a] = o[a];
    }
  }
  __syncthreads();
  // ---- rows of node values; the face between x-neighbours of the block is added here
  for (int it = tid; it < C * NP; it += 128) {
    const int c = it / NP, p = it % NP, w = p / Q, a = p % Q;  // x-line w, node a
    const uint32_t t = t0 + (uint32_t)c;
    if (t >= P.cells) continue;
    const int cx = (int)(t % (uint32_t)n), row = (int)(t / (uint32_t)n);
    T r[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) r[f] = U(c, f)[p];
    T* out = P.rows + (((int64_t)row * NL + w) * M + K * cx + a) * 4;
    if (a == 0 && c > 0 && cx > 0)
#pragma unroll
      for (int f = 0; f < 4; ++f) r[f] += U(c - 1, f)[p + K];
    if (a == K && cx < n - 1) {
      if (c < C - 1) continue;  // added by the neighbour
      out = P.tails + ((int64_t)blk * NL + w) * 4;
    }
    *reinterpret_cast<double2*>(out) = make_double2(r[0], r[1]);
    *reinterpret_cast<double2*>(out + 2) = make_double2(r[2], r[3]);
  }
}

// ------------------------------------------------------------------------------------ FP32: planes
// FP32 threads own a whole z-plane of points of a cell (Q x Q points, four fields in registers): the x
// and y contractions need no exchange at all, the z contractions one pass of 16-byte words through
// shared memory each way.  Bound by the DRAM stream of the point values; the line kernel above, with
// a thread per line, is bound by shared-memory bandwidth here (Q2 64^3: 125 us against 95 us for the
// cells alone), but its shorter threads are faster on levels without full blocks (Q2 8^3 and below:
// 5.2 us against 6.8 us).
//
// For Q = 4 the loop over the rows of points stays a loop (ROLL): unrolled, the kernel is 97 KB of
// instructions, which a pass behind other kernels waits for (Q3 31^3, product: first pass on new vectors
// 95 us, repeated 58 us; rolled, 55 KB: 76 and 51 us; the colour launches that both replace 84 and 61 us).
// The loop turns the rows of the registers, so that the current one keeps its place (Q = 3 is faster
// unrolled: 64^3 130 us against 143 us), and asks for no prefetch of the block's point values: its loads wait
// behind it (8 warps a SM; rolled with the prefetch 79 and 54 us).
template <int K>
struct NsPlane {
  static constexpr int Q = K + 1, NL = Q * Q, THREADS = 32 * Q;
  static constexpr int MINB = Q == 2 ? 8 : Q == 3 ? 5 : 2;
  static constexpr bool ROLL = Q == 4;
  static constexpr int RING = Q == 3 ? 2 : 4;  // points of a thread's plane on their way (shared memory allows)
  static_assert(!ROLL || RING == Q, "rolled rows: the slot of a point is its place in the row");
  static constexpr size_t BUF = (size_t)NL * Q * 32 * 16;
  static constexpr size_t SMEM = 2 * BUF + (size_t)RING * 4 * THREADS * 16;
};

template <int K, bool MULTI>
__global__ void __launch_bounds__(NsPlane<K>::THREADS, NsPlane<K>::MINB)
k_ns_planes(const __grid_constant__ NsArgs<float, K + 1> args) {
  using T = float;
  constexpr int Q = K + 1, NL = Q * Q;
  extern __shared__ __align__(128) unsigned char ns_smem[];
  const NsDesc<T, Q>& desc = MULTI ? args.probs[args.block_pid[blockIdx.x]] : args.one;
  const NsTab<T, Q>& tab = desc.tab;
  const NsProb<T>& P = desc.p;
  const int blk = (int)blockIdx.x - (MULTI ? P.first_block : 0);
  const int C = P.C, n = P.n;
  const int l = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);  // the plane
  const int lane = threadIdx.x & 31;
  T* E = reinterpret_cast<T*>(ns_smem);
  T* Z = E + NL * Q * 32 * 4;
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const T* fqb = P.fq + ns_fq_at<T, Q>(blk, 0, 0, 0, 0, 0, C);
  if (!NsPlane<K>::ROLL && threadIdx.x == 0) {  // the block's point values (constant data) towards the L2
    const unsigned bytes = (unsigned)(NL * Q * 64) * (unsigned)C;
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(fqb), "r"(bytes) : "memory");
  }
  // ... and of this thread's first points into its slots of the ring (read back by the same thread)
  constexpr int RING = NsPlane<K>::RING, NT = NsPlane<K>::THREADS;
  const int fl = lane < C ? lane : C - 1;
  const float4* fp = reinterpret_cast<const float4*>(fqb) + (int64_t)l * 4 * C + fl;
  const float4* ring = reinterpret_cast<const float4*>(ns_smem + 2 * NsPlane<K>::BUF) + threadIdx.x;
  const unsigned ring_s = (unsigned)__cvta_generic_to_shared(ring);
  auto fetch = [&](int pt, int slot) {  // a group per point, empty past the last one
    if (pt < NL)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(ring_s + (unsigned)((slot * 4 + q) * NT * 16)),
                     "l"(fp + ((int64_t)pt * Q * 4 + q) * C)
                     : "memory");
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
#pragma unroll
  for (int pt = 0; pt < RING; ++pt) fetch(pt, pt);
  const uint32_t t = (uint32_t)blk * (uint32_t)C + (uint32_t)lane;
  const bool valid = lane < C && t < P.cells;
  const uint32_t tt = t < P.cells ? t : P.cells - 1;
  const int cx = (int)(tt % (uint32_t)n), row = (int)(tt / (uint32_t)n);
  const int cy = row % n, cz = row / n;
  const int M = K * n + 1;
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  // ---- trial side: the nodal plane l, x and y contractions in registers
  T val[4][Q][Q];  // [field][y][x]
  {
    const int iz = K * cz + l;
    const T* s = P.src + ((int64_t)(K * cx) + (int64_t)M * ((int64_t)(K * cy) + (int64_t)M * iz)) * 4;
    const bool bz = iz == 0 || iz == M - 1;
#pragma unroll
    for (int b = 0; b < Q; ++b) {
      const bool by = bz || (b == 0 && cy == 0) || (b == K && cy == n - 1);
#pragma unroll
      for (int a = 0; a < Q; ++a) {
        const bool bnd = by || (a == 0 && cx == 0) || (a == K && cx == n - 1);
        const float4 q = reinterpret_cast<const float4*>(s)[(int64_t)M * b + a];
        val[0][b][a] = bnd ? T(0) : q.x;
        val[1][b][a] = bnd ? T(0) : q.y;
        val[2][b][a] = bnd ? T(0) : q.z;
        val[3][b][a] = q.w;
      }
    }
  }
#pragma unroll
  for (int f = 0; f < 4; ++f) {
#pragma unroll
    for (int b = 0; b < Q; ++b) {
      T o[Q];
      if (f < 3) line_sym<Q, kTrial, false>(tab.S, tab.hS, val[f][b], o);
      else line_sym<Q, kTrial, true>(tab.Sp, tab.hSp, val[f][b], o);
#pragma unroll
      for (int a = 0; a < Q; ++a) val[f][b][a] = o[a];
    }
#pragma unroll
    for (int a = 0; a < Q; ++a) {
      T u[Q], o[Q];
#pragma unroll
      for (int b = 0; b < Q; ++b) u[b] = val[f][b][a];
      line_sym<Q, kTrial, false>(tab.S, tab.hS, u, o);
#pragma unroll
      for (int b = 0; b < Q; ++b) val[f][b][a] = o[b];
    }
  }
#pragma unroll
  for (int j = 0; j < Q; ++j)
#pragma unroll
    for (int i = 0; i < Q; ++i)
      ns_st(E, NL * l + i + Q * j, lane, 32, val[0][j][i], val[1][j][i], val[2][j][i], val[3][j][i]);
  __syncthreads();
  // values on the Gauss plane l
#pragma unroll
  for (int j = 0; j < Q; ++j)
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const T so = tab.S[l][l];
#pragma unroll
      for (int f = 0; f < 4; ++f) val[f][j][i] = mul_rn(so, val[f][j][i]);
#pragma unroll
      for (int c = 1; c < Q; ++c) {
        const int o = l + c < Q ? l + c : l + c - Q;
        T e[4];
        ns_ld(E, NL * o + i + Q * j, lane, 32, e);
        const T sc = tab.S[l][o];
#pragma unroll
        for (int f = 0; f < 4; ++f) val[f][j][i] = fma(sc, e[f], val[f][j][i]);
      }
    }
  // ---- pointwise terms, row by row; the test side of x and y accumulates in registers
  T acc[4][Q][Q];
#pragma unroll
  for (int f = 0; f < 4; ++f)
#pragma unroll
    for (int j = 0; j < Q; ++j)
#pragma unroll
      for (int i = 0; i < Q; ++i) acc[f][j][i] = T(0);
  constexpr bool ROLL = NsPlane<K>::ROLL;
  constexpr int UNROLL = ROLL ? 1 : Q;
#pragma unroll UNROLL
  for (int j = 0; j < Q; ++j) {
    // register row r of val and acc: row of points at(r); the current one is r = j0
    const int j0 = ROLL ? 0 : j;
    auto at = [&](int r) { return ROLL ? (j + r) % Q : r; };
    T dx[4][Q], xx[4][Q], cxr[4][Q];
#pragma unroll
    for (int f = 0; f < 3; ++f) line_deriv<Q, true>(tab.D, tab.hD, tab.D2, val[f][j0], dx[f], xx[f]);
    line_deriv<Q, false>(tab.D, tab.hD, tab.D2, val[3][j0], dx[3], xx[3]);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      T F[4][4];
      const int slot = ROLL ? i : (i + Q * j) % RING;
      asm volatile("cp.async.wait_group %0;\n" ::"n"(RING - 1) : "memory");
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 v4 = ring[(slot * 4 + q) * NT];
        F[q][0] = v4.x; F[q][1] = v4.y; F[q][2] = v4.z; F[q][3] = v4.w;
      }
      T gx[4], gy[4], gz[4], v[4], lap[3], c0[4], cxp[4], cyp[4], czp[4];
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        v[f] = val[f][j0][i];
        gx[f] = dx[f][i];
        T s = mul_rn(tab.D[j][at(0)], val[f][0][i]);
#pragma unroll
        for (int a = 1; a < Q; ++a) s = fma(tab.D[j][at(a)], val[f][a][i], s);
        gy[f] = s;
      }
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        lap[f] = Q > 2 ? xx[f][i] : T(0);
        if (Q > 2)
#pragma unroll
          for (int a = 0; a < Q; ++a) lap[f] = fma(tab.D2[j][at(a)], val[f][a][i], lap[f]);
      }
#pragma unroll
      for (int c = 0; c < Q; ++c) {
        T e[4];
        ns_ld(E, NL * c + i + Q * j, lane, 32, e);
        const T d = tab.DS[l][c], d2 = tab.D2S[l][c];
#pragma unroll
        for (int f = 0; f < 4; ++f) gz[f] = c ? fma(d, e[f], gz[f]) : mul_rn(d, e[f]);
        if (Q > 2)
#pragma unroll
          for (int f = 0; f < 3; ++f) lap[f] = fma(d2, e[f], lap[f]);
      }
      ns_point<T>(v, gx, gy, gz, lap, F, P, c0, cxp, cyp, czp);
      fetch(i + Q * j + RING, slot);  // into the slots just read
      ns_st(Z, NL * l + i + Q * j, lane, 32, czp[0], czp[1], czp[2], czp[3]);
      const T dl = tab.Dw[l][l];
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        cxr[f][i] = cxp[f];
        acc[f][j0][i] += fma(dl, czp[f], c0[f]);
#pragma unroll
        for (int a = 0; a < Q; ++a) acc[f][a][i] = fma(tab.Dw[at(a)][j], cyp[f], acc[f][a][i]);
      }
    }
#pragma unroll
    for (int f = 0; f < 4; ++f) line_dwt<Q, true>(tab.Dw, tab.hDw, cxr[f], acc[f][j0]);
    if constexpr (ROLL) {
#pragma unroll
      for (int f = 0; f < 4; ++f)
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          const T v0 = val[f][0][i], a0 = acc[f][0][i];
#pragma unroll
          for (int r = 0; r + 1 < Q; ++r) {
            val[f][r][i] = val[f][r + 1][i];
            acc[f][r][i] = acc[f][r + 1][i];
          }
          val[f][Q - 1][i] = v0;
          acc[f][Q - 1][i] = a0;
        }
    }
  }
  __syncthreads();
  // ---- test side: z derivatives of the other planes, then the transposed values y, x and z
#pragma unroll
  for (int j = 0; j < Q; ++j)
#pragma unroll
    for (int i = 0; i < Q; ++i)
#pragma unroll
      for (int c = 1; c < Q; ++c) {
        const int o = l + c < Q ? l + c : l + c - Q;
        T e[4];
        ns_ld(Z, NL * o + i + Q * j, lane, 32, e);
        const T d = tab.Dw[l][o];
#pragma unroll
        for (int f = 0; f < 4; ++f) acc[f][j][i] = fma(d, e[f], acc[f][j][i]);
      }
#pragma unroll
  for (int f = 0; f < 4; ++f) {
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      T u[Q], o[Q];
#pragma unroll
      for (int j = 0; j < Q; ++j) u[j] = acc[f][j][i];
      line_sym<Q, kTest, false>(tab.St, tab.hSt, u, o);
#pragma unroll
      for (int b = 0; b < Q; ++b) acc[f][b][i] = o[b];
    }
#pragma unroll
    for (int b = 0; b < Q; ++b) {
      T o[Q];
      line_sym<Q, kTest, true>(f < 3 ? tab.Sf : tab.Sfp, f < 3 ? tab.hSf : tab.hSfp, acc[f][b], o);
#pragma unroll
      for (int a = 0; a < Q; ++a) acc[f][b][a] = o[a];
    }
  }
#pragma unroll
  for (int b = 0; b < Q; ++b)
#pragma unroll
    for (int a = 0; a < Q; ++a)
      ns_st(E, NL * l + a + Q * b, lane, 32, acc[0][b][a], acc[1][b][a], acc[2][b][a], acc[3][b][a]);
  __syncthreads();
  const bool joined = lane > 0 && cx > 0;
  T* out = P.rows + (((int64_t)row * NL + Q * l) * M + K * cx) * 4;
#pragma unroll
  for (int b = 0; b < Q; ++b) {
    T r[4][Q];
    const T so = tab.St[l][l];
#pragma unroll
    for (int a = 0; a < Q; ++a) {
#pragma unroll
      for (int f = 0; f < 4; ++f) r[f][a] = mul_rn(so, acc[f][b][a]);
#pragma unroll
      for (int c = 1; c < Q; ++c) {
        const int o = l + c < Q ? l + c : l + c - Q;
        T e[4];
        ns_ld(E, NL * o + a + Q * b, lane, 32, e);
        const T sc = tab.St[l][o];
#pragma unroll
        for (int f = 0; f < 4; ++f) r[f][a] = fma(sc, e[f], r[f][a]);
      }
    }
    // the face between x-neighbours of the block, then the node values of the row
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const T left = __shfl_up_sync(0xffffffffu, r[f][K], 1);
      r[f][0] += joined ? left : T(0);
    }
    if (valid) {
      float4* o4 = reinterpret_cast<float4*>(out + (int64_t)b * M * 4);
#pragma unroll
      for (int a = 0; a < K; ++a) st_keep(o4 + a, r[0][a], r[1][a], r[2][a], r[3][a]);
      const float4 e = make_float4(r[0][K], r[1][K], r[2][K], r[3][K]);
      if (cx == n - 1) o4[K] = e;
      else if (lane == C - 1) *reinterpret_cast<float4*>(P.tails + ((int64_t)blk * NL + b + Q * l) * 4) = e;
    }
  }
}

// What follows a product, applied to the node's sum in registers.
enum NsAfter { kStore = 0, kUpdate = 1, kResidual = 2 };

template <typename T>
struct NsNodeArgs {
  T* dst;           // kStore: A src; kUpdate: the iterate (= src); kResidual: b - A src
  const T* src;
  const T* rows;
  const T* tails;
  const T* b;
  const T* dinv;
  T* d;
  T c1, c2;         // kUpdate: d = c1 d + c2 dinv (b - A x), x += d (c1 = 0: d is not read)
  int32_t n, C;
  uint32_t magic;   // ceil(2^32 / C)
};

// Node pass: bound by the reads of `rows` (L2-resident up to 64^3 in FP32) and the vectors.  One
// thread per node; the (at most four) rows of a node are loaded together.  (Two nodes per thread: 64^3
// FP32 product 119 -> 135 us; registers bounded for six or eight blocks a SM: 133, 140 us.)
template <typename T, int K, int AFTER>
__global__ void __launch_bounds__(256) k_ns_nodes(const NsNodeArgs<T> a) {
  constexpr int Q = K + 1, NL = Q * Q;
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const int n = a.n, M = K * n + 1;
  const uint32_t i = blockIdx.x * 256u + threadIdx.x;
  const bool in = i < (uint32_t)(M * M);
  const int iy = in ? (int)(i / (uint32_t)M) : 0, ix = in ? (int)i - iy * M : 0, iz = blockIdx.y;
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  if (!in) return;
  const int64_t node = (int64_t)i + (int64_t)M * M * iz;
  auto ld4 = [](const T* p, T (&v)[4]) {
    if constexpr (sizeof(T) == 4) {
      const float4 q = *reinterpret_cast<const float4*>(p);
      v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    } else {
      const double2 q0 = *reinterpret_cast<const double2*>(p), q1 = *reinterpret_cast<const double2*>(p + 2);
      v[0] = q0.x; v[1] = q0.y; v[2] = q1.x; v[3] = q1.y;
    }
  };
  auto st4 = [](T* p, const T (&v)[4]) {
    if constexpr (sizeof(T) == 4) {
      *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
      *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
      *reinterpret_cast<double2*>(p + 2) = make_double2(v[2], v[3]);
    }
  };
  const int qy = iy / K, ry = iy - K * qy, qz = iz / K, rz = iz - K * qz;
  const int qx = ix / K;
  const bool face_x = ix == K * qx && qx > 0 && qx < n;  // a block of the cell row may end here
  // rows (lower, lower), (upper, lower), (lower, upper), (upper, upper) in (y, z); upper: the cell row that
  // starts at or holds the node, lower: the one that ends at it.  All loads are issued before the
  // first is used.
  T v[4][4], tl[4][4];
  bool ok[4], cut[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const bool uy = k & 1, uz = k >> 1;
    const int cy = uy ? qy : qy - 1, cz = uz ? qz : qz - 1;
    ok[k] = (uy ? cy < n : (ry == 0 && cy >= 0)) && (uz ? cz < n : (rz == 0 && cz >= 0));
    cut[k] = false;
    if (ok[k]) {
      const int w = (uy ? ry : K) + Q * (uz ? rz : K);
      const int64_t row = (int64_t)cz * n + cy;
      if constexpr (sizeof(T) == 4) ld_last(a.rows + ((row * NL + w) * M + ix) * 4, v[k]);
      else ld4(a.rows + ((row * NL + w) * M + ix) * 4, v[k]);
      if (face_x) {
        const uint32_t t = (uint32_t)row * (uint32_t)n + (uint32_t)qx;
        const uint32_t blk = a.C == 1 ? t : __umulhi(t, a.magic);
        cut[k] = blk * (uint32_t)a.C == t;
        if (cut[k]) ld4(a.tails + ((int64_t)(blk - 1) * NL + w) * 4, tl[k]);
      }
    }
  }
  T sum[4];
  T x4[4], b4[4], q4[4], d4[4];
  // the source only where it is used: the iterate, or identity rows (64^3 FP32 product 123.2 -> 118.7 us)
  const bool bnd = ix == 0 || ix == M - 1 || iy == 0 || iy == M - 1 || iz == 0 || iz == M - 1;
  if (AFTER == kUpdate || bnd) ld4(a.src + node * 4, x4);
  if constexpr (AFTER != kStore) ld4(a.b + node * 4, b4);
  if constexpr (AFTER == kUpdate) {
    ld4(a.dinv + node * 4, q4);
    if (a.c1 != T(0)) ld4(a.d + node * 4, d4);
    else d4[0] = d4[1] = d4[2] = d4[3] = T(0);
  }
  bool first = true;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (!ok[k]) continue;
#pragma unroll
    for (int f = 0; f < 4; ++f) sum[f] = first ? v[k][f] : sum[f] + v[k][f];
    first = false;
    if (cut[k])
#pragma unroll
      for (int f = 0; f < 4; ++f) sum[f] += tl[k][f];
  }
  if (bnd)  // identity rows
#pragma unroll
    for (int f = 0; f < 3; ++f) sum[f] = x4[f];
  if constexpr (AFTER == kStore) {
    st4(a.dst + node * 4, sum);
  } else if constexpr (AFTER == kResidual) {
#pragma unroll
    for (int f = 0; f < 4; ++f) sum[f] = b4[f] - sum[f];
    st4(a.dst + node * 4, sum);
  } else {
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      d4[f] = smoother_direction(a.c1, a.c2, d4[f], q4[f], b4[f] - sum[f]);
      x4[f] += d4[f];
    }
    st4(a.d + node * 4, d4);
    st4(a.dst + node * 4, x4);
  }
}

}  // namespace mfns
