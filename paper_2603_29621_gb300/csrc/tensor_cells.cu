// Cell products as sums of tensor products of 1D matrices, in registers (see tensor_cells.hpp).
//
// The Gauss rule of the general kernel integrates every product of two 1D basis functions exactly, so
// the cell matrix of the vector Laplacian is nu h (K x M x M + M x K x M + M x M x K) with the 1D mass
// and stiffness matrices of the reference interval, and the pressure coupling uses the mixed 1D
// matrices of the velocity and pressure bases.  Seven 1D contractions replace the twelve of
// interpolation, derivatives and their transposes.
//
// One thread owns one component of one cell: its (k + 1)^3 <= 27 values, the two intermediate fields
// and the hanging-node interpolation stay in registers, and nothing is exchanged but the sum of the
// three components' divergence (two shuffles per pressure value).  Three adjacent lanes share a cell,
// ten cells a warp; tables are uniform operands and index lists are stored by slot, so their loads are
// consecutive over cells.  Bound by instruction issue and the latency of the gather.
#include "common.hpp"
#include "op_kernel.cuh"
#include "tensor_cells.hpp"

namespace mfns {

template <typename T, int N, int NP>
struct TpTab {
  T M[N][N], K[N][N];    // 1D mass and stiffness, velocity (or the scalar) basis
  T Mr[N][NP], Dr[N][NP];  // int phi_a psi_m, int phi_a' psi_m
  T P[2][N][N], Pp[2][NP][NP];  // hanging-node interpolation to child half h
};

template <typename T, int N, int NP>
struct TpArgs {
  TpTab<T, N, NP> tab;
  const T* src;
  T *buf, *buf_p;
  const int32_t *cu, *cp;   // node per (slot, cell); bit 31: Dirichlet velocity
  const uint32_t* mask;
  const T* h;
  int32_t cells;
  int64_t p_offset;
  T nu, div_sign;
};

// o = A u for a matrix that is symmetric about its centre
template <int N, typename T>
__device__ __forceinline__ void sym_line(const T (&A)[N][N], const T (&u)[N], T (&o)[N]) {
#pragma unroll
  for (int i = 0; i < N; ++i) {
    T s = A[i][0] * u[0];
#pragma unroll
    for (int j = 1; j < N; ++j) s = fma(A[i][j], u[j], s);
    o[i] = s;
  }
}

// constraint pass along direction D of one component (TR: transposed)
template <int N, int D, bool TR, typename T>
__device__ __forceinline__ void hang_pass(T (&u)[N * N * N], uint32_t m, const T (&P)[2][N][N]) {
  const bool hi = (m >> (24 + D)) & 1u;
  T W[N][N];
#pragma unroll
  for (int r = 0; r < N; ++r)
#pragma unroll
    for (int c = 0; c < N; ++c) W[r][c] = TR ? (hi ? P[1][c][r] : P[0][c][r]) : (hi ? P[1][r][c] : P[0][r][c]);
  constexpr int st = D == 0 ? 1 : D == 1 ? N : N * N;
#pragma unroll
  for (int q = 0; q < N; ++q)
#pragma unroll
    for (int p = 0; p < N; ++p) {
      // line (p, q): the other two coordinates in ascending order of direction
      const bool f = D == 0 ? LineFlags<3, N>::x(m, p, q) : D == 1 ? LineFlags<3, N>::y(m, p, q)
                                                                  : LineFlags<3, N>::z(m, p, q);
      const int p0 = D == 0 ? N * (p + N * q) : D == 1 ? p + N * N * q : p + N * q;
      if (f) {
        T v[N];
#pragma unroll
        for (int a = 0; a < N; ++a) v[a] = u[p0 + st * a];
#pragma unroll
        for (int a = 0; a < N; ++a) {
          T s = W[a][0] * v[0];
#pragma unroll
          for (int b = 1; b < N; ++b) s = fma(W[a][b], v[b], s);
          u[p0 + st * a] = s;
        }
      }
    }
}

// KIND 0: vector Laplacian, 1: Stokes, 2: scalar mass
template <int N, int NP, int KIND, typename T>
__global__ void __launch_bounds__(128) k_tensor_cells(const __grid_constant__ TpArgs<T, N, NP> a) {
  constexpr int NB = N * N * N, NBP = NP * NP * NP, COMP = KIND == 2 ? 1 : 3, CW = KIND == 2 ? 32 : 10;
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int sub = COMP == 3 ? lane / 3 : lane, f = COMP == 3 ? lane - 3 * sub : 0;
  const int64_t c0 = ((int64_t)blockIdx.x * 4 + warp) * CW + sub;
  const bool valid = sub < CW && c0 < a.cells;
  const int32_t cell = valid ? (int32_t)c0 : 0;
  const int64_t nc = a.cells;
  const uint32_t m = a.mask[cell];
  const T h = a.h[cell];
  const bool hang = (m & 0x3FFFFu) != 0;
  int32_t id[NB];
#pragma unroll
  for (int s = 0; s < NB; ++s) id[s] = a.cu[s * nc + cell];
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  T u[NB];
#pragma unroll
  for (int s = 0; s < NB; ++s) {
    const T v = a.src[(int64_t)(id[s] & 0x7fffffff) * COMP + f];
    u[s] = KIND != 2 && id[s] < 0 ? T(0) : v;
  }
  if (hang) {
    hang_pass<N, 0, false>(u, m, a.tab.P);
    hang_pass<N, 1, false>(u, m, a.tab.P);
    hang_pass<N, 2, false>(u, m, a.tab.P);
  }
  // the 1D matrix of the component's direction is the derivative one in the coupling terms
  [[maybe_unused]] T q[NBP];
  if constexpr (KIND == 1) {
    // divergence: q = X^T Y^T Z^T u, summed over the components
    T w1[NP * N * N], w2[NP * NP * N];
#pragma unroll
    for (int c = 0; c < N; ++c)
#pragma unroll
      for (int b = 0; b < N; ++b)
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          T s = T(0);
#pragma unroll
          for (int x = 0; x < N; ++x) s = fma(f == 0 ? a.tab.Dr[x][i] : a.tab.Mr[x][i], u[(c * N + b) * N + x], s);
          w1[(c * N + b) * NP + i] = s;
        }
#pragma unroll
    for (int c = 0; c < N; ++c)
#pragma unroll
      for (int j = 0; j < NP; ++j)
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          T s = T(0);
#pragma unroll
          for (int b = 0; b < N; ++b) s = fma(f == 1 ? a.tab.Dr[b][j] : a.tab.Mr[b][j], w1[(c * N + b) * NP + i], s);
          w2[(c * NP + j) * NP + i] = s;
        }
#pragma unroll
    for (int k = 0; k < NP; ++k)
#pragma unroll
      for (int j = 0; j < NP; ++j)
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          T s = T(0);
#pragma unroll
          for (int c = 0; c < N; ++c) s = fma(f == 2 ? a.tab.Dr[c][k] : a.tab.Mr[c][k], w2[(c * NP + j) * NP + i], s);
          s *= a.div_sign * h * h;
          s += __shfl_sync(0xffffffffu, s, lane - f + (f + 1) % 3) + __shfl_sync(0xffffffffu, s, lane - f + (f + 2) % 3);
          q[(k * NP + j) * NP + i] = s;
        }
  }
  if constexpr (KIND == 2) {
    const T h3 = h * h * h;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int st = d == 0 ? 1 : d == 1 ? N : N * N;
#pragma unroll
      for (int r = 0; r < N; ++r)
#pragma unroll
        for (int p = 0; p < N; ++p) {
          const int p0 = d == 0 ? N * (p + N * r) : d == 1 ? p + N * N * r : p + N * r;
          T v[N], o[N];
#pragma unroll
          for (int i = 0; i < N; ++i) v[i] = u[p0 + st * i];
          sym_line<N>(a.tab.M, v, o);
#pragma unroll
          for (int i = 0; i < N; ++i) u[p0 + st * i] = d == 2 ? h3 * o[i] : o[i];
        }
    }
  } else {
    T w[NB];  // u: M along the directions done so far; w: their sum with K along one of them
#pragma unroll
    for (int r = 0; r < N * N; ++r) {
      T v[N], o[N], o2[N];
#pragma unroll
      for (int i = 0; i < N; ++i) v[i] = u[N * r + i];
      sym_line<N>(a.tab.M, v, o);
      sym_line<N>(a.tab.K, v, o2);
#pragma unroll
      for (int i = 0; i < N; ++i) {
        u[N * r + i] = o[i];
        w[N * r + i] = o2[i];
      }
    }
#pragma unroll
    for (int c = 0; c < N; ++c)
#pragma unroll
      for (int x = 0; x < N; ++x) {
        T v[N], z[N], o[N], o2[N], o3[N];
#pragma unroll
        for (int i = 0; i < N; ++i) {
          v[i] = u[(c * N + i) * N + x];
          z[i] = w[(c * N + i) * N + x];
        }
        sym_line<N>(a.tab.M, v, o);
        sym_line<N>(a.tab.K, v, o2);
        sym_line<N>(a.tab.M, z, o3);
#pragma unroll
        for (int i = 0; i < N; ++i) {
          u[(c * N + i) * N + x] = o[i];
          w[(c * N + i) * N + x] = o2[i] + o3[i];
        }
      }
    const T sc = a.nu * h;
#pragma unroll
    for (int r = 0; r < N * N; ++r) {
      T v[N], z[N], o[N], o2[N];
#pragma unroll
      for (int i = 0; i < N; ++i) {
        v[i] = u[N * N * i + r];
        z[i] = w[N * N * i + r];
      }
      sym_line<N>(a.tab.K, v, o);
      sym_line<N>(a.tab.M, z, o2);
#pragma unroll
      for (int i = 0; i < N; ++i) u[N * N * i + r] = sc * (o[i] + o2[i]);
    }
  }
  if constexpr (KIND == 1) {
    // pressure gradient: u -= h^2 X Y Z p
    T p[NBP];
#pragma unroll
    for (int s = 0; s < NBP; ++s) p[s] = a.src[a.p_offset + a.cp[s * nc + cell]];
    if (hang) {
      hang_pass<NP, 0, false>(p, m, a.tab.Pp);
      hang_pass<NP, 1, false>(p, m, a.tab.Pp);
      hang_pass<NP, 2, false>(p, m, a.tab.Pp);
    }
    const T sp = -h * h;
    T w1[NP * NP * N], w2[NP * N * N];
#pragma unroll
    for (int r = 0; r < NP * NP; ++r)
#pragma unroll
      for (int x = 0; x < N; ++x) {
        T s = T(0);
#pragma unroll
        for (int i = 0; i < NP; ++i) s = fma(f == 0 ? a.tab.Dr[x][i] : a.tab.Mr[x][i], p[r * NP + i], s);
        w1[r * N + x] = sp * s;
      }
#pragma unroll
    for (int k = 0; k < NP; ++k)
#pragma unroll
      for (int b = 0; b < N; ++b)
#pragma unroll
        for (int x = 0; x < N; ++x) {
          T s = T(0);
#pragma unroll
          for (int j = 0; j < NP; ++j) s = fma(f == 1 ? a.tab.Dr[b][j] : a.tab.Mr[b][j], w1[(k * NP + j) * N + x], s);
          w2[(k * N + b) * N + x] = s;
        }
#pragma unroll
    for (int c = 0; c < N; ++c)
#pragma unroll
      for (int r = 0; r < N * N; ++r) {
        T s = u[c * N * N + r];
#pragma unroll
        for (int k = 0; k < NP; ++k) s = fma(f == 2 ? a.tab.Dr[c][k] : a.tab.Mr[c][k], w2[k * N * N + r], s);
        u[c * N * N + r] = s;
      }
  }
  if (hang) {
    hang_pass<N, 2, true>(u, m, a.tab.P);
    hang_pass<N, 1, true>(u, m, a.tab.P);
    hang_pass<N, 0, true>(u, m, a.tab.P);
  }
  if (!valid) return;
#pragma unroll
  for (int s = 0; s < NB; ++s) a.buf[(s * nc + cell) * defer_stride(COMP) + f] = u[s];
  if constexpr (KIND == 1) {
    if (f == 0) {
      if (hang) {
        hang_pass<NP, 2, true>(q, m, a.tab.Pp);
        hang_pass<NP, 1, true>(q, m, a.tab.Pp);
        hang_pass<NP, 0, true>(q, m, a.tab.Pp);
      }
#pragma unroll
      for (int s = 0; s < NBP; ++s) a.buf_p[s * nc + cell] = q[s];
    }
  }
}

// ------------------------------------------------------------------------------------------ host
bool tensor_cells(const OpLaunch& L) {
  return L.dim == 3 && ((L.op == OP_STOKES_A && L.k <= 2) || (L.op == OP_PMASS && L.k <= 2) ||
                        (L.op == OP_STOKES && L.k == 2));
}

template <int N, int NP, int KIND, typename T>
static void launch(const OpLaunch& L, const NodeGather& g, int prec, const void* src, cudaStream_t s) {
  TpArgs<T, N, NP> a{};
  // 1D integrals on the reference interval by the level's Gauss rule (exact)
  auto integral = [&](auto f) {
    double v = 0.0;
    for (int q = 0; q < L.Q; ++q) v += L.W[q] * f(q);
    return v;
  };
  auto S = [&](int q, int i) { return L.S[q * N + i]; };
  auto dS = [&](int q, int i) {
    double v = 0.0;
    for (int r = 0; r < L.Q; ++r) v += L.D[q * L.Q + r] * L.S[r * N + i];
    return v;
  };
  for (int i = 0; i < N; ++i)
    for (int j = 0; j < N; ++j) {
      a.tab.M[i][j] = (T)integral([&](int q) { return S(q, i) * S(q, j); });
      a.tab.K[i][j] = (T)integral([&](int q) { return dS(q, i) * dS(q, j); });
      for (int hf = 0; hf < 2; ++hf) a.tab.P[hf][i][j] = (T)L.P[(hf * N + i) * N + j];
    }
  if (KIND == 1)
    for (int i = 0; i < N; ++i)
      for (int m = 0; m < NP; ++m) {
        a.tab.Mr[i][m] = (T)integral([&](int q) { return S(q, i) * L.Sp[q * NP + m]; });
        a.tab.Dr[i][m] = (T)integral([&](int q) { return dS(q, i) * L.Sp[q * NP + m]; });
      }
  if (KIND == 1)
    for (int hf = 0; hf < 2; ++hf)
      for (int i = 0; i < NP; ++i)
        for (int m = 0; m < NP; ++m) a.tab.Pp[hf][i][m] = (T)L.Pp[(hf * NP + i) * NP + m];
  a.src = static_cast<const T*>(src);
  a.buf = g.buf[prec].as<T>();
  a.buf_p = a.buf + g.main_values();
  a.cu = g.cell_u.as<int32_t>();
  a.cp = g.cell_p.as<int32_t>();
  a.mask = g.cell_mask.as<uint32_t>();
  a.h = g.cell_h[prec].as<T>();
  a.cells = (int32_t)L.n_cells;
  a.p_offset = L.p_offset;
  a.nu = (T)L.nu;
  a.div_sign = (T)L.div_sign;
  constexpr int per_block = 4 * (KIND == 2 ? 32 : 10);
  const bool timed = L.timer && L.timer->enabled;
  if (timed) L.timer->record_pair_begin(s);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((L.n_cells + per_block - 1) / per_block));
  cfg.blockDim = dim3(128);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  MFNS_CUDA(cudaLaunchKernelEx(&cfg, k_tensor_cells<N, NP, KIND, T>, a));
  if (timed) L.timer->record_pair_end(s);
}

void tensor_product(const OpLaunch& L, const NodeGather& g, int prec, const void* src, cudaStream_t s) {
#define CASE(OP, K, NP, KIND)                                           \
  if (L.op == OP && L.k == K) {                                         \
    if (prec == 0) return launch<K + 1, NP, KIND, double>(L, g, prec, src, s); \
    return launch<K + 1, NP, KIND, float>(L, g, prec, src, s);          \
  }
  CASE(OP_STOKES_A, 1, 1, 0) CASE(OP_STOKES_A, 2, 1, 0) CASE(OP_PMASS, 1, 1, 2) CASE(OP_PMASS, 2, 1, 2)
  CASE(OP_STOKES, 2, 2, 1)
#undef CASE
  throw Error(kErrUnsupported, "tensor-product cells: operator or degree");
}

}  // namespace mfns
