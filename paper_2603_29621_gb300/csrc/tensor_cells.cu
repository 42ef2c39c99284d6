// Cell products as sums of tensor products of 1D matrices, in registers (see tensor_cells.hpp).
//
// The Gauss rule of the general kernel integrates every product of two 1D basis functions exactly, so
// the cell matrix of the vector Laplacian is nu h (K x M x M + M x K x M + M x M x K) with the 1D mass
// and stiffness matrices of the reference interval, and the pressure coupling uses the mixed 1D
// matrices of the velocity and pressure bases.  Seven 1D contractions replace the twelve of
// interpolation, derivatives and their transposes.
//
// FP32, degrees 1 and 2: one thread owns one component of one cell: its (k + 1)^3 <= 27 values, the two
// intermediate fields and the hanging-node interpolation stay in registers, and nothing is exchanged but
// the sum of the three components' divergence (two shuffles per pressure value).  Three adjacent lanes
// share a cell, ten cells a warp; tables are uniform operands and index lists are stored by slot, so
// their loads are consecutive over cells.  Bound by instruction issue and the latency of the gather
// (Stokes Q2/Q1, 24^3 with two refinements, whole product against the general kernel 70 -> 30 us).
// FP64 and degrees 3 and 4: lines, below.
#include <array>
#include <atomic>
#include <cmath>
#include <type_traits>
#include <vector>

#include "common.hpp"
#include "op_kernel.cuh"
#include "tensor_cells.hpp"

namespace mfns {

template <typename T, int N, int NP>
struct TpTab {
  // 1D mass and stiffness of the velocity (or scalar) basis in even-odd form: half the sum and half the
  // difference of a row's outer entries, the centre column and the centre row (odd N)
  struct Sym {
    T e[N / 2][N / 2], o[N / 2][N / 2], col[N / 2], row[N / 2], mid;
  } M, K;
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

// Products with a matrix that is symmetric about its centre: u split into u_j +- u_{N-1-j}, the even and odd
// parts of A u + B v formed with half the products, then joined (N = 3: 55 operations instead of 63 for
// the seven contractions of a line of each direction, N = 4: 96 instead of 112).
template <int N, typename T>
struct EvenOdd {
  static constexpr int H = N / 2;
  T e[H], o[H], mid;
  __device__ __forceinline__ explicit EvenOdd(const T (&u)[N]) {
#pragma unroll
    for (int j = 0; j < H; ++j) {
      e[j] = u[j] + u[N - 1 - j];
      o[j] = u[j] - u[N - 1 - j];
    }
    mid = u[H];
  }
};
template <int N, bool TWO, typename Sym, typename T>
__device__ __forceinline__ void sym_line(const Sym& A, const EvenOdd<N, T>& u, const Sym& B, const EvenOdd<N, T>& v,
                                         T (&out)[N]) {
  constexpr int H = N / 2;
  constexpr bool ODD = N % 2 == 1;
#pragma unroll
  for (int i = 0; i < H; ++i) {
    T E = A.e[i][0] * u.e[0];
#pragma unroll
    for (int j = 1; j < H; ++j) E = fma(A.e[i][j], u.e[j], E);
    if (ODD) E = fma(A.col[i], u.mid, E);
    if (TWO) {
#pragma unroll
      for (int j = 0; j < H; ++j) E = fma(B.e[i][j], v.e[j], E);
      if (ODD) E = fma(B.col[i], v.mid, E);
    }
    if constexpr (H == 1 && !TWO) {
      out[0] = fma(A.o[0][0], u.o[0], E);
      out[N - 1] = fma(-A.o[0][0], u.o[0], E);
    } else {
      T O = A.o[i][0] * u.o[0];
#pragma unroll
      for (int j = 1; j < H; ++j) O = fma(A.o[i][j], u.o[j], O);
      if (TWO)
#pragma unroll
        for (int j = 0; j < H; ++j) O = fma(B.o[i][j], v.o[j], O);
      out[i] = E + O;
      out[N - 1 - i] = E - O;
    }
  }
  if (ODD) {
    T m = A.mid * u.mid;
#pragma unroll
    for (int j = 0; j < H; ++j) m = fma(A.row[j], u.e[j], m);
    if (TWO) {
      m = fma(B.mid, v.mid, m);
#pragma unroll
      for (int j = 0; j < H; ++j) m = fma(B.row[j], v.e[j], m);
    }
    out[H] = m;
  }
}
template <int N, typename Sym, typename T>
__device__ __forceinline__ void sym_line(const Sym& A, const EvenOdd<N, T>& u, T (&out)[N]) {
  sym_line<N, false>(A, u, A, u, out);
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
          sym_line<N>(a.tab.M, EvenOdd<N, T>(v), o);
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
      const EvenOdd<N, T> ev(v);
      sym_line<N>(a.tab.M, ev, o);
      sym_line<N>(a.tab.K, ev, o2);
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
        T v[N], z[N], o[N], o2[N];
#pragma unroll
        for (int i = 0; i < N; ++i) {
          v[i] = u[(c * N + i) * N + x];
          z[i] = w[(c * N + i) * N + x];
        }
        const EvenOdd<N, T> ev(v);
        sym_line<N>(a.tab.M, ev, o);
        sym_line<N, true>(a.tab.K, ev, a.tab.M, EvenOdd<N, T>(z), o2);
#pragma unroll
        for (int i = 0; i < N; ++i) {
          u[(c * N + i) * N + x] = o[i];
          w[(c * N + i) * N + x] = o2[i];
        }
      }
    const T sc = a.nu * h;
#pragma unroll
    for (int r = 0; r < N * N; ++r) {
      T v[N], z[N], o[N];
#pragma unroll
      for (int i = 0; i < N; ++i) {
        v[i] = u[N * N * i + r];
        z[i] = w[N * N * i + r];
      }
      sym_line<N, true>(a.tab.K, EvenOdd<N, T>(v), a.tab.M, EvenOdd<N, T>(z), o);
#pragma unroll
      for (int i = 0; i < N; ++i) u[N * N * i + r] = sc * o[i];
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

// ------------------------------------------------------------------------ FP64, degrees 3 and 4: lines
// A component's (k + 1)^3 values no longer fit a thread, or (FP64) one thread's operations take too long
// in a row: a thread owns one line of one component, and the fields go through shared memory between the
// directions, three stages and two barriers (six more in a block with hanging nodes).  FP64 products are
// bound by the number of operations (Stokes Q3/Q2 24^3 341 -> 249 us).
template <int N, int NP, int KIND, int TH>
struct TpLines {
  static constexpr int NL = N * N, NB = NL * N, NBP = NP * NP * NP, COMP = KIND == 2 ? 1 : 3;
  static constexpr int C = TH / (COMP * NL);
  // per cell: A, B [COMP][NB]; Stokes: W [3][NP N N], T1, T2 [NP NP N], P0, P1 [NP NP N], P00, P01, P10 [NP N N]
  static constexpr int oB = COMP * NB, oW = KIND == 2 ? oB : 2 * oB, oT = oW + 3 * NP * NL, oP = oT + 2 * NP * NP * N,
                       oPP = oP + 2 * NP * NP * N, CELL = KIND == 1 ? oPP + 3 * NP * NL : oW;
};

// row r of X (TR: column) times v, or of Y where `second` (a select of the coefficient: lanes of a warp differ)
template <int R, int S, bool TR, typename T, int D0, int D1>
__device__ __forceinline__ T row_dot(const T (&X)[D0][D1], int r, const T (&v)[S]) {
  T s = (TR ? X[0][r] : X[r][0]) * v[0];
#pragma unroll
  for (int j = 1; j < S; ++j) s = fma(TR ? X[j][r] : X[r][j], v[j], s);
  return s;
}
template <int R, int S, bool TR, typename T, int D0, int D1>
__device__ __forceinline__ T row_dot(const T (&X)[D0][D1], const T (&Y)[D0][D1], bool second, int r, const T (&v)[S]) {
  T s = T(0);
#pragma unroll
  for (int j = 0; j < S; ++j) {
    const T x = second ? (TR ? Y[j][r] : Y[r][j]) : (TR ? X[j][r] : X[r][j]);
    s = j ? fma(x, v[j], s) : x * v[j];
  }
  return s;
}

// interpolation of one line at a hanging face or edge (TR: transposed)
template <int N, bool TR, typename T>
__device__ __forceinline__ void hang_line(T (&v)[N], const T (&P)[2][N][N], bool hi) {
  T o[N];
#pragma unroll
  for (int a = 0; a < N; ++a) {
    T s = T(0);
#pragma unroll
    for (int b = 0; b < N; ++b) s = fma(TR ? (hi ? P[1][b][a] : P[0][b][a]) : (hi ? P[1][a][b] : P[0][a][b]), v[b], s);
    o[a] = s;
  }
#pragma unroll
  for (int a = 0; a < N; ++a) v[a] = o[a];
}
template <int N>
__device__ __forceinline__ bool line_hangs(uint32_t m, int dir, int w) {
  const int p = w % N, q = w / N;
  return dir == 0 ? LineFlags<3, N>::x(m, p, q) : dir == 1 ? LineFlags<3, N>::y(m, p, q) : LineFlags<3, N>::z(m, p, q);
}

template <int N, int NP, int KIND, int TH, typename T>
__global__ void __launch_bounds__(TH, 768 / TH) k_tensor_lines(const __grid_constant__ TpArgs<T, N, NP> a) {
  using Tl = TpLines<N, NP, KIND, TH>;
  constexpr int NL = Tl::NL, NB = Tl::NB, NPL = NP * NP, COMP = Tl::COMP, C = Tl::C, CELL = Tl::CELL;
  constexpr int OUT = defer_stride(COMP);
  extern __shared__ __align__(16) unsigned char tp_smem[];
  T* mem = reinterpret_cast<T*>(tp_smem);
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const int64_t nc = a.cells, c0 = (int64_t)blockIdx.x * C;
  const int ncell = (int)min((int64_t)C, nc - c0);
  const bool any = __syncthreads_or(threadIdx.x < (unsigned)ncell && (a.mask[c0 + threadIdx.x] & 0x3FFFFu) != 0);
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  const int vel = ncell * COMP * NL;
  auto at = [](int dir, int w, int n, int& p0, int& st) {
    p0 = dir == 0 ? n * w : dir == 1 ? w % n + n * n * (w / n) : w;
    st = dir == 0 ? 1 : dir == 1 ? n : n * n;
  };
  auto nodal = [&](int c, int f, int slot) {
    const int32_t v = a.cu[(int64_t)slot * nc + c0 + c];
    const T x = a.src[(int64_t)(v & 0x7fffffff) * COMP + f];
    return KIND != 2 && v < 0 ? T(0) : x;
  };
  auto pnodal = [&](int c, int slot) { return a.src[a.p_offset + a.cp[(int64_t)slot * nc + c0 + c]]; };
  if (any) {  // resolve the hanging nodes first: velocity into A, pressure into P00
    for (int dir = 0; dir < 3; ++dir) {
      if (dir) __syncthreads();
      for (int it = threadIdx.x; it < vel; it += TH) {
        const int c = it / (COMP * NL), f = it / NL % COMP, w = it % NL;
        const uint32_t m = a.mask[c0 + c];
        int p0, st;
        at(dir, w, N, p0, st);
        T* A = mem + c * CELL + f * NB;
        T v[N];
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] = dir ? A[p0 + st * i] : nodal(c, f, p0 + st * i);
        if (line_hangs<N>(m, dir, w)) hang_line<N, false>(v, a.tab.P, (m >> (24 + dir)) & 1u);
#pragma unroll
        for (int i = 0; i < N; ++i) A[p0 + st * i] = v[i];
      }
      if constexpr (KIND == 1)
        for (int it = threadIdx.x; it < ncell * NPL; it += TH) {
          const int c = it / NPL, w = it % NPL;
          const uint32_t m = a.mask[c0 + c];
          int p0, st;
          at(dir, w, NP, p0, st);
          T* q = mem + c * CELL + Tl::oPP;
          T v[NP];
#pragma unroll
          for (int i = 0; i < NP; ++i) v[i] = dir ? q[p0 + st * i] : pnodal(c, p0 + st * i);
          if (line_hangs<NP>(m, dir, w)) hang_line<NP, false>(v, a.tab.Pp, (m >> (24 + dir)) & 1u);
#pragma unroll
          for (int i = 0; i < NP; ++i) q[p0 + st * i] = v[i];
        }
    }
    __syncthreads();
  }
  // ---- x
  for (int it = threadIdx.x; it < vel; it += TH) {
    const int c = it / (COMP * NL), f = it / NL % COMP, w = it % NL;
    T* A = mem + c * CELL + f * NB;
    T v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = any ? A[N * w + i] : nodal(c, f, N * w + i);
    T o[N], o2[N];
    const EvenOdd<N, T> ev(v);
    sym_line<N>(a.tab.M, ev, o);
    if (KIND != 2) sym_line<N>(a.tab.K, ev, o2);
#pragma unroll
    for (int i = 0; i < N; ++i) {
      A[N * w + i] = o[i];
      if (KIND != 2) A[Tl::oB + N * w + i] = o2[i];
    }
    if constexpr (KIND == 1) {
      T* W = mem + c * CELL + Tl::oW + f * NP * NL;
#pragma unroll
      for (int m = 0; m < NP; ++m)
        W[NP * w + m] = row_dot<NP, N, true>(a.tab.Mr, a.tab.Dr, f == 0, m, v);
    }
  }
  if constexpr (KIND == 1)
    for (int it = threadIdx.x; it < ncell * NPL; it += TH) {
      const int c = it / NPL, w = it % NPL;
      T* cell = mem + c * CELL;
      T v[NP];
#pragma unroll
      for (int i = 0; i < NP; ++i) v[i] = any ? cell[Tl::oPP + NP * w + i] : pnodal(c, NP * w + i);
#pragma unroll
      for (int i = 0; i < N; ++i) {
        cell[Tl::oP + N * w + i] = row_dot<N, NP, false>(a.tab.Mr, i, v);
        cell[Tl::oP + NPL * N + N * w + i] = row_dot<N, NP, false>(a.tab.Dr, i, v);
      }
    }
  __syncthreads();
  // ---- y
  for (int it = threadIdx.x; it < vel; it += TH) {
    const int c = it / (COMP * NL), f = it / NL % COMP, w = it % NL;
    T* A = mem + c * CELL + f * NB + w % N + NL * (w / N);
    T v[N], z[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      v[i] = A[N * i];
      if (KIND != 2) z[i] = A[Tl::oB + N * i];
    }
    T o[N], o2[N];
    const EvenOdd<N, T> ev(v);
    sym_line<N>(a.tab.M, ev, o);
    if (KIND != 2) sym_line<N, true>(a.tab.K, ev, a.tab.M, EvenOdd<N, T>(z), o2);
#pragma unroll
    for (int i = 0; i < N; ++i) {
      A[N * i] = o[i];
      if (KIND != 2) A[Tl::oB + N * i] = o2[i];
    }
  }
  if constexpr (KIND == 1) {
    for (int it = threadIdx.x; it < ncell * NP * N; it += TH) {  // divergence, lines (m, z)
      const int c = it / (NP * N), w = it % (NP * N), m = w % NP, zc = w / NP;
      const T* W = mem + c * CELL + Tl::oW + zc * N * NP + m;
      T* t = mem + c * CELL + Tl::oT + zc * NPL + m;
      T v0[N], v1[N], v2[N];
#pragma unroll
      for (int i = 0; i < N; ++i) {
        v0[i] = W[NP * i];
        v1[i] = W[NP * NL + NP * i];
        v2[i] = W[2 * NP * NL + NP * i];
      }
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        t[NP * j] = row_dot<NP, N, true>(a.tab.Mr, j, v0) + row_dot<NP, N, true>(a.tab.Dr, j, v1);
        t[NPL * N + NP * j] = row_dot<NP, N, true>(a.tab.Mr, j, v2);
      }
    }
    for (int it = threadIdx.x; it < ncell * N * NP; it += TH) {  // pressure, lines (x, k)
      const int c = it / (N * NP), w = it % (N * NP), x = w % N, kz = w / N;
      const T* q = mem + c * CELL + Tl::oP + kz * NP * N + x;
      T* o = mem + c * CELL + Tl::oPP + kz * NL + x;
      T v0[NP], v1[NP];
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        v0[j] = q[N * j];
        v1[j] = q[NPL * N + N * j];
      }
#pragma unroll
      for (int b = 0; b < N; ++b) {
        o[N * b] = row_dot<N, NP, false>(a.tab.Mr, b, v0);
        o[NP * NL + N * b] = row_dot<N, NP, false>(a.tab.Dr, b, v0);
        o[2 * NP * NL + N * b] = row_dot<N, NP, false>(a.tab.Mr, b, v1);
      }
    }
  }
  __syncthreads();
  // ---- z, and the output where nothing hangs
  for (int it = threadIdx.x; it < vel; it += TH) {
    const int c = it / (COMP * NL), f = it / NL % COMP, w = it % NL;
    T* A = mem + c * CELL + f * NB + w;
    const T h = a.h[c0 + c];
    T v[N], z[N], g[NP], o[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      v[i] = A[NL * i];
      if (KIND != 2) z[i] = A[Tl::oB + NL * i];
    }
    if constexpr (KIND == 1) {  // P10, P01, P00 for the three components
      const T* pp = mem + c * CELL + Tl::oPP + (2 - f) * NP * NL + w;
#pragma unroll
      for (int k = 0; k < NP; ++k) g[k] = pp[NL * k];
    }
    if constexpr (KIND == 2) sym_line<N>(a.tab.M, EvenOdd<N, T>(v), o);
    else sym_line<N, true>(a.tab.K, EvenOdd<N, T>(v), a.tab.M, EvenOdd<N, T>(z), o);
    const T sc = KIND == 2 ? h * h * h : a.nu * h, sp = -h * h;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      o[i] *= sc;
      if constexpr (KIND == 1) o[i] = fma(sp, row_dot<N, NP, false>(a.tab.Mr, a.tab.Dr, f == 2, i, g), o[i]);
    }
    if (any) {
      const uint32_t m = a.mask[c0 + c];
      if (line_hangs<N>(m, 2, w)) hang_line<N, true>(o, a.tab.P, (m >> 26) & 1u);
#pragma unroll
      for (int i = 0; i < N; ++i) A[NL * i] = o[i];
    } else {
#pragma unroll
      for (int i = 0; i < N; ++i) a.buf[((int64_t)(w + NL * i) * nc + c0 + c) * OUT + f] = o[i];
    }
  }
  if constexpr (KIND == 1)
    for (int it = threadIdx.x; it < ncell * NPL; it += TH) {
      const int c = it / NPL, w = it % NPL;
      const T* t = mem + c * CELL + Tl::oT + w;
      const T h = a.h[c0 + c];
      T v0[N], v1[N], o[NP];
#pragma unroll
      for (int i = 0; i < N; ++i) {
        v0[i] = t[NPL * i];
        v1[i] = t[NPL * N + NPL * i];
      }
#pragma unroll
      for (int k = 0; k < NP; ++k)
        o[k] = a.div_sign * h * h * (row_dot<NP, N, true>(a.tab.Mr, k, v0) + row_dot<NP, N, true>(a.tab.Dr, k, v1));
      if (any) {
        const uint32_t m = a.mask[c0 + c];
        if (line_hangs<NP>(m, 2, w)) hang_line<NP, true>(o, a.tab.Pp, (m >> 26) & 1u);
        T* q = mem + c * CELL + Tl::oW + w;
#pragma unroll
        for (int k = 0; k < NP; ++k) q[NPL * k] = o[k];
      } else {
#pragma unroll
        for (int k = 0; k < NP; ++k) a.buf_p[(int64_t)(w + NPL * k) * nc + c0 + c] = o[k];
      }
    }
  if (!any) return;
  for (int dir = 1; dir >= 0; --dir) {  // the remaining transposed interpolations, then the output
    __syncthreads();
    for (int it = threadIdx.x; it < vel; it += TH) {
      const int c = it / (COMP * NL), f = it / NL % COMP, w = it % NL;
      const uint32_t m = a.mask[c0 + c];
      int p0, st;
      at(dir, w, N, p0, st);
      T* A = mem + c * CELL + f * NB;
      T v[N];
#pragma unroll
      for (int i = 0; i < N; ++i) v[i] = A[p0 + st * i];
      if (line_hangs<N>(m, dir, w)) hang_line<N, true>(v, a.tab.P, (m >> (24 + dir)) & 1u);
#pragma unroll
      for (int i = 0; i < N; ++i) {
        if (dir) A[p0 + st * i] = v[i];
        else a.buf[((int64_t)(p0 + st * i) * nc + c0 + c) * OUT + f] = v[i];
      }
    }
    if constexpr (KIND == 1)
      for (int it = threadIdx.x; it < ncell * NPL; it += TH) {
        const int c = it / NPL, w = it % NPL;
        const uint32_t m = a.mask[c0 + c];
        int p0, st;
        at(dir, w, NP, p0, st);
        T* q = mem + c * CELL + Tl::oW;
        T v[NP];
#pragma unroll
        for (int i = 0; i < NP; ++i) v[i] = q[p0 + st * i];
        if (line_hangs<NP>(m, dir, w)) hang_line<NP, true>(v, a.tab.Pp, (m >> (24 + dir)) & 1u);
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          if (dir) q[p0 + st * i] = v[i];
          else a.buf_p[(int64_t)(p0 + st * i) * nc + c0 + c] = v[i];
        }
      }
  }
}

// ------------------------------------------------------------------------------------------ host
bool tensor_cells(const OpLaunch& L) {
  return L.dim == 3 && ((L.op == OP_STOKES_A && L.k <= 4) || (L.op == OP_PMASS && L.k <= 3) ||
                        (L.op == OP_STOKES && L.k >= 2 && L.k <= 4));
}

// 1D integrals on the reference interval of the bases of degree k (a) and k - 1 (p) on their
// Gauss--Lobatto nodes, exact in extended precision: polynomials in t = 2 x - 1.  Every product of three
// tables then carries their roundings alone; formed by a Gauss sum in FP64, the tables were off by up
// to 9e-15 and the products' error by 1.1 to 1.8 times that of quadrature (Q2 vector Laplacian FP64,
// 5^3 cells: quadrature 3.7e-16, Gauss-sum tables 6.6e-16, these 1.3e-16).
struct Integrals {
  long double m[5][5], k[5][5], mr[5][5], dr[5][5];  // a a, a' a', a p, a' p
};
using Poly = std::vector<long double>;
static std::vector<Poly> lobatto_basis(int k) {
  const long double c = k == 3 ? 1 / sqrtl(5.0L) : sqrtl(3.0L / 7.0L);
  const std::vector<long double> t = k == 0   ? std::vector<long double>{0}
                                     : k == 1 ? std::vector<long double>{-1, 1}
                                     : k == 2 ? std::vector<long double>{-1, 0, 1}
                                     : k == 3 ? std::vector<long double>{-1, -c, c, 1}
                                              : std::vector<long double>{-1, -c, 0, c, 1};
  std::vector<Poly> out;
  for (int a = 0; a <= k; ++a) {
    Poly p{1};
    for (int m = 0; m <= k; ++m) {
      if (m == a) continue;
      p.push_back(0);
      for (size_t i = p.size(); i-- > 0;) p[i] = ((i ? p[i - 1] : 0) - t[m] * p[i]) / (t[a] - t[m]);
    }
    out.push_back(p);
  }
  return out;
}
static const Integrals& integrals(int k) {
  static const std::array<Integrals, 5> all = [] {
    std::array<Integrals, 5> r{};
    auto derivative = [](const Poly& p) {  // with respect to x
      Poly d;
      for (size_t i = 1; i < p.size(); ++i) d.push_back(2 * (long double)i * p[i]);
      return d;
    };
    auto integral = [](const Poly& p, const Poly& q) {
      long double v = 0;
      for (size_t i = 0; i < p.size(); ++i)
        for (size_t j = i % 2; j < q.size(); j += 2) v += p[i] * q[j] / (long double)(i + j + 1);
      return v;
    };
    for (int k = 1; k <= 4; ++k) {
      const std::vector<Poly> a = lobatto_basis(k), p = lobatto_basis(k - 1);
      for (int i = 0; i <= k; ++i) {
        for (int j = 0; j <= k; ++j) {
          r[k].m[i][j] = integral(a[i], a[j]);
          r[k].k[i][j] = integral(derivative(a[i]), derivative(a[j]));
        }
        for (int j = 0; j < k; ++j) {
          r[k].mr[i][j] = integral(a[i], p[j]);
          r[k].dr[i][j] = integral(derivative(a[i]), p[j]);
        }
      }
    }
    return r;
  }();
  return all[k];
}

// the tables of a kernel, but for the hanging-node interpolation
template <int N, int NP, int KIND, typename T>
static TpTab<T, N, NP> make_tables() {
  TpTab<T, N, NP> tab{};
  const Integrals& I = integrals(N - 1);
  auto fold = [](const long double (&x)[5][5], auto& t) {
    constexpr int H = N / 2;
    for (int i = 0; i < H; ++i) {
      for (int j = 0; j < H; ++j) {
        t.e[i][j] = (T)(0.5L * (x[i][j] + x[i][N - 1 - j]));
        t.o[i][j] = (T)(0.5L * (x[i][j] - x[i][N - 1 - j]));
      }
      t.col[i] = (T)x[i][H];
      t.row[i] = (T)x[H][i];
    }
    t.mid = (T)x[H][H];
  };
  fold(I.m, tab.M);
  fold(I.k, tab.K);
  if (KIND == 1)
    for (int i = 0; i < N; ++i)
      for (int m = 0; m < NP; ++m) {
        tab.Mr[i][m] = (T)I.mr[i][m];
        tab.Dr[i][m] = (T)I.dr[i][m];
      }
  return tab;
}

template <int N, int NP, int KIND, typename T>
static void launch(const OpLaunch& L, const NodeGather& g, int prec, const void* src, cudaStream_t s) {
  // (formed once: extended precision is software on Arm, 1 to 2 us of a call's 11)
  static const TpTab<T, N, NP> tables = make_tables<N, NP, KIND, T>();
  TpArgs<T, N, NP> a{};
  a.tab = tables;
  for (int hf = 0; hf < 2; ++hf)
    for (int i = 0; i < N; ++i)
      for (int j = 0; j < N; ++j) a.tab.P[hf][i][j] = (T)L.P[(hf * N + i) * N + j];
  if (KIND == 1)
    for (int hf = 0; hf < 2; ++hf)
      for (int i = 0; i < NP; ++i)
        for (int m = 0; m < NP; ++m) a.tab.Pp[hf][i][m] = (T)L.Pp[(hf * NP + i) * NP + m];
  a.src = static_cast<const T*>(src);
  a.buf = static_cast<T*>(g.scratch->get());
  a.buf_p = a.buf + g.main_values();
  a.cu = g.cell_u.as<int32_t>();
  a.cp = g.cell_p.as<int32_t>();
  a.mask = g.cell_mask.as<uint32_t>();
  a.h = g.cell_h[prec].as<T>();
  a.cells = (int32_t)L.n_cells;
  a.p_offset = L.p_offset;
  a.nu = (T)L.nu;
  a.div_sign = (T)L.div_sign;
  const bool timed = L.timer && L.timer->enabled;
  if (timed) L.timer->record_pair_begin(s);
  cudaLaunchConfig_t cfg = {};
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  // (FP64 starts on an idle chip, see ns_lines.cu)
  if (sizeof(T) == 8) cfg.numAttrs = 0;
  auto lines = [&](auto th) {
    constexpr int TH = decltype(th)::value;
    using Tl = TpLines<N, NP, KIND, TH>;
    constexpr size_t smem = (size_t)Tl::C * Tl::CELL * sizeof(T);
    if (smem > 48 * 1024) {
      static std::atomic<uint64_t> done{0};  // per device
      int dev = 0;
      MFNS_CUDA(cudaGetDevice(&dev));
      const uint64_t bit = 1ull << (dev & 63);
      if (!(done.load() & bit)) {
        MFNS_CUDA(cudaFuncSetAttribute(k_tensor_lines<N, NP, KIND, TH, T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem));
        done.fetch_or(bit);
      }
    }
    cfg.gridDim = dim3((unsigned)((L.n_cells + Tl::C - 1) / Tl::C));
    cfg.blockDim = dim3(TH);
    cfg.dynamicSmemBytes = smem;
    MFNS_CUDA(cudaLaunchKernelEx(&cfg, k_tensor_lines<N, NP, KIND, TH, T>, a));
  };
  if constexpr (N > 3) {
    lines(std::integral_constant<int, 256>());
  } else if constexpr (sizeof(T) == 8) {
    // FP64: a warp's operations take 64 cycles each, so a cell's lines go to many lanes (Q2 Stokes in registers
    // 37 us from 4^3 to 16^3 cells, lines 14 to 31 us); the smaller blocks spread further, the larger
    // ones waste fewer lanes and are the better ones from two a SM on (Q2 48^3 379 against 421 us)
    if (KIND != 2 && L.n_cells >= 2 * 152 * (256 / (3 * N * N))) lines(std::integral_constant<int, 256>());
    else lines(std::integral_constant<int, 128>());
  } else {
    constexpr int per_block = 4 * (KIND == 2 ? 32 : 10);
    cfg.gridDim = dim3((unsigned)((L.n_cells + per_block - 1) / per_block));
    cfg.blockDim = dim3(128);
    MFNS_CUDA(cudaLaunchKernelEx(&cfg, k_tensor_cells<N, NP, KIND, T>, a));
  }
  if (timed) L.timer->record_pair_end(s);
}

void tensor_product(const OpLaunch& L, const NodeGather& g, int prec, const void* src, cudaStream_t s) {
#define CASE(OP, K, NP, KIND)                                           \
  if (L.op == OP && L.k == K) {                                         \
    if (prec == 0) return launch<K + 1, NP, KIND, double>(L, g, prec, src, s); \
    return launch<K + 1, NP, KIND, float>(L, g, prec, src, s);          \
  }
  CASE(OP_STOKES_A, 1, 1, 0) CASE(OP_STOKES_A, 2, 1, 0) CASE(OP_PMASS, 1, 1, 2) CASE(OP_PMASS, 2, 1, 2)
  CASE(OP_STOKES_A, 3, 1, 0) CASE(OP_STOKES_A, 4, 1, 0) CASE(OP_PMASS, 3, 1, 2)
  CASE(OP_STOKES, 2, 2, 1) CASE(OP_STOKES, 3, 3, 1) CASE(OP_STOKES, 4, 4, 1)
#undef CASE
  throw Error(kErrUnsupported, "tensor-product cells: operator or degree");
}

}  // namespace mfns
