// Diagonal of the stabilised operator on uniform 3D levels, from the stored point values.
//
// For one basis function phi the pointwise Jacobian (ns_point) collapses to
//   w (A + B (cm + G_ii) + a_i phi d_i phi)  for velocity component i,   w h tau |grad phi|^2  for the pressure,
//   A = nu/h^2 |grad phi|^2 + phi c + cs tau (U grad phi) (c + lap),  B = phi (phi + cs tau U grad phi),
// with c = cc (U grad phi): all four entries of a node at a Gauss point in some forty operations, where one
// product per local unit vector spends the operations of a whole cell (4,600 for Q2) on each entry.
// A thread sums the points of the at most two cells of a cell row that share a row entry (the row
// buffer of the product, tails unused), then one thread per node adds the at most four rows.
// No colours, no additions in memory.  Whole diagonal, against colour launches of unit-vector passes:
// FP64 Q2 30^3 49.6 -> 2.2 ms, Q3 6^3 2.2 -> 0.20 ms; setting a new state of a Q2 30^3 FP32 hierarchy (point
// values, diagonals, coarse inverse) 3.4 -> 1.05 ms.  Bound by the FP64 operations; FP32 by the loads of the
// point values, which the threads of a cell share in the L1.
#include "common.hpp"
#include "ns_lines.hpp"
#include "opkind.hpp"
#include "ns_lines.cuh"

namespace mfns {

template <typename T, int Q>
struct NsDiagArgs {
  T S[Q][Q], DS[Q][Q], D2S[Q][Q];  // [point][node]: value, derivative, second derivative (times -nu / h^2)
  T W[Q];
  const T* fq;
  T* rows;
  int32_t n, C;
  T cmm, nuh2, cfc, cfs, h3, hp;  // hp: h with the PSPG term, else 0
};

template <int K, typename T>
__global__ void __launch_bounds__(128) k_ns_diag(const __grid_constant__ NsDiagArgs<T, K + 1> a) {
  constexpr int Q = K + 1, NL = Q * Q;
  __shared__ T tS[Q][Q], tD[Q][Q], tL[Q][Q];
  if (threadIdx.x < NL) {
    const int l = threadIdx.x / Q, m = threadIdx.x % Q;
    tS[l][m] = a.S[l][m];
    tD[l][m] = a.DS[l][m];
    tL[l][m] = a.D2S[l][m];
  }
  __syncthreads();
  const int n = a.n, M = K * n + 1;
  const int e = blockIdx.x * 128 + threadIdx.x, w = e / M, ix = e - w * M;
  if (w >= NL) return;
  const int b = w % Q, c = w / Q, q0 = ix / K;
  T sy[Q], dy[Q], ly[Q];
#pragma unroll
  for (int l = 0; l < Q; ++l) {
    sy[l] = tS[l][b];
    dy[l] = tD[l][b];
    ly[l] = tL[l][b];
  }
  T d[4] = {T(0), T(0), T(0), T(0)};
  const int first = ix - K * q0 == 0 && q0 > 0 ? q0 - 1 : q0, last = q0 < n ? q0 : n - 1;
  for (int cx = first; cx <= last; ++cx) {
    const int ax = ix - K * cx;
    T sx[Q], dx[Q], lx[Q];
#pragma unroll
    for (int l = 0; l < Q; ++l) {
      sx[l] = tS[l][ax];
      dx[l] = tD[l][ax];
      lx[l] = tL[l][ax];
    }
    const int64_t cell = cx + (int64_t)n * (blockIdx.y + (int64_t)n * blockIdx.z), blk = cell / a.C;
    const int slot = (int)(cell - blk * a.C);
#pragma unroll 1
    for (int z = 0; z < Q; ++z) {
      const T sz = tS[z][c], dz = tD[z][c], lz = tL[z][c];
#pragma unroll
      for (int y = 0; y < Q; ++y) {
        const T s = sy[y] * sz, gy = dy[y] * sz, gz = sy[y] * dz, lap = fma(ly[y], sz, sy[y] * lz), wyz = a.W[y] * a.W[z];
#pragma unroll
        for (int x = 0; x < Q; ++x) {
          T F[4][4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if constexpr (sizeof(T) == 4) {
              const float4 v = *reinterpret_cast<const float4*>(a.fq + ns_fq_at<T, Q>(blk, x + Q * y, z, q, 0, slot, a.C));
              F[q][0] = v.x, F[q][1] = v.y, F[q][2] = v.z, F[q][3] = v.w;
            } else {
#pragma unroll
              for (int hf = 0; hf < 2; ++hf) {
                const double2 v =
                    *reinterpret_cast<const double2*>(a.fq + ns_fq_at<T, Q>(blk, x + Q * y, z, q, hf, slot, a.C));
                F[q][2 * hf] = v.x, F[q][2 * hf + 1] = v.y;
              }
            }
          }
          const T phi = sx[x] * s, px = dx[x] * s, py = sx[x] * gy, pz = sx[x] * gz, wq = a.W[x] * wyz;
          const T ug = fma(F[0][0], px, fma(F[0][1], py, F[0][2] * pz)), cv = a.cfc * ug;
          const T g2 = fma(px, px, fma(py, py, pz * pz)), st = a.cfs * F[0][3] * ug;
          const T L = fma(lx[x], s, sx[x] * lap);
          const T A = fma(a.nuh2, g2, fma(phi, cv, st * (cv + L))), B = phi * (phi + st), wp = wq * phi;
          d[0] = fma(wq, fma(B, a.cmm + F[1][0], A), fma(wp * F[1][3], px, d[0]));
          d[1] = fma(wq, fma(B, a.cmm + F[2][1], A), fma(wp * F[2][3], py, d[1]));
          d[2] = fma(wq, fma(B, a.cmm + F[3][2], A), fma(wp * F[3][3], pz, d[2]));
          d[3] = fma(wq * F[0][3], g2, d[3]);
        }
      }
    }
  }
  T* o = a.rows + (((int64_t)blockIdx.z * n + blockIdx.y) * NL * M + e) * 4;
  o[0] = a.h3 * d[0];
  o[1] = a.h3 * d[1];
  o[2] = a.h3 * d[2];
  o[3] = a.hp * d[3];
}

// rows of a node added; identity rows (velocity of boundary nodes) 1
template <int K, typename T>
__global__ void __launch_bounds__(256) k_ns_diag_nodes(const T* __restrict__ rows, T* __restrict__ diag, int n) {
  constexpr int Q = K + 1, NL = Q * Q;
  const int M = K * n + 1, t = blockIdx.x * 256 + threadIdx.x;
  if (t >= M * M) return;
  const int ix = t % M, iy = t / M, iz = blockIdx.y;
  T d[4] = {T(0), T(0), T(0), T(0)};
  for (int sz = 0; sz < 2; ++sz) {
    const int cz = iz / K - sz, c = iz - K * cz;
    if (cz < 0 || cz >= n || c > K) continue;
    for (int sy = 0; sy < 2; ++sy) {
      const int cy = iy / K - sy, b = iy - K * cy;
      if (cy < 0 || cy >= n || b > K) continue;
      const T* r = rows + ((((int64_t)cz * n + cy) * NL + c * Q + b) * M + ix) * 4;
#pragma unroll
      for (int f = 0; f < 4; ++f) d[f] += r[f];
    }
  }
  if (ix == 0 || ix == M - 1 || iy == 0 || iy == M - 1 || iz == 0 || iz == M - 1) d[0] = d[1] = d[2] = T(1);
  T* o = diag + ((int64_t)iz * M * M + t) * 4;
#pragma unroll
  for (int f = 0; f < 4; ++f) o[f] = d[f];
}

template <int K, typename T>
static void diagonal(const OpLaunch& L, int prec, void* diag, void* rows, cudaStream_t s) {
  constexpr int Q = K + 1;
  NsDiagArgs<T, Q> a{};
  auto on = [&](int b) { return (L.terms >> b) & 1 ? 1.0 : 0.0; };
  const double lapc = on(6) * L.nu / (L.h * L.h);
  for (int i = 0; i < Q; ++i) {
    for (int m = 0; m < Q; ++m) {
      double ds = 0.0, d2s = 0.0;
      for (int r = 0; r < Q; ++r) {
        ds += L.D[i * Q + r] * L.S[r * Q + m];
        d2s += L.D2[i * Q + r] * L.S[r * Q + m];
      }
      a.S[i][m] = (T)L.S[i * Q + m];
      a.DS[i][m] = (T)ds;
      a.D2S[i][m] = (T)(-lapc * d2s);
    }
    a.W[i] = (T)L.W[i];
  }
  a.fq = static_cast<const T*>(L.lq[prec]);
  a.rows = static_cast<T*>(rows);
  a.n = L.n;
  a.C = L.lc[prec];
  a.cmm = (T)(L.dt > 0 ? on(0) * L.alpha / L.dt : 0.0);
  a.nuh2 = (T)(L.nu / (L.h * L.h));
  a.cfc = (T)on(1);
  a.cfs = (T)on(3);
  a.h3 = (T)(L.h * L.h * L.h);
  a.hp = (T)(L.h * on(5));
  const unsigned n = (unsigned)L.n, M = K * n + 1;
  k_ns_diag<K, T><<<dim3((Q * Q * M + 127) / 128, n, n), 128, 0, s>>>(a);
  MFNS_CUDA(cudaGetLastError());
  k_ns_diag_nodes<K, T><<<dim3((M * M + 255) / 256, M), 256, 0, s>>>(a.rows, static_cast<T*>(diag), L.n);
  MFNS_CUDA(cudaGetLastError());
}

void ns_diagonal(const OpLaunch& L, int prec, void* diag, void* rows, cudaStream_t s) {
  switch (L.k * 2 + (prec == 0 ? 0 : 1)) {
    case 2: return diagonal<1, double>(L, prec, diag, rows, s);
    case 3: return diagonal<1, float>(L, prec, diag, rows, s);
    case 4: return diagonal<2, double>(L, prec, diag, rows, s);
    case 5: return diagonal<2, float>(L, prec, diag, rows, s);
    case 6: return diagonal<3, double>(L, prec, diag, rows, s);
    case 7: return diagonal<3, float>(L, prec, diag, rows, s);
  }
  throw Error(kErrUnsupported, "diagonal on a uniform level: degree");
}

}  // namespace mfns
