// Separable transfers between uniform meshes (Eq. 4 on tensor-product grids), nested
// (n -> n/2) or non-nested (odd n -> (n+1)/2, Section 2) h-steps and p-steps.
//
// On a uniform mesh the Q_k space is the tensor product of 1D spaces, and the
// interpolation P of Eq. 4 (coarse FE function evaluated at the fine nodes) is
// the tensor product of one 1D matrix P1 per direction: h-steps (n -> 2n cells,
// same degree) and p-steps (same cells, degree k-1 -> k) alike.  Restriction
// (P^T) and prolongation therefore need no cell loop and no colouring: each is one launch over the
// global node grid that applies the three 1D stencils to a tile (below).  Constrained (Dirichlet) velocity entries are
// masked exactly as in the cell-based transfer: P ignores the coarse ones and
// gives zero on the fine ones, so the restriction reads fine boundary velocity
// entries as zero and the prolongation never adds into them.
#include <atomic>

#include "problem.hpp"
#include "vec.hpp"

namespace mfns {

namespace {

// One 1D pass along `axis` of a grid (Mx, My, Mz) -> (Mx', My', Mz') with only the axis
// extent changing (the state interpolation): out[node'] = sum_j w_j in[node along axis = idx_j].
template <int NC>
__global__ void k_pass(const double* __restrict__ in, double* __restrict__ out, int axis, int64_t ix, int64_t iy,
                       int64_t iz, int64_t mo, const int32_t* __restrict__ ptr, const int32_t* __restrict__ idx,
                       const double* __restrict__ w) {
  int64_t ext_in[3] = {ix, iy, iz};
  int64_t ext_out[3] = {ix, iy, iz};
  ext_out[axis] = mo;
  const int64_t total = ext_out[0] * ext_out[1] * ext_out[2];
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    int64_t c[3] = {t % ext_out[0], (t / ext_out[0]) % ext_out[1], t / (ext_out[0] * ext_out[1])};
    const int64_t o = c[axis];
    double acc[NC];
#pragma unroll
    for (int f = 0; f < NC; ++f) acc[f] = 0;
    for (int32_t j = ptr[o]; j < ptr[o + 1]; ++j) {
      c[axis] = idx[j];
      const double* src = in + ((c[2] * ext_in[1] + c[1]) * ext_in[0] + c[0]) * NC;
      const double wj = w[j];
#pragma unroll
      for (int f = 0; f < NC; ++f) acc[f] += wj * src[f];
    }
#pragma unroll
    for (int f = 0; f < NC; ++f) out[t * NC + f] = acc[f];
  }
}

template <int NC>
void pass(const double* in, double* out, int axis, const int64_t ext[3], int64_t mo, const DevBuf& ptr,
          const DevBuf& idx, const DevBuf& w, cudaStream_t s) {
  int64_t eo[3] = {ext[0], ext[1], ext[2]};
  eo[axis] = mo;
  const int64_t total = eo[0] * eo[1] * eo[2];
  const unsigned grid = (unsigned)std::min<int64_t>((total + 255) / 256, 152 * 16);
  k_pass<NC><<<grid, 256, 0, s>>>(in, out, axis, ext[0], ext[1], ext[2], mo, ptr.as<int32_t>(), idx.as<int32_t>(),
                                  w.as<double>());
  MFNS_CUDA(cudaGetLastError());
}

template <typename T, int NC>
__device__ __forceinline__ void load_node(const T* p, T (&v)[NC]) {
  if constexpr (NC == 4 && sizeof(T) == 4) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  } else if constexpr (NC == 4) {
    const double2 a = *reinterpret_cast<const double2*>(p), b = *reinterpret_cast<const double2*>(p + 2);
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
  } else {
#pragma unroll
    for (int f = 0; f < NC; ++f) v[f] = p[f];
  }
}
template <typename T, int NC>
__device__ __forceinline__ void store_node(T* p, const T (&v)[NC]) {
  if constexpr (NC == 4 && sizeof(T) == 4) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  } else if constexpr (NC == 4) {
    *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
    *reinterpret_cast<double2*>(p + 2) = make_double2(v[2], v[3]);
  } else {
#pragma unroll
    for (int f = 0; f < NC; ++f) p[f] = v[f];
  }
}

template <typename T>
struct TensorArgs {
  const T* in;
  T* out;
  const int32_t *ptr, *idx;  // rows of the 1D matrix: output nodes
  const T* w;
  const int32_t *lo, *hi;    // first / last input node of the rows >= r / <= r
  int Mi, Mo, dim, nvel;
  int rows, cols, xblocks;   // output tile of a block, blocks along x
  // first smoothing step of the coarse level from a zero iterate: x = d = c2 dinv out (x null: none)
  T *x, *d;
  const T* dinv;
  T c2;
};

// out = (R (x) R (x) R) in (restriction, R = P1^T) or out += (R (x) R (x) R) in (ADD: prolongation, R = P1)
// in one launch.  A block owns a tile (rows x cols) of one output z-plane: it sums the input planes
// of its z-row over the input nodes that the tile touches (global memory, consecutive in x), then y and
// x from shared memory.  This order does the fewest operations, which is what counts in FP64 (1D passes
// nested per output node did 27 products instead of 9 and made the 21^3 FP64 V-cycle 0.6 ms slower),
// and only overlapping tile borders are read twice.  The 1D rows of the tile are copied to shared
// memory before the wait for the previous kernel.  Against one launch per direction: 48^3 -> 24^3 Q2
// FP32 restriction 39 -> 18 us, prolongation 56 -> 14 us, and two launches less per transfer,
// which is most of a small level's.
template <typename T, int NC, bool ADD>
__global__ void __launch_bounds__(256) k_tensor(const TensorArgs<T> a) {
  extern __shared__ __align__(16) unsigned char sep_smem[];
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const int Mi = a.Mi, Mo = a.Mo;
  const int by = blockIdx.x / a.xblocks, bx = blockIdx.x - by * a.xblocks, oz = blockIdx.y;
  const int y0 = by * a.rows, nr = min(a.rows, Mo - y0), x0 = bx * a.cols, nc = min(a.cols, Mo - x0);
  const int ylo = a.lo[y0], ny = a.hi[y0 + nr - 1] + 1 - ylo, xlo = a.lo[x0], nx = a.hi[x0 + nc - 1] + 1 - xlo;
  // the 1D rows of the tile: x, y, z
  const int yp0 = a.ptr[y0], xp0 = a.ptr[x0], zp0 = a.dim == 3 ? a.ptr[oz] : 0;
  const int nxe = a.ptr[x0 + nc] - xp0, nye = a.ptr[y0 + nr] - yp0, nz = a.dim == 3 ? a.ptr[oz + 1] - zp0 : 1;
  T* S1 = reinterpret_cast<T*>(sep_smem);
  T* S2 = S1 + (int64_t)ny * nx * NC;
  T* wx = S2 + (int64_t)nr * nx * NC;
  T* wy = wx + nxe;
  T* wz = wy + nye;
  int32_t* ixs = reinterpret_cast<int32_t*>(wz + nz);
  int32_t* iys = ixs + nxe;
  int32_t* izs = iys + nye;
  int32_t* px = izs + nz;
  int32_t* py = px + nc + 1;
  for (int e = threadIdx.x; e < nxe; e += 256) {
    wx[e] = a.w[xp0 + e];
    ixs[e] = a.idx[xp0 + e] - xlo;
  }
  for (int e = threadIdx.x; e < nye; e += 256) {
    wy[e] = a.w[yp0 + e];
    iys[e] = a.idx[yp0 + e] - ylo;
  }
  for (int e = threadIdx.x; e < nz; e += 256) {
    wz[e] = a.dim == 3 ? a.w[zp0 + e] : T(1);
    izs[e] = a.dim == 3 ? a.idx[zp0 + e] : 0;
  }
  for (int e = threadIdx.x; e <= nc; e += 256) px[e] = a.ptr[x0 + e] - xp0;
  for (int e = threadIdx.x; e <= nr; e += 256) py[e] = a.ptr[y0 + e] - yp0;
  __syncthreads();
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  for (int it = threadIdx.x; it < ny * nx; it += 256) {
    const int q = it / nx, y = ylo + q, x = xlo + it - q * nx;
    const bool edge = y == 0 || y == Mi - 1 || x == 0 || x == Mi - 1;
    const T* p = a.in + ((int64_t)y * Mi + x) * NC;
    T s[NC];
#pragma unroll
    for (int f = 0; f < NC; ++f) s[f] = T(0);
#pragma unroll 4
    for (int e = 0; e < nz; ++e) {
      const int z = izs[e];
      const T w = wz[e];
      const bool bnd = edge || (a.dim == 3 && (z == 0 || z == Mi - 1));
      T v[NC];
      load_node<T, NC>(p + (int64_t)z * Mi * Mi * NC, v);
#pragma unroll
      for (int f = 0; f < NC; ++f) s[f] = fma(w, bnd && f < a.nvel ? T(0) : v[f], s[f]);
    }
    store_node<T, NC>(S1 + (int64_t)it * NC, s);
  }
  __syncthreads();
  for (int it = threadIdx.x; it < nr * nx; it += 256) {
    const int r = it / nx, x = it - r * nx;
    T s[NC];
#pragma unroll
    for (int f = 0; f < NC; ++f) s[f] = T(0);
    const int e1 = py[r + 1];
#pragma unroll 4
    for (int e = py[r]; e < e1; ++e) {
      T v[NC];
      load_node<T, NC>(S1 + ((int64_t)iys[e] * nx + x) * NC, v);
#pragma unroll
      for (int f = 0; f < NC; ++f) s[f] = fma(wy[e], v[f], s[f]);
    }
    store_node<T, NC>(S2 + (int64_t)it * NC, s);
  }
  __syncthreads();
  for (int it = threadIdx.x; it < nr * nc; it += 256) {
    const int r = it / nc, c = it - r * nc, oy = y0 + r, ox = x0 + c;
    const bool bnd = ox == 0 || ox == Mo - 1 || oy == 0 || oy == Mo - 1 || (a.dim == 3 && (oz == 0 || oz == Mo - 1));
    const int64_t o = (((int64_t)oz * Mo + oy) * Mo + ox) * NC;
    T s[NC], old[NC];
    if (ADD) load_node<T, NC>(a.out + o, old);
#pragma unroll
    for (int f = 0; f < NC; ++f) s[f] = T(0);
    const int e1 = px[c + 1];
#pragma unroll 4
    for (int e = px[c]; e < e1; ++e) {
      T v[NC];
      load_node<T, NC>(S2 + ((int64_t)r * nx + ixs[e]) * NC, v);
#pragma unroll
      for (int f = 0; f < NC; ++f) s[f] = fma(wx[e], v[f], s[f]);
    }
    // constrained rows of a uniform level: the velocity of boundary nodes
#pragma unroll
    for (int f = 0; f < NC; ++f) {
      const bool fixed = bnd && f < a.nvel;
      s[f] = ADD ? (fixed ? old[f] : old[f] + s[f]) : (fixed ? T(0) : s[f]);
    }
    store_node<T, NC>(a.out + o, s);
    if (!ADD && a.x) {
      T v[NC];
      load_node<T, NC>(a.dinv + o, v);
#pragma unroll
      for (int f = 0; f < NC; ++f) v[f] = a.c2 * v[f] * s[f];
      store_node<T, NC>(a.x + o, v);
      store_node<T, NC>(a.d + o, v);
    }
  }
}

template <typename Kern, typename Args>
void launch_pdl(Kern kern, dim3 grid, unsigned block, size_t smem, cudaStream_t s, const Args& a, bool fp64) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  // (FP64 starts on an idle chip: blocks that start early pile up on the first SMs that are free, Q2 24^3 ->
  // Q1 prolongation 26.9 -> 16.4 us, restriction 23.2 -> 14.4 us)
  cfg.numAttrs = fp64 ? 0 : 1;
  MFNS_CUDA(cudaLaunchKernelEx(&cfg, kern, a));
}

// CSR of a 1D matrix given as dense rows (drop exact zeros)
void to_csr(const std::vector<double>& M, int64_t rows, int64_t cols, std::vector<int32_t>& ptr,
            std::vector<int32_t>& idx, std::vector<double>& w) {
  ptr.assign(1, 0);
  idx.clear();
  w.clear();
  for (int64_t r = 0; r < rows; ++r) {
    for (int64_t c = 0; c < cols; ++c) {
      const double v = M[r * cols + c];
      if (std::fabs(v) > 1e-15) {
        idx.push_back((int32_t)c);
        w.push_back(v);
      }
    }
    ptr.push_back((int32_t)idx.size());
  }
}

constexpr size_t kTensorSmem = 72 * 1024;  // three blocks per SM

// tables and tiles of one 1D matrix applied along every axis
void plan_dir(SepDir& d, const SepTransfer& t, const std::vector<int32_t>& ptr, const std::vector<int32_t>& idx,
              const std::vector<double>& w, int rows_max, Budget* bud) {
  const int Mo = (int)ptr.size() - 1;
  std::vector<int32_t> lo(Mo), hi(Mo);
  d.width = 1;
  for (int c = 0; c < Mo; ++c) {
    d.width = std::max(d.width, ptr[c + 1] - ptr[c]);
    hi[c] = std::max(c ? hi[c - 1] : 0, idx[ptr[c + 1] - 1]);
  }
  for (int c = Mo - 1; c >= 0; --c) lo[c] = std::min(c + 1 < Mo ? lo[c + 1] : idx[ptr[c]], idx[ptr[c]]);
  d.ptr = upload(bud, ptr);
  d.idx = upload(bud, idx);
  d.w[0] = upload(bud, w);
  d.w[1] = upload(bud, std::vector<float>(w.begin(), w.end()));
  d.lo = upload(bud, lo);
  d.hi = upload(bud, hi);
  // input nodes of the widest tile of r output nodes
  auto span = [&](int r) {
    int m = 1;
    for (int c = 0; c < Mo; c += r) m = std::max(m, hi[std::min(c + r, Mo) - 1] - lo[c] + 1);
    return m;
  };
  for (int prec = 0; prec < 2; ++prec) {
    auto smem = [&](int rows, int cols) {
      const size_t es = esize(prec), nx = span(cols);
      return ((size_t)span(rows) + rows) * nx * t.ncomp * es + ((size_t)(rows + cols + 1) * d.width) * (es + 4) +
             (size_t)(rows + cols + 2) * 4;
    };
    // few rows overlap little with the next tile; fewer while the chip is not full, and columns until
    // the sums fit
    int rows = std::min(rows_max, Mo), cols = Mo;
    const int64_t planes = t.dim == 3 ? Mo : 1;
    while (cols > 1 && smem(rows, cols) > kTensorSmem) cols = (cols + 1) / 2;
    auto blocks = [&] { return (int64_t)((Mo + rows - 1) / rows) * ((Mo + cols - 1) / cols) * planes; };
    while (rows > 1 && blocks() < 152) rows = (rows + 1) / 2;
    d.rows[prec] = rows;
    d.cols[prec] = cols;
    d.smem[prec] = smem(rows, cols);
  }
}

}  // namespace

bool build_separable(SepTransfer& t, const OpLevel& fine, const OpLevel& coarse, Budget* bud) {
  if (!fine.forest.uniform() || !coarse.forest.uniform() || !fine.L.structured || !coarse.L.structured) return false;
  const int nf = fine.forest.n, nc = coarse.forest.n, kf = fine.k, kc = coarse.k;
  const bool h = kf == kc && nc == (nf + 1) / 2 && nc < nf;  // nested (even nf) or non-nested (odd nf)
  const bool p = nf == nc && kf > kc;
  if (!h && !p) return false;
  t.dim = fine.dim;
  t.ncomp = fine.NU;
  t.nvel = fine.op == OP_PMASS ? 0 : fine.dim;
  t.Mf = (int64_t)kf * nf + 1;
  t.Mc = (int64_t)kc * nc + 1;
  // dense 1D interpolation P1 (Mf x Mc): coarse basis at every fine node
  std::vector<double> xf = gll_nodes(kf), xc = gll_nodes(kc);
  std::vector<double> P1(t.Mf * t.Mc, 0.0);
  for (int64_t g = 0; g < t.Mf; ++g) {
    int64_t cf = g / kf, s = g % kf;
    if (cf == nf) { cf = nf - 1; s = kf; }
    int64_t cc = cf;
    double xi = xf[s];
    if (h && nf == 2 * nc) {  // nested: child half of the parent cell
      cc = cf / 2;
      xi = 0.5 * ((cf % 2) + xf[s]);
    } else if (h) {           // non-nested: locate the fine node in the coarse mesh
      const double X = (double(cf) + xf[s]) * double(nc) / double(nf);
      cc = std::min<int64_t>((int64_t)std::floor(X), nc - 1);
      xi = X - double(cc);
    }
    for (int m = 0; m <= kc; ++m) P1[g * t.Mc + (int64_t)kc * cc + m] = lagrange(xc, m, xi);
  }
  std::vector<double> P1T(t.Mc * t.Mf);
  for (int64_t g = 0; g < t.Mf; ++g)
    for (int64_t c = 0; c < t.Mc; ++c) P1T[c * t.Mf + g] = P1[g * t.Mc + c];
  std::vector<int32_t> ptr, idx;
  std::vector<double> w;
  to_csr(P1, t.Mf, t.Mc, ptr, idx, w);
  plan_dir(t.p, t, ptr, idx, w, 16, bud);
  to_csr(P1T, t.Mc, t.Mf, ptr, idx, w);
  plan_dir(t.r, t, ptr, idx, w, 8, bud);
  // dense 1D interpolation I1 (Mc x Mf): fine basis at every coarse node (used to carry a fine
  // FE function, e.g. a Newton state, down the hierarchy)
  std::vector<double> I1(t.Mc * t.Mf, 0.0);
  for (int64_t g = 0; g < t.Mc; ++g) {
    int64_t cc = g / kc, s = g % kc;
    if (cc == nc) { cc = nc - 1; s = kc; }
    const double X = (double(cc) + xc[s]) * double(nf) / double(nc);  // position in fine cells
    const int64_t cf = std::min<int64_t>((int64_t)std::floor(X), nf - 1);
    const double xi = X - double(cf);
    for (int m = 0; m <= kf; ++m) I1[g * t.Mf + (int64_t)kf * cf + m] = lagrange(xf, m, xi);
  }
  to_csr(I1, t.Mc, t.Mf, ptr, idx, w);
  t.i_ptr = upload(bud, ptr);
  t.i_idx = upload(bud, idx);
  t.i_w = upload(bud, w);
  // intermediate grids of the state interpolation: after the first pass and after the second (3D)
  const int64_t a = t.dim == 3 ? t.Mc * t.Mf * t.Mf : t.Mc * t.Mf;
  const int64_t b = t.dim == 3 ? t.Mc * t.Mc * t.Mf : 0;
  t.tmp1.alloc(bud, std::max<int64_t>(a, 1) * t.ncomp * 8);
  t.tmp2.alloc(bud, std::max<int64_t>(b, 1) * t.ncomp * 8);
  return true;
}

template <typename T, int NC, bool ADD>
static void sep_apply(const SepTransfer& t, const SepDir& d, int64_t Mi, int64_t Mo, int prec, const T* in, T* out,
                      const SepStart* st, cudaStream_t s) {
  TensorArgs<T> a{};
  a.in = in;
  a.out = out;
  a.ptr = d.ptr.as<int32_t>();
  a.idx = d.idx.as<int32_t>();
  a.w = d.w[prec].as<T>();
  a.lo = d.lo.as<int32_t>();
  a.hi = d.hi.as<int32_t>();
  a.Mi = (int)Mi;
  a.Mo = (int)Mo;
  a.dim = t.dim;
  a.nvel = t.nvel;
  a.rows = d.rows[prec];
  a.cols = d.cols[prec];
  a.xblocks = (int)((Mo + a.cols - 1) / a.cols);
  if (st) {
    a.x = static_cast<T*>(st->x);
    a.d = static_cast<T*>(st->d);
    a.dinv = static_cast<const T*>(st->dinv);
    a.c2 = (T)st->c2;
  }
  static std::atomic<uint64_t> done{0};  // per device
  int dev = 0;
  MFNS_CUDA(cudaGetDevice(&dev));
  const uint64_t bit = 1ull << (dev & 63);
  if (!(done.load() & bit)) {
    MFNS_CUDA(cudaFuncSetAttribute(k_tensor<T, NC, ADD>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024));
    done.fetch_or(bit);
  }
  const dim3 grid((unsigned)((Mo + a.rows - 1) / a.rows * a.xblocks), (unsigned)(t.dim == 3 ? Mo : 1));
  launch_pdl(k_tensor<T, NC, ADD>, grid, 256, d.smem[prec], s, a, sizeof(T) == 8);
}

template <typename T>
static void sep_dispatch(const SepTransfer& t, int prec, const T* in, T* out, bool restrict_, const SepStart* st,
                         cudaStream_t s) {
  switch (t.ncomp) {
#define C(NC)                                                                            \
  case NC:                                                                               \
    if (restrict_) sep_apply<T, NC, false>(t, t.r, t.Mf, t.Mc, prec, in, out, st, s);    \
    else sep_apply<T, NC, true>(t, t.p, t.Mc, t.Mf, prec, in, out, nullptr, s);          \
    return;
    C(1) C(2) C(3) C(4)
#undef C
  }
  throw Error(kErrUnsupported, "separable transfer: unsupported component count");
}

template <int NC>
static void sep_interpolate_t(const SepTransfer& t, const double* fine, double* coarse, cudaStream_t s) {
  const int64_t Mf = t.Mf, Mc = t.Mc;
  double* t1 = t.tmp1.as<double>();
  double* t2 = t.tmp2.as<double>();
  if (t.dim == 3) {
    const int64_t e0[3] = {Mf, Mf, Mf}, e1[3] = {Mc, Mf, Mf}, e2[3] = {Mc, Mc, Mf};
    pass<NC>(fine, t1, 0, e0, Mc, t.i_ptr, t.i_idx, t.i_w, s);
    pass<NC>(t1, t2, 1, e1, Mc, t.i_ptr, t.i_idx, t.i_w, s);
    pass<NC>(t2, coarse, 2, e2, Mc, t.i_ptr, t.i_idx, t.i_w, s);
  } else {
    const int64_t e0[3] = {Mf, Mf, 1}, e1[3] = {Mc, Mf, 1};
    pass<NC>(fine, t1, 0, e0, Mc, t.i_ptr, t.i_idx, t.i_w, s);
    pass<NC>(t1, coarse, 1, e1, Mc, t.i_ptr, t.i_idx, t.i_w, s);
  }
}

void sep_interpolate(const SepTransfer& t, const double* fine, double* coarse, cudaStream_t s) {
  switch (t.ncomp) {
    case 1: return sep_interpolate_t<1>(t, fine, coarse, s);
    case 2: return sep_interpolate_t<2>(t, fine, coarse, s);
    case 3: return sep_interpolate_t<3>(t, fine, coarse, s);
    case 4: return sep_interpolate_t<4>(t, fine, coarse, s);
  }
  throw Error(kErrUnsupported, "separable interpolation: unsupported component count");
}

void sep_restrict(const SepTransfer& t, int prec, const void* fine, void* coarse, const SepStart* st, cudaStream_t s) {
  if (prec == 0) sep_dispatch<double>(t, 0, (const double*)fine, (double*)coarse, true, st, s);
  else sep_dispatch<float>(t, 1, (const float*)fine, (float*)coarse, true, st, s);
}

void sep_prolongate_add(const SepTransfer& t, int prec, const void* coarse, void* fine, cudaStream_t s) {
  if (prec == 0) sep_dispatch<double>(t, 0, (const double*)coarse, (double*)fine, false, nullptr, s);
  else sep_dispatch<float>(t, 1, (const float*)coarse, (float*)fine, false, nullptr, s);
}

}  // namespace mfns
