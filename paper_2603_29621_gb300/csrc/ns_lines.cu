// Launchers of the stabilised operator on uniform 3D levels (kernels in ns_lines.cuh).
#include <algorithm>
#include <atomic>

#include "common.hpp"
#include "ns_lines.hpp"
#include "opkind.hpp"
#include "ns_lines.cuh"

namespace mfns {

bool ns_lines(const OpLaunch& L) {
  return L.op == OP_STAB_NS && L.dim == 3 && L.structured && L.k >= 1 && L.k <= 3;
}

// Which cell kernel, and the cells per block.  FP32: planes with 32 cells (full warps) where that gives
// every SM a block, else lines with fewer cells.  FP64: lines with four warps per block where the
// chip gets many, else two (finer balance); items on levels that do not fill the SMs' FP64 issue
// ports, with cells for one item per thread and stage, or a third of them on the smallest.
int ns_cells_per_block(int k, int prec, int64_t cells) {
  const int nl = (k + 1) * (k + 1);
  if (prec == 1) {
    int C = 32;
    while (C > 4 && cells / C < 152) C /= 2;
    return C;
  }
  const int items = 32 / nl, least = k == 1 ? 2 : 1;
  if (cells <= 152 * 4 * least) return least;
  if (cells <= 152 * 4 * items) return items;
  return cells / (128 / nl) >= 152 * 8 ? 128 / nl : 64 / nl;
}

enum NsKernel { kLines, kPlanes, kItems };
static NsKernel kernel_of(int k, int prec, int C) {
  if (prec == 1) return C == 32 ? kPlanes : kLines;
  return C <= 32 / ((k + 1) * (k + 1)) ? kItems : kLines;
}
int ns_kernel(const OpLaunch& L, int prec) { return kernel_of(L.k, prec, L.lc[prec]); }

int64_t ns_blocks(const OpLaunch& L, int prec) {
  const int64_t cells = (int64_t)L.n * L.n * L.n;
  return (cells + L.lc[prec] - 1) / L.lc[prec];
}

size_t ns_fq_bytes(const OpLaunch& L, int prec) {
  const int64_t q = L.k + 1;
  return (size_t)(ns_blocks(L, prec) * L.lc[prec] * q * q * q * 16) * (prec == 0 ? 8 : 4);
}

static int64_t rows_values(const OpLaunch& L) {
  const int64_t q = L.k + 1, M = (int64_t)L.k * L.n + 1;
  return (int64_t)L.n * L.n * q * q * M * 4;
}

size_t ns_rows_bytes(const OpLaunch& L, int prec) {
  const int64_t q = L.k + 1;
  return (size_t)(rows_values(L) + ns_blocks(L, prec) * q * q * 4) * (prec == 0 ? 8 : 4);
}

template <typename T, int Q>
static void fill_tab(const OpLaunch& L, NsTab<T, Q>& t) {
  const double h = L.h, lapc = ((L.terms >> 6) & 1) ? L.nu / (h * h) : 0.0;
  const double norm = Q == 3 ? L.W[1] : 1.0;
  for (int i = 0; i < Q; ++i)
    for (int a = 0; a < Q; ++a) {
      const double s = L.S[i * Q + a];
      t.S[i][a] = (T)s;
      t.Sp[i][a] = (T)(s / h);
      t.D[i][a] = (T)L.D[i * Q + a];
      t.D2[i][a] = (T)(-lapc * L.D2[i * Q + a]);
      const double st = L.S[a * Q + i] * L.W[a];
      t.St[i][a] = (T)(st / norm);
      t.Sf[i][a] = (T)(st * norm * norm * h * h * h);
      t.Sfp[i][a] = (T)(st * norm * norm * h * h * L.div_sign);
      double ds = 0.0, d2s = 0.0;
      for (int r = 0; r < Q; ++r) {
        ds += L.D[i * Q + r] * L.S[r * Q + a];
        d2s += L.D2[i * Q + r] * L.S[r * Q + a];
      }
      t.DS[i][a] = (T)ds;
      t.D2S[i][a] = (T)(-lapc * d2s);
      t.Dw[i][a] = (T)(L.D[a * Q + i] * L.W[a] / L.W[i]);
    }
  auto halves = [](const T (&m)[Q][Q], T (&h)[2]) {
    h[0] = (T)(0.5 * ((double)m[0][0] + (double)m[0][Q - 1]));
    h[1] = (T)(0.5 * ((double)m[0][0] - (double)m[0][Q - 1]));
  };
  halves(t.S, t.hS);
  halves(t.Sp, t.hSp);
  halves(t.D, t.hD);
  halves(t.St, t.hSt);
  halves(t.Dw, t.hDw);
  halves(t.Sf, t.hSf);
  halves(t.Sfp, t.hSfp);
}

template <typename T>
static NsProb<T> ns_prob(const OpLaunch& L, int prec, const T* src, void* rows) {
  NsProb<T> p{};
  p.src = src;
  p.fq = static_cast<const T*>(L.lq[prec]);
  p.rows = static_cast<T*>(rows);
  p.tails = p.rows + rows_values(L);
  p.n = L.n;
  p.C = L.lc[prec];
  p.cells = (uint32_t)((int64_t)L.n * L.n * L.n);
  const double dt_inv = L.dt > 0 ? 1.0 / L.dt : 0.0;
  auto on = [&](int b) { return (L.terms >> b) & 1 ? 1.0 : 0.0; };
  p.cmm = (T)(on(0) * L.alpha * dt_inv);
  p.nuh2 = (T)(L.nu / (L.h * L.h));
  p.cfc = (T)on(1);
  p.cfs = (T)on(3);
  p.cfp = (T)(on(5) / L.div_sign);
  p.gen = !(p.cfc == T(1) && p.cfs == T(1) && p.cfp == T(1));
  return p;
}

// launch as a programmatic dependent of the previous kernel of the stream (both kernels here wait for
// it before they touch what it writes)
template <typename Kern, typename Args>
static void launch_pdl(Kern kern, dim3 grid, unsigned block, size_t smem, cudaStream_t s, const Args& a,
                       bool dependent = true) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = dependent ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  MFNS_CUDA(cudaLaunchKernelEx(&cfg, kern, a));
}

// shared memory of the largest block, once per device
template <typename Kern>
static void set_smem(Kern kern, size_t bytes, std::atomic<uint64_t>& done) {
  int dev = 0;
  MFNS_CUDA(cudaGetDevice(&dev));
  const uint64_t bit = 1ull << (dev & 63);
  if (done.load() & bit) return;
  MFNS_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
  MFNS_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
  done.fetch_or(bit);
}

// Shared memory of a cell launch, raised so that no SM takes more than its share of a grid that does not
// fill the chip: a dependent launch finds some SMs free before others, and its blocks would pile up
// there (V-cycles FP32 48^3 1115 -> 1086 us, 8^3 181 -> 173 us).  It keeps other streams' blocks off those
// SMs for as long as the launch lasts; problems on streams of their own are still faster than with colour launches
// (8 V-cycles of Q2 8^3 at a time, each: 61 -> 40 us, of 20^3 176 -> 116, of Q3 8^3 92 -> 87 us).
static size_t spread_smem(size_t need, int64_t blocks) {
  const int64_t per_sm = (blocks + 151) / 152;
  if (per_sm > 16) return need;
  const size_t share = (size_t)(228 * 1024 / per_sm - 1024) / 128 * 128;
  return std::max(need, std::min(share, (size_t)227 * 1024));
}

template <int K, typename T, bool MULTI>
static void launch_cells(const NsArgs<T, K + 1>& a, int64_t blocks, int cmax, cudaStream_t s) {
  const NsKernel kind = kernel_of(K, sizeof(T) == 4, cmax);
  const dim3 grid((unsigned)blocks);
  // FP64 cells start on an idle chip, spread evenly over the SMs: every warp's operations take 64 cycles,
  // and an early start that doubles the load of a few SMs costs more than the launch it hides (V-cycle
  // 21^3 2417 -> 2367 us; 3170 us when the blocks may also pile up)
  const bool early = sizeof(T) == 4;
  if constexpr (sizeof(T) == 8) {
    if (kind == kItems) {
      static std::atomic<uint64_t> done{0};
      set_smem(k_ns_items<K, MULTI>, 227 * 1024, done);
      return launch_pdl(k_ns_items<K, MULTI>, grid, NsItems<K>::THREADS, spread_smem(NsItems<K>::smem(cmax), blocks), s,
                        a, early);
    }
  }
  if constexpr (sizeof(T) == 4) {
    if (kind == kPlanes) {
      static std::atomic<uint64_t> done{0};
      set_smem(k_ns_planes<K, MULTI>, 227 * 1024, done);
      return launch_pdl(k_ns_planes<K, MULTI>, grid, NsPlane<K>::THREADS, spread_smem(NsPlane<K>::SMEM, blocks), s, a);
    }
  }
  using Sh = NsShape<K, T>;
  static std::atomic<uint64_t> done{0};
  set_smem(k_ns_cells<K, T, MULTI>, 227 * 1024, done);
  launch_pdl(k_ns_cells<K, T, MULTI>, grid, (unsigned)Sh::threads(cmax), spread_smem(Sh::smem(cmax), blocks), s, a,
             early);
}

template <int K, typename T>
static void cells_t(const OpLaunch& L, int prec, const void* src, void* rows, cudaStream_t s) {
  NsArgs<T, K + 1> a{};
  fill_tab(L, a.one.tab);
  a.one.p = ns_prob<T>(L, prec, static_cast<const T*>(src), rows);
  a.err = op_wait_flag();
  const bool timed = L.timer && L.timer->enabled;
  if (timed) L.timer->record_pair_begin(s);
  launch_cells<K, T, false>(a, ns_blocks(L, prec), L.lc[prec], s);
  if (timed) L.timer->record_pair_end(s);
}

template <int K, typename T>
static void desc_t(const OpLaunch& L, int prec, const void* src, void* rows, int32_t first_block,
                   std::vector<char>& out) {
  NsDesc<T, K + 1> d{};
  fill_tab(L, d.tab);
  d.p = ns_prob<T>(L, prec, static_cast<const T*>(src), rows);
  d.p.first_block = first_block;
  const char* c = reinterpret_cast<const char*>(&d);
  out.insert(out.end(), c, c + sizeof(d));
}

template <int K, typename T>
static void multi_t(const NsMulti& m, cudaStream_t s) {
  NsArgs<T, K + 1> a{};
  a.probs = static_cast<const NsDesc<T, K + 1>*>(m.probs);
  a.block_pid = m.block_pid;
  a.err = op_wait_flag();
  launch_cells<K, T, true>(a, m.blocks, m.cmax, s);
}

template <int K, typename T>
static void nodes_t(const OpLaunch& L, int prec, const NsAfterArgs& f, void* rows, cudaStream_t s) {
  NsNodeArgs<T> a{};
  a.dst = static_cast<T*>(f.dst);
  a.src = static_cast<const T*>(f.src);
  a.rows = static_cast<const T*>(rows);
  a.tails = a.rows + rows_values(L);
  a.b = static_cast<const T*>(f.b);
  a.dinv = static_cast<const T*>(f.dinv);
  a.d = static_cast<T*>(f.d);
  a.c1 = (T)f.c1;
  a.c2 = (T)f.c2;
  a.n = L.n;
  a.C = L.lc[prec];
  a.magic = a.C > 1 ? (uint32_t)(((1ull << 32) + a.C - 1) / a.C) : 0u;
  const unsigned M = (unsigned)(K * L.n + 1);
  const dim3 grid((M * M + 255) / 256, M);
  const bool early = sizeof(T) == 4;  // (FP64: V-cycle 21^3 1794 -> 1766 us without)
  if (f.after == 0)
    launch_pdl(k_ns_nodes<T, K, kStore>, grid, 256, 0, s, a, early);
  else if (f.after == 1)
    launch_pdl(k_ns_nodes<T, K, kUpdate>, grid, 256, 0, s, a, early);
  else
    launch_pdl(k_ns_nodes<T, K, kResidual>, grid, 256, 0, s, a, early);
}

#define MFNS_NS_DISPATCH(CALL)                                      \
  switch (L.k * 2 + (prec == 0 ? 0 : 1)) {                          \
    case 2: return CALL(1, double);                                 \
    case 3: return CALL(1, float);                                  \
    case 4: return CALL(2, double);                                 \
    case 5: return CALL(2, float);                                  \
    case 6: return CALL(3, double);                                 \
    case 7: return CALL(3, float);                                  \
  }                                                                 \
  throw Error(kErrUnsupported, "stabilised operator on a uniform level: degree");

void ns_cells(const OpLaunch& L, int prec, const void* src, void* rows, cudaStream_t s) {
#define CALL(K, T) cells_t<K, T>(L, prec, src, rows, s)
  MFNS_NS_DISPATCH(CALL)
#undef CALL
}
void ns_cells_multi(const OpLaunch& L, int prec, const NsMulti& m, cudaStream_t s) {
#define CALL(K, T) multi_t<K, T>(m, s)
  MFNS_NS_DISPATCH(CALL)
#undef CALL
}
void ns_descriptor(const OpLaunch& L, int prec, const void* src, void* rows, int32_t first_block,
                   std::vector<char>& out) {
#define CALL(K, T) desc_t<K, T>(L, prec, src, rows, first_block, out)
  MFNS_NS_DISPATCH(CALL)
#undef CALL
}
void ns_nodes(const OpLaunch& L, int prec, const NsAfterArgs& f, void* rows, cudaStream_t s) {
#define CALL(K, T) nodes_t<K, T>(L, prec, f, rows, s)
  MFNS_NS_DISPATCH(CALL)
#undef CALL
}

}  // namespace mfns
