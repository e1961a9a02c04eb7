// A*X products of SNMPBB: the only O(n^2 r) (dense) / O(nnz r) (sparse) step of an
// iteration (Sec. 4.1 complexity list; the V H^T product of Eqs. (2.1)-(2.2)).
//
//   k_gemm_dense : CUDA-core tiled product for FP64 / FP32 A, and for the final evaluation of
//                  BF16 and E4M3 A (gemm_dev.cuh).  Split-K writes each split to its own
//                  workspace slice; the finish pass sums the slices in a fixed order, so
//                  results are deterministic.
//   k_spmm_csr   : lanes across the factor columns (coalesced rows of X), with Y += c X2.
//   k_ax_finish  : fused epilogue: sum of split slices, Y += c X2, and per-restart FP64
//                  partials of <P1, A X> and <P2, A X> (e.g. tr(W^T A W)).
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "gemm_dev.cuh"

namespace snmf {

namespace {

__device__ __forceinline__ float ld_a(const float* p) { return *p; }
__device__ __forceinline__ double ld_a(const double* p) { return *p; }

template <typename C, typename TA, int PER_SM>
__global__ void __launch_bounds__(C::NT, PER_SM)
k_gemm_dense(const TA* __restrict__ A, int64_t lda, const typename C::T* __restrict__ X, int64_t ld,
             typename C::T* __restrict__ Y, int64_t n, int cols, int64_t kchunk, bool avec, bool xvec, GemmA8 a8,
             const int* run) {
  using T = typename C::T;
  extern __shared__ __align__(16) unsigned char gemm_sm[];
  if (run && *run == 0) return;
  const int64_t row0 = (int64_t)blockIdx.y * C::BM, k0 = (int64_t)blockIdx.z * kchunk;
  const int col0 = blockIdx.x * C::BN;
  T acc[C::TM][C::TN];
  gemm_tile<C>(A, lda, X, ld, n, cols, row0, col0, k0, min(n, k0 + kchunk), avec, xvec, a8,
               reinterpret_cast<T*>(gemm_sm), acc);
  T* Yout = Y + (int64_t)blockIdx.z * n * ld;
  const int tx = threadIdx.x % C::TX, ty = threadIdx.x / C::TX;
#pragma unroll
  for (int i = 0; i < C::TM; ++i) {
    const int64_t r = row0 + ty + C::TY * i;
    if (r >= n) continue;
#pragma unroll
    for (int j = 0; j < C::TN; j += C::VW) {
      const int c = col0 + C::col(tx, j);
      T* p = Yout + r * ld + c;
      if (C::VW == 4 && xvec) {  // the pitch and the columns of Y are X's
        if (c < cols) *reinterpret_cast<float4*>(p) = make_float4(acc[i][j], acc[i][j + 1 < C::TN ? j + 1 : j],
                                                                  acc[i][j + 2 < C::TN ? j + 2 : j],
                                                                  acc[i][j + 3 < C::TN ? j + 3 : j]);
      } else {
#pragma unroll
        for (int u = 0; u < C::VW; ++u)
          if (c + u < cols) p[u] = acc[i][j + u];
      }
    }
  }
}

// CSR SpMM, Y = A X (+ c X2): LPR lanes per row, V consecutive columns (16 bytes where the columns
// allow it) per lane; blockIdx.y = window of LPR V columns, the slowest index of the grid, so the
// windows of X pass through L2 one after the other.  The entries of a row are taken U at a time with
// the next indices already in flight, and added in their order.  Bound by the gather from L2 (n =
// 20000, 15 entries per row, 640 columns: 353 us with single columns and one entry at a time, and a
// finish pass of its own).
// What is read ahead is tested with an index up to 2 U - 2 beyond the row's end, which has to fit into 32 bits:
// kCsrAhead (the test by the entries that are left instead: n = 20000, 640 columns 12 per cent slower).
constexpr int64_t kCsrAhead = INT32_MAX - 16;

template <typename TV, typename T, int V, int LPR, int U = V * sizeof(T) == 16 ? 4 : 8>
__global__ void __launch_bounds__(256)
k_spmm_csr(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colidx,
           const TV* __restrict__ vals, const T* __restrict__ X, int64_t ld,
           T* __restrict__ Y, int64_t n, int cols, T c, const T* __restrict__ X2, const int* run) {
  struct alignas(V * sizeof(T)) Vec {
    T v[V];
  };
  if (run && *run == 0) return;
  const int lane = threadIdx.x & 31;
  const int64_t row = ((int64_t)blockIdx.x * 8 + (threadIdx.x >> 5)) * (32 / LPR) + lane / LPR;
  const int col = (blockIdx.y * LPR + lane % LPR) * V;
  if (row >= n || col >= cols) return;
  Vec acc;
#pragma unroll
  for (int k = 0; k < V; ++k) acc.v[k] = T(0);
  const int beg = rowptr[row], end = rowptr[row + 1];
  int32_t ci[U];
  T va[U];
  auto load = [&](int e) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      ci[u] = e + u < end ? __ldg(colidx + e + u) : -1;
      va[u] = e + u < end ? (T)__ldg(vals + e + u) : T(0);
    }
  };
  load(beg);
  for (int e = beg; e < end; e += U) {
    Vec x[U];
    T w[U];
    bool on[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      on[u] = ci[u] >= 0;
      w[u] = va[u];
      if (on[u]) x[u] = *reinterpret_cast<const Vec*>(X + (int64_t)ci[u] * ld + col);
    }
    load(e + U);
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (on[u]) {
#pragma unroll
        for (int k = 0; k < V; ++k) acc.v[k] = fma(w[u], x[u].v[k], acc.v[k]);
      }
  }
  const int64_t idx = row * ld + col;
  if (X2) {
    const Vec x2 = *reinterpret_cast<const Vec*>(X2 + idx);
#pragma unroll
    for (int k = 0; k < V; ++k) acc.v[k] = acc.v[k] + c * x2.v[k];
  }
  *reinterpret_cast<Vec*>(Y + idx) = acc;
}

// Y = sum_s ws[s] (splits > 1, in slice order) or Y (+ c X2) over `total` contiguous values, V per
// thread (16 bytes), eight slices in flight.
template <typename T, int V>
__global__ void __launch_bounds__(256)
k_ax_sum(int64_t total, T* __restrict__ Y, const T* __restrict__ ws, int splits, T c, const T* __restrict__ X2,
         const int* run) {
  struct alignas(V * sizeof(T)) Vec {
    T v[V];
  };
  if (run && *run == 0) return;
  const int64_t idx = ((int64_t)blockIdx.x * 256 + threadIdx.x) * V;
  if (idx >= total) return;
  Vec x2, y = *reinterpret_cast<const Vec*>((splits > 1 ? ws : Y) + idx);
  if (X2) x2 = *reinterpret_cast<const Vec*>(X2 + idx);
#pragma unroll 8
  for (int s = 1; s < splits; ++s) {
    const Vec w = *reinterpret_cast<const Vec*>(ws + s * total + idx);
#pragma unroll
    for (int k = 0; k < V; ++k) y.v[k] += w.v[k];
  }
  if (X2) {
#pragma unroll
    for (int k = 0; k < V; ++k) y.v[k] = y.v[k] + c * x2.v[k];
  }
  *reinterpret_cast<Vec*>(Y + idx) = y;
}

// Epilogue with inner products over a row tile x one restart.  splits > 1: Y = sum_s ws[s] (fixed
// order).  V values of a row per access (16 bytes where r and the pitch allow it), two accesses of a
// thread and their slices in flight.  Single values are four times as many, for four times the threads.
template <int V>
constexpr int kFinishThreads = V > 1 ? 128 : 512;

template <typename T, int V>
__global__ void __launch_bounds__(kFinishThreads<V>, 1024 / kFinishThreads<V>)
k_ax_finish(int64_t n, int r, int64_t ld, T* __restrict__ Y, const T* __restrict__ ws,
            int splits, double c, const T* __restrict__ X2, const T* __restrict__ P1,
            const T* __restrict__ P2, double* __restrict__ part, int q0, int b,
            const int* run, int dots_after) {
  struct alignas(V * sizeof(T)) Vec {
    T v[V];
  };
  constexpr int NT = kFinishThreads<V>;
  __shared__ T sh[2][NT / 32];
  const int j = blockIdx.y;
  const int64_t i0 = (int64_t)blockIdx.x * kRowTile;
  T d1 = T(0), d2 = T(0);  // per-CTA partials in the working type (FP64 across CTAs)
  if (!(run && *run == 0)) {
    const int rv = r / V, rows = (int)min((int64_t)kRowTile, n - i0);
    const int tile = rows * rv;
    const int64_t slice = n * ld;
    constexpr int U = 2;
    for (int e0 = threadIdx.x; e0 < tile; e0 += NT * U) {
      Vec y[U];
      int64_t idx[U];
      bool ok[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int e = e0 + NT * u;
        ok[u] = e < tile;
        const int i = ok[u] ? e / rv : 0;
        idx[u] = (i0 + i) * ld + (int64_t)j * r + (ok[u] ? e - i * rv : 0) * V;
        if (ok[u]) y[u] = *reinterpret_cast<const Vec*>((splits > 1 ? ws : Y) + idx[u]);
      }
#pragma unroll 4
      for (int s = 1; s < splits; ++s) {
        Vec w[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (ok[u]) w[u] = *reinterpret_cast<const Vec*>(ws + s * slice + idx[u]);
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (ok[u]) {
#pragma unroll
            for (int k = 0; k < V; ++k) y[u].v[k] += w[u].v[k];
          }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (!ok[u]) continue;
        auto dots = [&] {
          if (P1) {
            const Vec p = *reinterpret_cast<const Vec*>(P1 + idx[u]);
#pragma unroll
            for (int k = 0; k < V; ++k) d1 += p.v[k] * y[u].v[k];
          }
          if (P2) {
            const Vec p = *reinterpret_cast<const Vec*>(P2 + idx[u]);
#pragma unroll
            for (int k = 0; k < V; ++k) d2 += p.v[k] * y[u].v[k];
          }
        };
        if (!dots_after) dots();
        if (X2) {
          const Vec x2 = *reinterpret_cast<const Vec*>(X2 + idx[u]);
#pragma unroll
          for (int k = 0; k < V; ++k) y[u].v[k] = y[u].v[k] + (T)c * x2.v[k];
        }
        if (dots_after) dots();
        if (splits > 1 || X2) *reinterpret_cast<Vec*>(Y + idx[u]) = y[u];
      }
    }
  }
  d1 = warp_sum(d1);
  d2 = warp_sum(d2);
  if ((threadIdx.x & 31) == 0) {
    sh[0][threadIdx.x >> 5] = d1;
    sh[1][threadIdx.x >> 5] = d2;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    T v = sh[threadIdx.x][0];
#pragma unroll
    for (int w = 1; w < NT / 32; ++w) v += sh[threadIdx.x][w];
    part[((int64_t)blockIdx.x * b + j) * kNQ + q0 + threadIdx.x] = (double)v;
  }
}

inline int cdiv64(int64_t a, int64_t b) { return (int)((a + b - 1) / b); }

// Structure check of a device-resident CSR matrix before its first product: rowptr[0] = 0,
// rowptr[n] = nnz, rowptr non-decreasing (bit 0 of *bad) and every column index in [0, n)
// (bit 1).  Grid-stride; only reads inside rowptr[0..n] and colidx[0..nnz).
__global__ void k_csr_check(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colidx, int64_t n,
                            int64_t nnz, int* __restrict__ bad) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int flag = 0;
  if (t0 == 0 && (rowptr[0] != 0 || (int64_t)rowptr[n] != nnz)) flag |= 1;
  for (int64_t i = t0; i < n; i += stride)
    if (rowptr[i + 1] < rowptr[i]) flag |= 1;
  for (int64_t e = t0; e < nnz; e += stride) {
    const int32_t c = colidx[e];
    if (c < 0 || (int64_t)c >= n) flag |= 2;
  }
  if (flag) atomicOr(bad, flag);
}

}  // namespace

void launch_csr_check(const int32_t* rowptr, const int32_t* colidx, int64_t n, int64_t nnz, int* bad,
                      cudaStream_t s) {
  const int64_t work = n > nnz ? n : nnz;
  int blocks = cdiv64(work > 0 ? work : 1, 256);
  if (blocks > 152 * 8) blocks = 152 * 8;
  k_csr_check<<<blocks, 256, 0, s>>>(rowptr, colidx, n, nnz, bad);
}

namespace {

template <typename C, typename TA, int PER_SM>
int launch_gemm_cfg(const AxArgs& a, int64_t n, int cols, int64_t ld, const void* X, void* Y, void* ws, size_t ws_elems,
                    const int* run, cudaStream_t s, const ProdTune* tune) {
  using T = typename C::T;
  static SmemLimit limit;
  raise_smem_limit(limit, (const void*)k_gemm_dense<C, TA, PER_SM>, C::SMEM);
  const int gx = cdiv64(cols, C::BN), gy = cdiv64(n, C::BM);
  // split-K.  FP32 (chunks of 64 columns and more): least time of an SM, its CTAs one after the other
  // at their chunk's columns plus 64 for the start and the end of a CTA, slower by the root of the
  // occupancy that its CTAs leave unused, plus a column's worth for each slice that the finish pass
  // reads; a last short chunk fills gaps (over 99 sizes up to n = 8192 1.5 per cent from the best
  // split, 20 at most; counting whole waves of CTAs 2.4 per cent, n = 3001, 300 columns 163 for 153 us).
  // FP64 (chunks of 32, where a CTA is long): the number of chunks that fills whole waves best; each
  // further slice has to gain a per cent, for the finish pass.
  constexpr int64_t kMin = sizeof(T) == 8 ? 32 : 64;
  const int64_t tiles = (int64_t)gx * gy, slots = (int64_t)152 * PER_SM;
  const int64_t most = std::min<int64_t>({(n + kMin - 1) / kMin, 32, (int64_t)(ws_elems / ((size_t)n * (size_t)ld))});
  int64_t splits = 1;
  double best = 0.0;
  for (int64_t sp = 1; sp <= std::max<int64_t>(1, most); ++sp) {
    double gain;
    if (sizeof(T) == 8) {
      const int64_t ctas = tiles * sp, waves = (ctas + slots - 1) / slots;
      gain = (double)ctas / (double)(waves * slots) * (1.0 - 0.01 * (double)sp);
    } else {
      const int64_t kc = (cdiv64(n, (int)sp) + 31) / 32 * 32;
      const double load = (double)tiles * std::max((double)(n / kc), (double)n / (double)kc);
      const double m = std::max(1.0, std::ceil(load / 152.0));
      const double slow = std::sqrt(std::max(1.0, (double)PER_SM / m));
      const double slice = 8.0 * (double)n * cols / 6e12 * (96 * 1.9e9) / (C::BM * C::BN);
      gain = 1.0 / (m * (double)(kc + 64) * slow + (sp > 1 ? (double)sp * slice : 0.0));
    }
    if (gain > best) { best = gain; splits = sp; }
  }
  if (tune && tune->splits > 0) splits = tune->splits;  // autotuned
  splits = std::max<int64_t>(1, std::min<int64_t>(splits, ws_elems / ((size_t)n * (size_t)ld)));
  int64_t kchunk = (cdiv64(n, (int)splits) + 31) / 32 * 32;
  if (C::KIND == GA_SAME && tune && tune->kchunk > 0) kchunk = tune->kchunk;
  splits = cdiv64(n, kchunk);
  constexpr int64_t KV = C::KV;
  const bool avec = C::KIND == GA_SAME && a.lda % KV == 0 && n % KV == 0 && !((uintptr_t)a.A & 15);
  const bool xvec = ld % KV == 0 && cols % KV == 0 && !((uintptr_t)X & 15) && !((uintptr_t)Y & 15);
  dim3 grid(gx, gy, (unsigned)splits);
  k_gemm_dense<C, TA, PER_SM><<<grid, C::NT, C::SMEM, s>>>((const TA*)a.A, a.lda, (const T*)X, ld,
                                                           (T*)(splits > 1 ? ws : Y), n, cols, kchunk, avec, xvec,
                                                           GemmA8{a.a_scale, (int)((n + 127) / 128)}, run);
  return (int)splits;
}

}  // namespace

int launch_ax(const AxArgs& a, int tdtype, int64_t n, int cols, int64_t ld, const void* X, void* Y, void* ws,
              size_t ws_elems, const int* run, cudaStream_t s, const ProdTune* tune, double c, const void* X2) {
  if (a.kind == AX_DENSE) {
    // The tile is as narrow as the columns allow: 128 columns where a tile of 64 would not save a
    // padded half (FP32 A: 8 x 16 values per thread, which reads a quarter less of the stages than
    // 8 x 8: n = 8192, 512 columns 1281 -> 1174 us; the widened A need the registers: 1349 -> 1408), else
    // 64 (three CTAs per SM, whose registers hold all operands, and for FP32 A stages of 32 columns: n =
    // 8192, 64 columns 176 -> 161 us), 32, 16; FP64, whose pipes bound every size, down to 8 in steps that
    // waste at most a third (n = 2500, 10 columns: 910 us in a 64-wide tile).  Fewer than two CTAs
    // per SM at the most splits: half the rows per tile.
#define GEMM(T, TA, KIND, BM, BN, TM, TN, BK, OCC) \
  return launch_gemm_cfg<GemmCfg<T, KIND, BM, BN, TM, TN, BK>, TA, OCC>(a, n, cols, ld, X, Y, ws, ws_elems, run, s, tune)
    if (a.a_dtype == 0) {
      if (cols <= 8) GEMM(double, double, GA_SAME, 64, 8, 4, 2, 16, 6);
      if (cols <= 12) GEMM(double, double, GA_SAME, 64, 12, 4, 3, 16, 6);
      if (cols <= 16) GEMM(double, double, GA_SAME, 64, 16, 4, 4, 16, 6);
      if (cols <= 24) GEMM(double, double, GA_SAME, 64, 24, 4, 3, 16, 4);
      if (cols <= 32) GEMM(double, double, GA_SAME, 64, 32, 4, 4, 16, 4);
      GEMM(double, double, GA_SAME, 64, 64, 4, 4, 16, 2);
    }
    const bool wide = cols > 64 && (cols + 127) / 128 * 2 <= (cols + 63) / 64;
#define GEMM_WIDTHS(TA, KIND, TNW, BK64)                          \
  if (wide) GEMM(float, TA, KIND, 128, 128, 8, TNW, 16, 2);       \
  if (cols > 32) GEMM(float, TA, KIND, 128, 64, 8, 8, BK64, 3);   \
  if (cols > 16) GEMM(float, TA, KIND, 128, 32, 8, 4, 32, 3);     \
  GEMM(float, TA, KIND, 128, 16, 4, 4, 32, 3)
    if (a.a_dtype == 3) { GEMM_WIDTHS(__nv_fp8_storage_t, GA_FP8, 8, 16); }
    if (a.a_dtype == 2 && a.sym) { GEMM_WIDTHS(__nv_bfloat16, GA_BF16_SYM, 8, 16); }
    if (a.a_dtype == 2) { GEMM_WIDTHS(__nv_bfloat16, GA_BF16, 8, 16); }
    if ((int64_t)cdiv64(n, 128) * cdiv64(cols, 64) * std::min<int64_t>(n / 64, 32) < 2 * 152) {
      if (cols > 32) GEMM(float, float, GA_SAME, 64, 64, 4, 8, 16, 4);
      if (cols > 16) GEMM(float, float, GA_SAME, 64, 32, 4, 4, 32, 4);
      GEMM(float, float, GA_SAME, 64, 16, 4, 4, 32, 6);
    }
    GEMM_WIDTHS(float, GA_SAME, 16, 32);
#undef GEMM_WIDTHS
#undef GEMM
  }
  // CSR
  const uintptr_t all = (uintptr_t)X | (uintptr_t)Y | (uintptr_t)X2;
#define SPMM(TV, T, V, L)                                                                                            \
  k_spmm_csr<TV, T, V, L><<<dim3(cdiv64(n, 8 * (32 / L)), cdiv64(cols, V * L)), 256, 0, s>>>(                        \
      a.rowptr, a.colidx, (const TV*)a.vals, (const T*)X, ld, (T*)Y, n, cols, (T)c, (const T*)X2, run)
#define SPMM_L(TV, T, V)                    \
  if (cols <= 4 * V) SPMM(TV, T, V, 4);     \
  else if (cols <= 8 * V) SPMM(TV, T, V, 8); \
  else if (cols <= 16 * V) SPMM(TV, T, V, 16); \
  else SPMM(TV, T, V, 32)
#define SPMM_V(TV, T)                                                                                   \
  if (sizeof(T) == 4 && cols % 4 == 0 && ld % 4 == 0 && !(all & 15)) { SPMM_L(TV, T, (16 / (int)sizeof(T))); } \
  else if (cols % 2 == 0 && ld % 2 == 0 && !(all & (2 * sizeof(T) - 1))) { SPMM_L(TV, T, 2); }          \
  else { SPMM_L(TV, T, 1); }
  if (a.lda > kCsrAhead) {  // entries one at a time, the next index at most the row's end
#define SPMM_ONE(TV, T)                                                                                              \
  k_spmm_csr<TV, T, 1, 32, 1><<<dim3(cdiv64(n, 8), cdiv64(cols, 32)), 256, 0, s>>>(                                  \
      a.rowptr, a.colidx, (const TV*)a.vals, (const T*)X, ld, (T*)Y, n, cols, (T)c, (const T*)X2, run)
    if (tdtype == 0) {
      if (a.v_dtype == 0) SPMM_ONE(double, double); else SPMM_ONE(float, double);
    } else {
      if (a.v_dtype == 0) SPMM_ONE(double, float); else SPMM_ONE(float, float);
    }
#undef SPMM_ONE
    return 1;
  }
  if (tdtype == 0) {
    if (a.v_dtype == 0) { SPMM_V(double, double) } else { SPMM_V(float, double) }
  } else {
    if (a.v_dtype == 0) { SPMM_V(double, float) } else { SPMM_V(float, float) }
  }
#undef SPMM_V
#undef SPMM_L
#undef SPMM
  return 1;
}

int launch_ax_finish_impl(int tdtype, const Dims& d, void* Y, const void* ws, int splits,
                          double c, const void* X2, const void* P1, const void* P2,
                          double* part, int q0, const int* run, cudaStream_t s, int dots_after) {
  dim3 grid(cdiv64(d.n, kRowTile), d.b);
  const int v = tdtype == 0 ? 2 : 4;
  const uintptr_t all = (uintptr_t)Y | (uintptr_t)ws | (uintptr_t)X2 | (uintptr_t)P1 | (uintptr_t)P2;
  if (!P1 && !P2 && d.ld == d.N) {  // no inner products: one flat array
    const int64_t total = d.n * d.N;
    const bool flat = total % v == 0 && !(all & 15);  // the slices start on 16 bytes as well
#define SUM(T, V)                                                                                            \
  k_ax_sum<T, V><<<cdiv64(total, 256 * V), 256, 0, s>>>(total, (T*)Y, (const T*)ws, splits, (T)c, (const T*)X2, run)
    if (tdtype == 0) {
      if (flat) SUM(double, 2); else SUM(double, 1);
    } else {
      if (flat) SUM(float, 4); else SUM(float, 1);
    }
#undef SUM
    return grid.x;
  }
  const bool vec = d.r % v == 0 && d.ld % v == 0 && !(all & 15);
#define FIN(T, V)                                                                                                    \
  k_ax_finish<T, V><<<grid, kFinishThreads<V>, 0, s>>>(d.n, d.r, d.ld, (T*)Y, (const T*)ws, splits, c, (const T*)X2, (const T*)P1, \
                                         (const T*)P2, part, q0, d.b, run, dots_after)
  if (tdtype == 0) {
    if (vec) FIN(double, 2); else FIN(double, 1);
  } else {
    if (vec) FIN(float, 4); else FIN(float, 1);
  }
#undef FIN
  return grid.x;
}

// ---------------------------------------------------------------------------------------
// The paper's normalized graph Laplacian L = I - D^-1/2 A D^-1/2, d_i = sum_j a_ij (Sec. 2.2):
// the scaling s_i = d_i^-1/2 (0 for rows of zero degree) and the operator -D^-1/2 A D^-1/2
// in the factor type, applied as L X = X + (-D^-1/2 A D^-1/2) X.
// ---------------------------------------------------------------------------------------
namespace {

template <typename TA>
__global__ void k_degree_scale(int kind, const TA* __restrict__ A, int64_t lda, const int32_t* __restrict__ rowptr,
                               int64_t n, double* __restrict__ s) {
  // one warp per row, FP64 sum in a fixed order (lane stride, then a fixed butterfly)
  const int lane = threadIdx.x & 31;
  const int64_t i = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= n) return;
  double acc = 0.0;
  if (kind == AX_DENSE) {
    for (int64_t k = lane; k < n; k += 32) acc += (double)ld_a(A + i * lda + k);
  } else {
    for (int64_t e = rowptr[i] + lane; e < rowptr[i + 1]; e += 32) acc += (double)A[e];
  }
  acc = warp_sum(acc);
  if (lane == 0) s[i] = acc > 0.0 ? 1.0 / sqrt(acc) : 0.0;
}

template <typename TA, typename T>
__global__ void k_scaled_neg_csr(const TA* __restrict__ vals, const int32_t* __restrict__ rowptr,
                                 const int32_t* __restrict__ colidx, int64_t n, const double* __restrict__ s,
                                 T* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int64_t i = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= n) return;
  for (int64_t e = rowptr[i] + lane; e < rowptr[i + 1]; e += 32)
    out[e] = (T)(-(s[i] * (double)vals[e] * s[colidx[e]]));
}

template <typename TA, typename T>
__global__ void k_scaled_neg_dense(const TA* __restrict__ A, int64_t lda, int64_t n, const double* __restrict__ s,
                                   T* __restrict__ out) {
  const int64_t total = n * n;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / n, k = e % n;
    out[e] = (T)(-(s[i] * (double)ld_a(A + i * lda + k) * s[k]));
  }
}

}  // namespace

void launch_normalized_adjacency(const AxArgs& a, int tdtype, int64_t n, double* s, void* out, cudaStream_t st) {
  const int rb = cdiv64(n, 8);
  if (a.kind == AX_DENSE) {
    const int blocks = (int)std::min<int64_t>(cdiv64(n * n, 256), 152 * 32);
    if (a.a_dtype == 0) {
      k_degree_scale<double><<<rb, 256, 0, st>>>(AX_DENSE, (const double*)a.A, a.lda, nullptr, n, s);
      if (tdtype == 0) k_scaled_neg_dense<double, double><<<blocks, 256, 0, st>>>((const double*)a.A, a.lda, n, s, (double*)out);
      else k_scaled_neg_dense<double, float><<<blocks, 256, 0, st>>>((const double*)a.A, a.lda, n, s, (float*)out);
    } else {
      k_degree_scale<float><<<rb, 256, 0, st>>>(AX_DENSE, (const float*)a.A, a.lda, nullptr, n, s);
      if (tdtype == 0) k_scaled_neg_dense<float, double><<<blocks, 256, 0, st>>>((const float*)a.A, a.lda, n, s, (double*)out);
      else k_scaled_neg_dense<float, float><<<blocks, 256, 0, st>>>((const float*)a.A, a.lda, n, s, (float*)out);
    }
    return;
  }
  if (a.v_dtype == 0) {
    k_degree_scale<double><<<rb, 256, 0, st>>>(AX_CSR, (const double*)a.vals, 0, a.rowptr, n, s);
    if (tdtype == 0) k_scaled_neg_csr<double, double><<<rb, 256, 0, st>>>((const double*)a.vals, a.rowptr, a.colidx, n, s, (double*)out);
    else k_scaled_neg_csr<double, float><<<rb, 256, 0, st>>>((const double*)a.vals, a.rowptr, a.colidx, n, s, (float*)out);
  } else {
    k_degree_scale<float><<<rb, 256, 0, st>>>(AX_CSR, (const float*)a.vals, 0, a.rowptr, n, s);
    if (tdtype == 0) k_scaled_neg_csr<float, double><<<rb, 256, 0, st>>>((const float*)a.vals, a.rowptr, a.colidx, n, s, (double*)out);
    else k_scaled_neg_csr<float, float><<<rb, 256, 0, st>>>((const float*)a.vals, a.rowptr, a.colidx, n, s, (float*)out);
  }
}

}  // namespace snmf
