// Graph pre-processing for Graph-SNMPBB and clustering scores on the GPU.
//
//   snmf_knn_graph      k nearest neighbours of every point (brute force, squared Euclidean
//                       distance, ties: lower index first), self-tuning scale s_i = distance to
//                       the sigma_rank-th neighbour, S_ij = exp(-d_ij^2 / (s_i s_j)) on the kNN
//                       pairs, symmetrised as max(S, S^T), degrees d_i = sum_j S_ij and the CSR
//                       matrix A^ = D^-1/2 S D^-1/2 (columns ascending per row).
//   snmf_cluster_assign label_i = argmax_c of the restart's H factor row (ties: lowest c).
//   snmf_cluster_scores contingency table of two labelings on the device; the adjusted Rand
//                       index and the accuracy of the best one-to-one label matching from it
//                       on the host (Hungarian method on the small table).
// Every reduction is in a fixed order: the outputs do not depend on thread scheduling.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <limits>
#include <vector>

#include "../../include/snmf.h"
#include "ax_tc.cuh"
#include "common.cuh"

namespace snmf {
namespace {

constexpr int QB = 64;    // queries per CTA
constexpr int CB = 128;   // candidates per tile
constexpr int DT = 32;    // coordinates staged per round
constexpr int KMAX = 32;
// the dimensions that the library takes (rows of QB + 64 points in 200 KB)
constexpr size_t kKnnMaxBytes = 200 * 1024;

// A list of the 32 best (distance, index) pairs, sorted, lane t holding rank t: insertion of (v, vi)
// by one warp.
__device__ __forceinline__ void knn_insert(float& kd, int32_t& ki, float v, int32_t vi) {
  const int pos = __popc(__ballot_sync(0xffffffffu, kd < v || (kd == v && ki < vi)));
  const float ud = __shfl_up_sync(0xffffffffu, kd, 1);
  const int32_t ui = __shfl_up_sync(0xffffffffu, ki, 1);
  const int lane = threadIdx.x & 31;
  if (lane > pos) {
    kd = ud;
    ki = ui;
  } else if (lane == pos) {
    kd = v;
    ki = vi;
  }
}

}  // namespace
}  // namespace snmf

#include "knn_tc.cuh"

namespace snmf {
namespace {

// The k nearest of the candidates [z per, (z + 1) per) for the 64 queries of CTA (x, z): partial
// lists at [z][n][k], sorted by distance and then index (empty slots are (inf, INT_MAX)).  Distances of
// a 128 x 64 tile, 8 candidates x 4 queries per thread, two candidates per instruction: sum over t
// ascending of (q_t - c_t)^2 with one FMA each, candidates staged negated.  A distance not above the
// query's k-th so far goes to the query's buffer in shared memory; after the tile its warp (eight queries
// each) inserts the buffer, in any order with the same result.  A non-finite distance counts as +inf and raises *bad.  Bound by the FP32 pipes (2 n^2 d
// lane operations): n = 20000, d = 64, k = 10 2.94 ms (23.1 ms with one thread per query and the list
// updated for every candidate).  For few or wide points, and where the filter (knn_tc.cuh) gave up.
struct KnnSmem {
  float q[2][DT][QB];
  float c[2][DT][CB];
  float bd[QB][CB + 1];
  uint8_t bi[QB][CB];
  float thr[QB];
  int cnt[QB];
};

__global__ void __launch_bounds__(256, 2)
k_knn(const float* __restrict__ X, int64_t n, int d, int k, int64_t per, bool vec, int32_t* __restrict__ nbr,
      float* __restrict__ nd2, int* __restrict__ bad, const int* __restrict__ only_if) {
  if (only_if && !*only_if) return;
  extern __shared__ __align__(16) unsigned char knn_raw[];
  KnnSmem& S = *reinterpret_cast<KnnSmem*>(knn_raw);
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  const int64_t q0 = (int64_t)blockIdx.x * QB;
  const int64_t cb = (int64_t)blockIdx.y * per, ce = min(n, cb + per);
  const int lane = t & 31, w8 = (t >> 5) * 8;  // the warp's queries w8 .. w8 + 7
  float kd[8];
  int32_t ki[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    kd[u] = INFINITY;
    ki[u] = INT_MAX;
  }
  if (t < QB) {
    S.thr[t] = INFINITY;
    S.cnt[t] = 0;
  }
  const int nd = (d + DT - 1) / DT;
  const int rounds = ce > cb ? (int)((ce - cb + CB - 1) / CB) * nd : 0;
  // staging: thread t loads 8 coordinates of query t % 64 and 16 of candidate t % 128
  float rq[8], rc[16];
  auto load = [&](int s) {
    const int t0 = s % nd * DT;
    const int64_t qi = q0 + (t & 63), ci = cb + (int64_t)(s / nd) * CB + (t & 127);
    const int tq = t0 + (t >> 6) * 8, tc = t0 + (t >> 7) * 16;
    auto get = [&](float* r, int m, int64_t i, bool on, int tt) {
#pragma unroll
      for (int u = 0; u < m; u += 4) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        const float* p = X + i * d + tt + u;
        if (on && vec) {
          if (tt + u < d) v = *reinterpret_cast<const float4*>(p);
        } else if (on) {
          if (tt + u < d) v.x = p[0];
          if (tt + u + 1 < d) v.y = p[1];
          if (tt + u + 2 < d) v.z = p[2];
          if (tt + u + 3 < d) v.w = p[3];
        }
        r[u] = v.x; r[u + 1] = v.y; r[u + 2] = v.z; r[u + 3] = v.w;
      }
    };
    get(rq, 8, qi, qi < n, tq);
    get(rc, 16, ci, ci < ce, tc);
  };
  auto put = [&](int s) {
#pragma unroll
    for (int u = 0; u < 8; ++u) S.q[s & 1][(t >> 6) * 8 + u][t & 63] = rq[u];
#pragma unroll
    for (int u = 0; u < 16; ++u) S.c[s & 1][(t >> 7) * 16 + u][t & 127] = -rc[u];
  };
  float2 acc[4][4];  // [query][candidate pair]
  if (rounds > 0) {
    load(0);
    put(0);
  }
  __syncthreads();
  for (int s = 0; s < rounds; ++s) {
    if (s + 1 < rounds) load(s + 1);
    const int ch = s % nd;
    if (ch == 0) {
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[a][c] = make_float2(0.f, 0.f);
    }
    const int dt = min(DT, d - ch * DT);
    const float* qp = &S.q[s & 1][0][4 * tx];
    const float* cp = &S.c[s & 1][0][4 * ty];
#pragma unroll 4
    for (int u = 0; u < dt; ++u) {
      const float4 q4 = *reinterpret_cast<const float4*>(qp + u * QB);
      const float4 ca = *reinterpret_cast<const float4*>(cp + u * CB);
      const float4 cc = *reinterpret_cast<const float4*>(cp + u * CB + 64);
      const float qs[4] = {q4.x, q4.y, q4.z, q4.w};
      const float2 c2[4] = {make_float2(ca.x, ca.y), make_float2(ca.z, ca.w), make_float2(cc.x, cc.y),
                            make_float2(cc.z, cc.w)};
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const float2 qq = make_float2(qs[a], qs[a]);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float2 df = __fadd2_rn(qq, c2[c]);
          acc[a][c] = __ffma2_rn(df, df, acc[a][c]);
        }
      }
    }
    if (ch == nd - 1) {
      const int64_t c0 = cb + (int64_t)(s / nd) * CB;
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const int ql = 4 * tx + a;
        const int64_t q = q0 + ql;
        const float thr = S.thr[ql];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const int cl = (c >> 2) * 64 + 4 * ty + (c & 3);
          const int64_t j = c0 + cl;
          float v = c & 1 ? acc[a][c >> 1].y : acc[a][c >> 1].x;
          if (q >= n || j >= ce || j == q) continue;
          if (!isfinite(v)) {
            v = INFINITY;
            atomicOr(bad, 1);
          }
          if (v <= thr) {
            const int pos = atomicAdd(&S.cnt[ql], 1);  // at most one entry per candidate of the tile
            S.bd[ql][pos] = v;
            S.bi[ql][pos] = (uint8_t)cl;
          }
        }
      }
      __syncthreads();
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int m = S.cnt[w8 + u];
        if (!m) continue;
        for (int e = 0; e < m; ++e) knn_insert(kd[u], ki[u], S.bd[w8 + u][e], (int32_t)(c0 + S.bi[w8 + u][e]));
        __syncwarp();
        if (lane == k - 1) {
          S.thr[w8 + u] = kd[u];
          S.cnt[w8 + u] = 0;
        }
      }
    }
    if (s + 1 < rounds) put(s + 1);  // the other buffer: its readers passed the last barrier
    __syncthreads();
  }
  if (lane < k) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int64_t q = q0 + w8 + u;
      if (q >= n) continue;
      const int64_t o = ((int64_t)blockIdx.y * n + q) * k + lane;
      nbr[o] = ki[u];
      nd2[o] = kd[u];
    }
  }
}

// one warp per query: the k best of its `parts` partial lists
__global__ void __launch_bounds__(256) k_knn_merge(const int32_t* __restrict__ pi, const float* __restrict__ pd, int64_t n,
                                                   int k, int parts, int32_t* __restrict__ nbr, float* __restrict__ nd2,
                                                   const int* __restrict__ only_if) {
  if (only_if && !*only_if) return;
  const int lane = threadIdx.x & 31;
  const int64_t q = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (q >= n) return;
  float kd = INFINITY;
  int32_t ki = INT_MAX;
  for (int z = 0; z < parts; ++z) {
    const int64_t o = ((int64_t)z * n + q) * k + lane;
    const float v = lane < k ? pd[o] : INFINITY;
    const int32_t vi = lane < k ? pi[o] : INT_MAX;
    for (int u = 0; u < k; ++u) knn_insert(kd, ki, __shfl_sync(0xffffffffu, v, u), __shfl_sync(0xffffffffu, vi, u));
  }
  if (lane < k) {
    nbr[q * k + lane] = ki;
    nd2[q * k + lane] = kd;
  }
}

// scale s_i, directed similarities, in-degree counts
__global__ void k_knn_sim(const int32_t* __restrict__ nbr, const float* __restrict__ nd2, int64_t n, int k,
                          int sigma_rank, float* __restrict__ sval, int32_t* __restrict__ cnt,
                          int* __restrict__ bad) {
  const int64_t total = n * k;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / k;
    const int32_t j = nbr[e];
    const float si = sqrtf(nd2[i * k + sigma_rank - 1]);
    const float sj = sqrtf(nd2[(int64_t)j * k + sigma_rank - 1]);
    const float v = expf(-nd2[e] / (si * sj));
    if (!(si * sj > 0.f) || !isfinite(v)) atomicOr(bad, 1);  // zero scale: duplicate points
    sval[e] = v;
    atomicAdd(&cnt[j], 1);  // the reverse entry (j, i)
  }
}

// exclusive scan of v[0..n) (+ k per element) into out[0..n], one block, fixed order
__global__ void __launch_bounds__(1024) k_scan(const int32_t* __restrict__ v, int64_t n, int add,
                                               int32_t* __restrict__ out) {
  __shared__ int64_t part[1024];
  const int64_t per = (n + blockDim.x - 1) / blockDim.x;
  const int64_t b = threadIdx.x * per, e = b + per < n ? b + per : n;
  int64_t s = 0;
  for (int64_t i = b; i < e; ++i) s += v[i] + add;
  part[threadIdx.x] = s;
  __syncthreads();
  if (threadIdx.x < 32) {  // 32 sums a lane, then a scan over the lanes
    int64_t* p = part + threadIdx.x * 32;
    int64_t sum = 0;
    for (int t = 0; t < 32; ++t) sum += p[t];
    int64_t run = sum;
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t x = __shfl_up_sync(0xffffffffu, run, o);
      if ((int)threadIdx.x >= o) run += x;
    }
    if (threadIdx.x == 31) out[n] = (int32_t)run;
    run -= sum;
    for (int t = 0; t < 32; ++t) {
      const int64_t x = p[t];
      p[t] = run;
      run += x;
    }
  }
  __syncthreads();
  int64_t run = part[threadIdx.x];
  for (int64_t i = b; i < e; ++i) {
    out[i] = (int32_t)run;
    run += v[i] + add;
  }
}

// both directions of every kNN pair into the rows' slots (order within a row arbitrary)
__global__ void k_knn_fill(const int32_t* __restrict__ nbr, const float* __restrict__ sval, int64_t n, int k,
                           const int32_t* __restrict__ off, int32_t* __restrict__ fill, int32_t* __restrict__ erow,
                           int32_t* __restrict__ ecol, float* __restrict__ eval) {
  const int64_t total = n * k;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int32_t i = (int32_t)(e / k), j = nbr[e];
    const float s = sval[e];
    const int32_t a = off[i] + atomicAdd(&fill[i], 1);
    erow[a] = i;
    ecol[a] = j;
    eval[a] = s;
    const int32_t bslot = off[j] + atomicAdd(&fill[j], 1);
    erow[bslot] = j;
    ecol[bslot] = i;
    eval[bslot] = s;
  }
}

// One thread per entry; a row holds each column at most twice (the forward kNN entry and the reverse
// one).  pass 0: an entry represents its column when no other entry of the column has a larger
// value (or the same value at a lower position); flags and counts.  pass 1: the representative's
// rank among the row's representatives by column is its CSR position.  (A warp per row left the few
// long rows of a graph's hubs to one warp each: 189 us at n = 20000, k = 10.)
__global__ void k_knn_dedupe(const int32_t* __restrict__ off, const int32_t* __restrict__ erow,
                             const int32_t* __restrict__ ecol, const float* __restrict__ eval, int64_t entries, int pass,
                             uint8_t* __restrict__ erep, int32_t* __restrict__ cntu, const int32_t* __restrict__ rowptr,
                             int32_t* __restrict__ colidx, float* __restrict__ sout) {
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= entries) return;
  const int32_t i = erow[x], cx = ecol[x], b = off[i], e = off[i + 1];
  const float vx = eval[x];
  if (pass == 0) {
    bool rep = true;
#pragma unroll 4
    for (int32_t y = b; y < e; ++y) {
      const int32_t cy = ecol[y];
      const float vy = eval[y];
      if (cy == cx && y != x && (vy > vx || (vy == vx && y < x))) rep = false;
    }
    erep[x] = rep ? 1 : 0;
    if (rep) atomicAdd(&cntu[i], 1);
  } else if (erep[x]) {
    int rank = 0;
#pragma unroll 4
    for (int32_t y = b; y < e; ++y) rank += (erep[y] && ecol[y] < cx) ? 1 : 0;
    colidx[rowptr[i] + rank] = cx;
    sout[rowptr[i] + rank] = vx;
  }
}

// degrees (fixed order: column order, lane-strided then a fixed butterfly)
__global__ void k_knn_degree(const int32_t* __restrict__ rowptr, const float* __restrict__ sv, int64_t n,
                             float* __restrict__ deg) {
  const int lane = threadIdx.x & 31;
  const int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (i >= n) return;
  double s = 0.0;
  for (int32_t e = rowptr[i] + lane; e < rowptr[i + 1]; e += 32) s += (double)sv[e];
  s = warp_sum(s);
  if (lane == 0) deg[i] = (float)s;
}

__global__ void k_knn_normalize(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colidx,
                                const float* __restrict__ sv, const float* __restrict__ deg, int64_t n,
                                float* __restrict__ ahat) {
  const int lane = threadIdx.x & 31;
  const int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (i >= n) return;
  for (int32_t e = rowptr[i] + lane; e < rowptr[i + 1]; e += 32)
    ahat[e] = (float)((double)sv[e] / sqrt((double)deg[i] * (double)deg[colidx[e]]));
}

__global__ void k_contingency(const int32_t* __restrict__ truth, const int32_t* __restrict__ pred, int64_t n, int k1,
                              int k2, unsigned long long* __restrict__ table, int* __restrict__ bad) {
  extern __shared__ unsigned int hist[];
  for (int e = threadIdx.x; e < k1 * k2; e += blockDim.x) hist[e] = 0u;
  __syncthreads();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int a = truth[i], b = pred[i];
    if (a < 0 || a >= k1 || b < 0 || b >= k2) { atomicOr(bad, 1); continue; }
    atomicAdd(&hist[a * k2 + b], 1u);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < k1 * k2; e += blockDim.x)
    if (hist[e]) atomicAdd(&table[e], (unsigned long long)hist[e]);
}

template <typename T>
__global__ void k_assign(const T* __restrict__ F, int64_t n, int64_t ld, int64_t col0, int r, int32_t* __restrict__ lab) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const T* row = F + i * ld + col0;
    int best = 0;
    T bv = row[0];
    for (int c = 1; c < r; ++c)
      if (row[c] > bv) { bv = row[c]; best = c; }
    lab[i] = best;
  }
}

// Candidate ranges (partial lists per query): the number that fills whole waves of CTAs (two per
// SM) best, each further list worth two per cent of merging, none shorter than 512 candidates.
int knn_parts(int64_t n) {
  const int64_t qb = (n + QB - 1) / QB, most = std::min<int64_t>(16, std::max<int64_t>(1, n / 512));
  int parts = 1;
  double best = 0.0;
  for (int64_t p = 1; p <= most; ++p) {
    const int64_t waves = (qb * p + 2 * 152 - 1) / (2 * 152);
    const double gain = (double)(qb * p) / (double)(waves * 2 * 152) * (1.0 - 0.02 * (double)p);
    if (gain > best) { best = gain; parts = (int)p; }
  }
  return parts;
}

// The filter: for rows that two CTAs of an SM hold beside their rings, and where its launches are worth
// it (whole call, d = 16, k = 10: n = 1024 256 us without it and 224 with it; n = 5001, d = 33, k = 12
// 511 and 315; n = 20000, d = 64 3250 and 890); up to 4 million points, whose candidate lists are 4 GB.
bool knn_tc_rule(int64_t n, int d) { return d <= KT_MAXD && n >= 1024 && n < (1 << 22); }

// Candidate ranges of its passes: about four waves of CTAs (n = 20000, d = 64: 1401 us with one range,
// 1171 with seven), none shorter than 256.
int knn_tc_parts(int64_t n) {
  const int64_t qt = (n + KT_Q - 1) / KT_Q;
  return (int)std::max<int64_t>(1, std::min<int64_t>(KT_PARTS, std::min<int64_t>(1216 / qt, n / 256)));
}

// Pass 0 over every second point halves it and doubles the candidates (n = 20000, d = 64, k = 10: pass 0
// 439 to 325 us, exact distances 24 to 42); every fourth would save another 60 us, but a cluster of
// fewer than 4 k points would then bring in all points.
int knn_tc_stride(int64_t n) { return n >= 4096 ? 2 : 1; }

struct KnnWork {
  int parts, tc_parts;  // tc_parts: 0 without the filter
  int32_t* pi;          // partial lists
  float* pd;
  float *Y, *nrm, *nrm0, *kth, *ctr, *lists;  // nrm, nrm0: room for a whole last tile
  int32_t* cand;
  int *ncand, *bad, *dense, *err;
};

template <int PASS, int KR>
cudaError_t launch_knn_pass(const CUtensorMap& map, const CUtensorMap& cmap, const float* cnrm, int stride, int64_t n, int d,
                            int k, const KnnWork& w, cudaStream_t s) {
  static SmemLimit limit;
  if (const cudaError_t e = raise_smem_limit(limit, (const void*)k_knn_tc<PASS, KR>, knn_tc_smem(KT_MAXD))) return e;
  const int64_t nc = (n + stride - 1) / stride, per = ((nc + w.tc_parts - 1) / w.tc_parts + KT_C - 1) / KT_C * KT_C;
  dim3 grid((unsigned)((n + KT_Q - 1) / KT_Q), w.tc_parts);
  k_knn_tc<PASS, KR><<<grid, KT_THREADS, knn_tc_smem(d), s>>>(map, cmap, w.nrm, cnrm, nc, stride, w.kth, n, d, k, per,
                                                              w.lists, w.cand, w.ncand, w.dense, w.err);
  return cudaGetLastError();
}

cudaError_t launch_knn(const float* X, int64_t n, int d, int k, const KnnWork& w, int32_t* nbr, float* nd2, cudaStream_t s) {
  static SmemLimit limit;
  if (const cudaError_t e = raise_smem_limit(limit, (const void*)k_knn, sizeof(KnnSmem))) return e;
  const bool vec = d % 4 == 0 && !((uintptr_t)X & 15);
  const unsigned mb = (unsigned)((n + 7) / 8);
  const int* only_if = nullptr;
  CUtensorMap map, map0;
  const int dp = (d + 31) / 32 * 32;
  const int st = knn_tc_stride(n);
  if (w.tc_parts && make_map_f32_tile(&map, w.Y, dp, n, dp, KT_C) &&
      make_map_f32_tile(&map0, w.Y, dp, (n + st - 1) / st, (int64_t)st * dp, KT_C)) {
    k_knn_center<<<1, 1024, 0, s>>>(X, n, d, w.ctr);
    k_knn_prep<<<mb, 256, 0, s>>>(X, n, d, dp, w.ctr, w.Y, w.nrm, w.kth, w.ncand, st, w.nrm0, w.dense);
    cudaError_t e = k <= 16 ? launch_knn_pass<0, 16>(map, map0, w.nrm0, st, n, d, k, w, s)
                            : launch_knn_pass<0, 32>(map, map0, w.nrm0, st, n, d, k, w, s);
    if (e != cudaSuccess) return e;
    k_knn_bound<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(w.lists, w.nrm, n, k, 2 * w.tc_parts, w.kth);
    e = launch_knn_pass<1, 1>(map, map, w.nrm, 1, n, d, k, w, s);
    if (e != cudaSuccess) return e;
    if (d % 8 == 0 && !((uintptr_t)X & 31)) k_knn_exact<8><<<mb, 256, 0, s>>>(X, n, d, k, w.cand, w.ncand, nbr, nd2, w.dense);
    else if (vec) k_knn_exact<4><<<mb, 256, 0, s>>>(X, n, d, k, w.cand, w.ncand, nbr, nd2, w.dense);
    else k_knn_exact<1><<<mb, 256, 0, s>>>(X, n, d, k, w.cand, w.ncand, nbr, nd2, w.dense);
    only_if = w.dense;
  }
  const int64_t per = ((n + w.parts - 1) / w.parts + CB - 1) / CB * CB;
  dim3 grid((unsigned)((n + QB - 1) / QB), w.parts);
  k_knn<<<grid, 256, sizeof(KnnSmem), s>>>(X, n, d, k, per, vec, w.parts > 1 ? w.pi : nbr, w.parts > 1 ? w.pd : nd2, w.bad,
                                           only_if);
  if (w.parts > 1) k_knn_merge<<<mb, 256, 0, s>>>(w.pi, w.pd, n, k, w.parts, nbr, nd2, only_if);
  return cudaGetLastError();
}

// Best one-to-one matching maximising the matched count: the Hungarian method with potentials
// on the square cost matrix -T (padded with zeros), shortest augmenting paths one row at a
// time.  Returns the matched total.
long long max_matching(const std::vector<long long>& T, int rows, int cols) {
  const int m = std::max(rows, cols);
  auto cost = [&](int a, int b) -> long long { return (a < rows && b < cols) ? -T[(size_t)a * cols + b] : 0; };
  const long long INF = std::numeric_limits<long long>::max() / 4;
  std::vector<long long> u(m + 1, 0), v(m + 1, 0);
  std::vector<int> match(m + 1, 0), way(m + 1, 0);  // match[col] = row (1-based; 0 = free)
  for (int a = 1; a <= m; ++a) {
    match[0] = a;
    int j0 = 0;
    std::vector<long long> minv(m + 1, INF);
    std::vector<char> used(m + 1, 0);
    do {
      used[j0] = 1;
      const int a0 = match[j0];
      long long delta = INF;
      int j1 = 0;
      for (int j = 1; j <= m; ++j) {
        if (used[j]) continue;
        const long long cur = cost(a0 - 1, j - 1) - u[a0] - v[j];
        if (cur < minv[j]) { minv[j] = cur; way[j] = j0; }
        if (minv[j] < delta) { delta = minv[j]; j1 = j; }
      }
      for (int j = 0; j <= m; ++j) {
        if (used[j]) { u[match[j]] += delta; v[j] -= delta; }
        else minv[j] -= delta;
      }
      j0 = j1;
    } while (match[j0] != 0);
    do {
      const int j1 = way[j0];
      match[j0] = match[j1];
      j0 = j1;
    } while (j0);
  }
  long long total = 0;
  for (int j = 1; j <= m; ++j)
    if (match[j] >= 1 && match[j] <= rows && j <= cols) total += T[(size_t)(match[j] - 1) * cols + (j - 1)];
  return total;
}

}  // namespace
}  // namespace snmf

using namespace snmf;

extern "C" snmf_status snmf_knn_graph(const float* X, int64_t n, int d, int k, int sigma_rank, int32_t* rowptr,
                                      int32_t* colidx, float* a_hat, float* s_values, float* degree,
                                      int64_t capacity, int64_t* nnz, void* stream) {
  if (!X || !rowptr || !colidx || !a_hat || !nnz || n < 2 || d < 1 || d > 1024 || k < 1 || k > KMAX || k >= n ||
      sigma_rank < 1 || sigma_rank > k || 2 * n * (int64_t)k > INT_MAX)
    return SNMF_ERR_ARG;
  if ((size_t)(QB + 64) * (d + 1) * sizeof(float) > kKnnMaxBytes) return SNMF_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  const int64_t nk = n * k;
  // the call's workspace in one piece
  KnnWork w{};
  w.parts = knn_parts(n);
  w.tc_parts = knn_tc_rule(n, d) ? knn_tc_parts(n) : 0;
  unsigned char* ws = nullptr;
  size_t bytes = 0;
  auto take = [&](size_t b) {
    const size_t at = bytes;
    bytes += (b + 255) / 256 * 256;
    return at;
  };
  const size_t o_nbr = take(nk * 4), o_nd2 = take(nk * 4), o_sval = take(nk * 4), o_cnt = take(n * 4), o_fill = take(n * 4),
               o_off = take((n + 1) * 4), o_cntu = take(n * 4), o_erow = take(2 * nk * 4), o_ecol = take(2 * nk * 4), o_eval = take(2 * nk * 4),
               o_sv = take(s_values ? 0 : 2 * nk * 4), o_dg = take(degree ? 0 : n * 4), o_erep = take(2 * nk),
               o_bad = take(12), always = bytes;
  size_t o_y, o_nrm, o_nrm0, o_kth, o_ctr, o_ncand, o_lists, o_cand, o_pi, o_pd;
  auto plan = [&] {  // the rest with or without the filter
    bytes = always;
    const int64_t dp = w.tc_parts ? (d + 31) / 32 * 32 : 0;
    o_y = take(n * dp * 4);
    o_nrm = take(dp ? (n + KT_C) * 4 : 0);
    o_nrm0 = take(dp ? (n + KT_C) * 4 : 0);
    o_kth = take(dp ? n * 4 : 0);
    o_ctr = take(dp * 4);
    o_ncand = take(dp ? n * 4 : 0);
    // k_knn's partial lists come after the filter's lists and candidates are done with
    o_lists = o_pi = bytes;
    o_cand = o_lists + (2 * w.tc_parts * nk * 4 + 255) / 256 * 256;
    const size_t part = w.parts > 1 ? (w.parts * nk * 4 + 255) / 256 * 256 : 0;
    o_pd = o_pi + part;
    take(std::max((o_cand - o_lists) + (dp ? n * KT_CAP * 4 : 0), 2 * part));
  };
  auto cleanup = [&] { workspace_free(ws, s); };
  snmf_status st = SNMF_OK;
#define KCK(call)                                                                                        \
  do {                                                                                                   \
    const cudaError_t e_ = (call);                                                                       \
    if (e_ != cudaSuccess) { st = e_ == cudaErrorMemoryAllocation ? SNMF_ERR_OOM : SNMF_ERR_CUDA; cleanup(); return st; } \
  } while (0)
  plan();
  cudaError_t got = workspace_alloc((void**)&ws, bytes, s);
  while (got == cudaErrorMemoryAllocation && (w.tc_parts || w.parts > 1)) {
    // without the filter's 1 KB of candidates and its copy of each point, then without partial lists: k_knn
    // gives the same lists alone
    cudaGetLastError();
    if (w.tc_parts) w.tc_parts = 0;
    else w.parts = 1;
    plan();
    got = workspace_alloc((void**)&ws, bytes, s);
  }
  KCK(got);
  auto i32 = [&](size_t o) { return reinterpret_cast<int32_t*>(ws + o); };
  auto f32 = [&](size_t o) { return reinterpret_cast<float*>(ws + o); };
  int32_t *nbr = i32(o_nbr), *cnt = i32(o_cnt), *off = i32(o_off), *fill = i32(o_fill), *erow = i32(o_erow), *ecol = i32(o_ecol),
          *cntu = i32(o_cntu);
  float *nd2 = f32(o_nd2), *sval = f32(o_sval), *eval = f32(o_eval);
  float* sv = s_values ? s_values : f32(o_sv);
  float* dg = degree ? degree : f32(o_dg);
  uint8_t* erep = ws + o_erep;
  int* bad = i32(o_bad);  // non-finite distances, the filter given up, a bounded wait ran out
  w.pi = i32(o_pi); w.pd = f32(o_pd); w.Y = f32(o_y); w.nrm = f32(o_nrm); w.nrm0 = f32(o_nrm0); w.kth = f32(o_kth); w.ctr = f32(o_ctr);
  w.lists = f32(o_lists); w.cand = i32(o_cand); w.ncand = i32(o_ncand);
  w.bad = bad; w.dense = bad + 1; w.err = bad + 2;
  KCK(cudaMemsetAsync(bad, 0, 3 * sizeof(int), s));
  KCK(cudaMemsetAsync(cnt, 0, n * sizeof(int32_t), s));
  KCK(cudaMemsetAsync(cntu, 0, n * sizeof(int32_t), s));
  KCK(cudaMemsetAsync(fill, 0, n * sizeof(int32_t), s));
  KCK(launch_knn(X, n, d, k, w, nbr, nd2, s));
  const int g = (int)std::min<int64_t>((nk + 255) / 256, 152 * 16);
  k_knn_sim<<<g, 256, 0, s>>>(nbr, nd2, n, k, sigma_rank, sval, cnt, bad);
  k_scan<<<1, 1024, 0, s>>>(cnt, n, k, off);  // row slots: k own + in-degree
  k_knn_fill<<<g, 256, 0, s>>>(nbr, sval, n, k, off, fill, erow, ecol, eval);
  const int rb = (int)((n + 7) / 8);
  const int eb = (int)((2 * nk + 255) / 256);
  k_knn_dedupe<<<eb, 256, 0, s>>>(off, erow, ecol, eval, 2 * nk, 0, erep, cntu, nullptr, nullptr, nullptr);
  k_scan<<<1, 1024, 0, s>>>(cntu, n, 0, rowptr);
  int32_t total = 0;
  int hbad[3] = {0, 0, 0};
  KCK(cudaMemcpyAsync(&total, rowptr + n, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  KCK(cudaMemcpyAsync(hbad, bad, sizeof(hbad), cudaMemcpyDeviceToHost, s));
  KCK(cudaStreamSynchronize(s));
  *nnz = total;
  if (hbad[2]) { cleanup(); return SNMF_ERR_TIMEOUT; }
  if (hbad[0]) { cleanup(); return SNMF_ERR_NUMERIC; }
  if (total > capacity) { cleanup(); return SNMF_ERR_ARG; }
  k_knn_dedupe<<<eb, 256, 0, s>>>(off, erow, ecol, eval, 2 * nk, 1, erep, cntu, rowptr, colidx, sv);
  k_knn_degree<<<rb, 256, 0, s>>>(rowptr, sv, n, dg);
  k_knn_normalize<<<rb, 256, 0, s>>>(rowptr, colidx, sv, dg, n, a_hat);
  KCK(cudaGetLastError());
  KCK(cudaStreamSynchronize(s));
#undef KCK
  cleanup();
  return SNMF_OK;
}

extern "C" snmf_status snmf_cluster_scores(const int32_t* truth, const int32_t* pred, int64_t n, int k_true,
                                           int k_pred, int64_t* table, double* ari, double* accuracy, void* stream) {
  if (!truth || !pred || n < 2 || k_true < 1 || k_pred < 1 || k_true > 512 || k_pred > 512 ||
      (int64_t)k_true * k_pred > 4096)
    return SNMF_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  unsigned long long* dt = nullptr;
  int* bad = nullptr;
  const size_t tb = (size_t)k_true * k_pred * sizeof(unsigned long long);
  if (cudaMalloc(&dt, tb) != cudaSuccess) return SNMF_ERR_OOM;
  if (cudaMalloc(&bad, sizeof(int)) != cudaSuccess) { cudaFree(dt); return SNMF_ERR_OOM; }
  std::vector<unsigned long long> ht((size_t)k_true * k_pred);
  int hbad = 0;
  cudaError_t e = cudaMemsetAsync(dt, 0, tb, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(bad, 0, sizeof(int), s);
  if (e == cudaSuccess) {
    const int blocks = (int)std::min<int64_t>((n + 255) / 256, 152 * 4);
    k_contingency<<<blocks, 256, (size_t)k_true * k_pred * sizeof(unsigned), s>>>(truth, pred, n, k_true, k_pred, dt, bad);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(ht.data(), dt, tb, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFree(dt);
  cudaFree(bad);
  if (e != cudaSuccess) return SNMF_ERR_CUDA;
  if (hbad) return SNMF_ERR_ARG;
  std::vector<long long> T(ht.begin(), ht.end());
  if (table) for (size_t x = 0; x < T.size(); ++x) table[x] = T[x];
  // adjusted Rand index (Hubert and Arabie) in FP64 from the table
  auto comb = [](double x) { return x * (x - 1.0) / 2.0; };
  double idx = 0.0, sa = 0.0, sb = 0.0, tot = 0.0;
  std::vector<double> rs(k_true, 0.0), cs(k_pred, 0.0);
  for (int a = 0; a < k_true; ++a)
    for (int b = 0; b < k_pred; ++b) {
      const double v = (double)T[(size_t)a * k_pred + b];
      idx += comb(v);
      rs[a] += v;
      cs[b] += v;
      tot += v;
    }
  for (double v : rs) sa += comb(v);
  for (double v : cs) sb += comb(v);
  const double expv = sa * sb / comb(tot), mx = 0.5 * (sa + sb);
  if (ari) *ari = (mx != expv) ? (idx - expv) / (mx - expv) : 1.0;
  if (accuracy) *accuracy = (double)max_matching(T, k_true, k_pred) / tot;
  return SNMF_OK;
}

// exported for capi.cu (the handle's factor buffers live there)
namespace snmf {
void launch_assign(int tdtype, const void* F, int64_t n, int64_t ld, int64_t col0, int r, int32_t* lab, cudaStream_t s) {
  const int blocks = (int)std::min<int64_t>((n + 255) / 256, 152 * 8);
  if (tdtype == 0) k_assign<double><<<blocks, 256, 0, s>>>((const double*)F, n, ld, col0, r, lab);
  else k_assign<float><<<blocks, 256, 0, s>>>((const float*)F, n, ld, col0, r, lab);
}
}  // namespace snmf
