// Nearest neighbours with the tensor cores as a filter: TF32 inner products of the centred points
// (tcgen05, kind::tf32) bound every squared distance from both sides, and only the pairs that can be
// among a query's k nearest are computed in FP32, with the sums of k_knn.  The lists are those of
// k_knn, bit for bit.
//
// The bounds.  y = fl(x - c) for any centre c, rounded to TF32 (relative error 2^-11), n = |x - c|^2:
//   | |x_q - x_j|^2 - (n_q + n_j - 2 <y_q, y_j>) | <= e (n_q + n_j) + a,
// where e covers 2 (2^-11 + 2^-11) |y_q| |y_j| <= 2^-10 (n_q + n_j) of the operands' rounding, 16 steps
// of truncating accumulation, the rounding of the centring, of the norms and of the comparison, and
// that of the FP32 sum which is bounded (1.13e-3 together for d <= 128; e = 1.25e-3).  a covers what
// underflows: a coordinate or a product below 2^-126 may count as zero, and a square rounds to a multiple of
// 2^-149.  Lost products and squares are at most 4 d 2^-126 = 6e-36 together, and lost coordinates at most
// 2 d 2^-126 |y|, which is below the 1.2e-4 n left in e for |y| > 3e-32 and below 1e-67 otherwise; a = 1e-34.
//
//   pass 0  the k smallest upper bounds of every query over every second point, values only, kept sorted
//           in registers (a lane per query and half a tile); k_knn_bound takes the k-th of all lists
//           of a query, T_q (with 2 a: a neighbour's lower bound is at most its distance plus a, and that at
//           most the k-th upper bound plus a)
//   pass 1  over all points the pairs whose lower bound is not above T_q, appended to the query's
//           candidates (about four times k of them for clustered data)
//   k_knn_exact  their distances and the k nearest, a warp per query
//
// CTA of a pass: 128 queries (their TF32 rows stay in shared memory) against tiles of 64 candidates:
// one warp feeds a ring by TMA, one issues the MMAs into two TMEM accumulators, and eight warps read
// and compare them.  What bounds a pass is that reading and comparing; the passes repeat the products
// because lists of distances kept during one pass cost more: 130 distances per query, by scattered
// loads, and their insertion.  n = 20000, d = 64, k = 10: pass 0 325 us, pass 1 217, the exact distances
// 42 (870 us in one pass; k_knn 2940).
//
// Where a query has more than KT_CAP candidates (clusters much tighter than their distance from the
// centre, many copies of a point), or a norm is too large for the bounds, *dense is set and k_knn
// computes all lists.
#pragma once

#include "ax_tc.cuh"
#include "tc_dev.cuh"

namespace snmf {

namespace {

constexpr int KT_Q = 128, KT_C = 64;   // queries and candidates of a tile
constexpr int KT_STAGES = 3;
constexpr int KT_THREADS = 320;        // 8 epilogue warps, TMA, MMA
constexpr int KT_MAXD = 128;
constexpr int KT_PARTS = 8;            // at most, of the candidates (two lists each)
constexpr int KT_CAP = 256;            // candidates of a query
constexpr float KT_E = 1.25e-3f;
constexpr float KT_UP = 2.f * KT_E / (1.f - KT_E);
constexpr float KT_ABS = 2e-34f;       // 2 a
constexpr float KT_MAXNORM = 1e36f;    // n below it: no distance or product overflows
constexpr long long KT_BUDGET = 2000000000LL;

struct KnnTcSmem {
  uint64_t full[KT_STAGES], empty[KT_STAGES], afull[2], aempty[2], abar;
  uint32_t tmem;
  int abort, skip;
};

inline size_t knn_tc_smem(int d) { return (size_t)((d + 31) / 32) * (KT_Q + KT_STAGES * KT_C) * 128 + 1024; }

// The mean of up to 64 points (any centre is valid: a good one keeps the norms small).
__global__ void __launch_bounds__(1024) k_knn_center(const float* __restrict__ X, int64_t n, int d, float* __restrict__ ctr) {
  __shared__ float part[8][KT_MAXD];
  const int c = threadIdx.x & (KT_MAXD - 1), g = threadIdx.x / KT_MAXD;
  const int m = (int)min(n, (int64_t)64);
  float s = 0.f;
  if (c < d)
#pragma unroll 8
    for (int u = g; u < m; u += 8) s += X[(int64_t)u * n / m * d + c];
  part[g][c] = s;
  __syncthreads();
  if (g == 0 && c < d) {
    for (int u = 1; u < 8; ++u) s += part[u][c];
    ctr[c] = s / (float)m;
  }
}

// TF32 rows of the centred points (pitch dp, zero-padded) and (1 - e) n of each; *dense where a norm is
// too large or not finite.  One warp per point.
__global__ void __launch_bounds__(256) k_knn_prep(const float* __restrict__ X, int64_t n, int d, int dp,
                                                  const float* __restrict__ ctr, float* __restrict__ Y,
                                                  float* __restrict__ nrm, float* __restrict__ kth, int* __restrict__ ncand, int stride,
                                                  float* __restrict__ nrm0, int* __restrict__ dense) {
  const int lane = threadIdx.x & 31;
  const int64_t i = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= n) return;
  float s = 0.f;
  for (int t = lane; t < dp; t += 32) {
    const float y = t < d ? X[i * d + t] - ctr[t] : 0.f;
    s = fmaf(y, y, s);
    Y[i * dp + t] = __uint_as_float(tc::to_tf32(y));
  }
  s = warp_sum(s);
  if (lane == 0) {
    nrm[i] = (1.f - KT_E) * s;
    if (i % stride == 0) nrm0[i / stride] = (1.f - KT_E) * s;
    kth[i] = INFINITY;
    ncand[i] = 0;
    if (!(s < KT_MAXNORM)) atomicOr(dense, 1);
  }
}

struct Float8 {
  float v[8];
};
__device__ __forceinline__ Float8 ldg8(const float* p) {
  Float8 r;
  asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=f"(r.v[0]), "=f"(r.v[1]), "=f"(r.v[2]), "=f"(r.v[3]), "=f"(r.v[4]), "=f"(r.v[5]), "=f"(r.v[6]), "=f"(r.v[7])
      : "l"(p));
  return r;
}

// sum over t ascending of (q_t - c_t)^2, one FMA each: k_knn's distance.  VEC: floats of one load (the
// lanes' rows are scattered, so a load costs its 32 lines whatever its width).
template <int VEC>
__device__ __forceinline__ float knn_dist(const float* __restrict__ q, const float* __restrict__ c, int d) {
  float s = 0.f;
  if (VEC == 8) {
#pragma unroll 2
    for (int t = 0; t < d; t += 8) {
      const Float8 a = ldg8(q + t), b = ldg8(c + t);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const float df = a.v[u] - b.v[u];
        s = __fmaf_rn(df, df, s);
      }
    }
  } else if (VEC == 4) {
#pragma unroll 4
    for (int t = 0; t < d; t += 4) {
      const float4 a = __ldg(reinterpret_cast<const float4*>(q + t)), b = __ldg(reinterpret_cast<const float4*>(c + t));
      const float d0 = a.x - b.x, d1 = a.y - b.y, d2 = a.z - b.z, d3 = a.w - b.w;
      s = __fmaf_rn(d0, d0, s);
      s = __fmaf_rn(d1, d1, s);
      s = __fmaf_rn(d2, d2, s);
      s = __fmaf_rn(d3, d3, s);
    }
  } else {
#pragma unroll 4
    for (int t = 0; t < d; ++t) {
      const float df = __ldg(q + t) - __ldg(c + t);
      s = __fmaf_rn(df, df, s);
    }
  }
  return s;
}

// The candidates are nc points, every stride-th one.  PASS 0: KR >= k registers for the list; lists[(part
// 2 + half) k + slot][n], kth[q] the smallest bound that a list has given so far.  PASS 1: cand[q][KT_CAP], ncand[q].
template <int PASS, int KR>
__global__ void __launch_bounds__(KT_THREADS, 2)
k_knn_tc(const __grid_constant__ CUtensorMap map, const __grid_constant__ CUtensorMap cmap, const float* __restrict__ nrm,
         const float* __restrict__ cnrm, int64_t nc, int stride, float* kth, int64_t n, int d, int k, int64_t per,
          float* __restrict__ lists, int32_t* __restrict__ cand, int* __restrict__ ncand, int* __restrict__ dense,
         int* __restrict__ err) {
  using namespace tc;
  extern __shared__ unsigned char kt_raw[];
  __shared__ KnnTcSmem S;
  unsigned char* base =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(kt_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t q0 = (int64_t)blockIdx.x * KT_Q, cb = (int64_t)blockIdx.y * per, ce = min(nc, cb + per);
  const int tiles = ce > cb ? (int)((ce - cb + KT_C - 1) / KT_C) : 0;
  const int dch = (d + 31) / 32;
  unsigned char* sA = base;
  unsigned char* sB = sA + (size_t)dch * KT_Q * 128;
  if (threadIdx.x == 0) {
    for (int s = 0; s < KT_STAGES; ++s) {
      mbar_init(&S.full[s], 1);
      mbar_init(&S.empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&S.afull[b], 1);
      mbar_init(&S.aempty[b], 8);
    }
    mbar_init(&S.abar, 1);
    S.abort = 0;
    S.skip = *(volatile int*)dense;
    mbar_init_fence();
  }
  if (warp == 9) tmem_alloc(&S.tmem, 2 * KT_C);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const bool go = tiles > 0 && !S.skip;
  auto gone = [&] { return *(volatile int*)&S.abort != 0; };
  auto wait = [&](uint64_t* bar, int phase, int code) {
    const bool ok = mbar_wait(bar, (uint32_t)(phase & 1), KT_BUDGET, &S.abort);
    if (!ok && !gone()) {
      atomicCAS(err, 0, code);
      atomicOr(dense, 1);  // incomplete lists are computed again
      *(volatile int*)&S.abort = 1;
    }
    return ok;
  };
  if (go && warp == 8) {
    if (lane == 0) {
      mbar_arrive_expect_tx(&S.abar, (uint32_t)dch * KT_Q * 128);
      for (int c = 0; c < dch; ++c)
        for (int u = 0; u < KT_Q; u += KT_C)
          tma_load_2d(sA + ((size_t)c * KT_Q + u) * 128, &map, &S.abar, 32 * c, (int)q0 + u);
      int i = 0;
      for (; i < tiles; ++i) {
        const int s = i % KT_STAGES;
        if (i >= KT_STAGES && !wait(&S.empty[s], i / KT_STAGES - 1, 41)) break;
        mbar_arrive_expect_tx(&S.full[s], (uint32_t)dch * KT_C * 128);
        for (int c = 0; c < dch; ++c)
          tma_load_2d(sB + ((size_t)s * dch + c) * KT_C * 128, &cmap, &S.full[s], 32 * c, (int)cb + i * KT_C);
      }
      // after an abort the copies in flight are waited for
      if (gone()) {
        mbar_wait(&S.abar, 0u, KT_BUDGET);
        for (int u = max(0, i - KT_STAGES); u < i; ++u)
          mbar_wait(&S.full[u % KT_STAGES], (uint32_t)((u / KT_STAGES) & 1), KT_BUDGET);
      }
    }
    __syncwarp();
  } else if (go && warp == 9) {
    if (lane == 0 && wait(&S.abar, 0, 42)) {
      constexpr uint32_t idesc = idesc_tf32(KT_Q, KT_C);
      const uint32_t a0 = smem_u32(sA), b0 = smem_u32(sB);
      const int steps = (d + 7) / 8;
      int i = 0;
      for (; i < tiles; ++i) {
        const int s = i % KT_STAGES, b = i & 1;
        if (i >= 2 && !wait(&S.aempty[b], (i >> 1) - 1, 43)) break;
        if (!wait(&S.full[s], i / KT_STAGES, 44)) break;
        tc_fence_after();
        for (int t = 0; t < steps; ++t) {
          const int c = t >> 2;
          mma_tf32(S.tmem + (uint32_t)(b * KT_C), sdesc_sw128(a0 + c * KT_Q * 128 + (t & 3) * 32),
                   sdesc_sw128(b0 + (s * dch + c) * KT_C * 128 + (t & 3) * 32), idesc, t > 0 ? 1u : 0u);
        }
        mma_commit(&S.empty[s]);
        mma_commit(&S.afull[b]);
      }
      if (gone() && i > 0) mbar_wait(&S.afull[(i - 1) & 1], (uint32_t)(((i - 1) >> 1) & 1), KT_BUDGET);
    }
    __syncwarp();
  } else if (warp < 8) {
    const int h = warp >> 2, qw = 32 * (warp & 3), ql = qw + lane;
    const int64_t q = q0 + ql;
    const bool qv = q < n;
    const float nq = qv ? nrm[q] : 0.f;
    const uint32_t taddr = S.tmem + ((uint32_t)qw << 16) + 32 * h;
    float kd[PASS == 0 ? KR : 1];
    if (PASS == 0) {
#pragma unroll
      for (int u = 0; u < KR; ++u) kd[u] = u < KR - k ? -INFINITY : INFINITY;
    }
    float told = INFINITY;
    // a pair passes when f n_j - <y_q, y_j> is not above thr, in both passes
    const float f = PASS == 0 ? 0.5f + 0.5f * KT_UP : 0.5f;
    float thr = PASS == 0 ? INFINITY : 0.5f * ((qv ? kth[q] : 0.f) - nq);
    for (int i = 0; go && i < tiles; ++i) {
      const int64_t c0 = cb + (int64_t)i * KT_C + 32 * h;
      const int left = (int)min((int64_t)32, ce - c0);  // columns of this half that exist
      float4 nj[8];  // the same in every lane; past the last candidate anything (masked below)
#pragma unroll
      for (int u = 0; u < 8; ++u) nj[u] = *reinterpret_cast<const float4*>(cnrm + c0 + 4 * u);
      const bool ok = wait(&S.afull[i & 1], i >> 1, 45);
      if (!__all_sync(0xffffffffu, ok)) break;
      tc_fence_after();
      uint32_t mask = 0u;
      float v[32];
#pragma unroll
      for (int g = 0; g < 2; ++g) tmem_ld16(taddr + (uint32_t)((i & 1) * KT_C + 16 * g), v + 16 * g);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&S.aempty[i & 1]);
#pragma unroll
      for (int u = 0; u < 32; ++u) {
        v[u] = fmaf(f, (&nj[u / 4].x)[u & 3], -v[u]);
        if (v[u] <= thr) mask |= 1u << u;
      }
      if (left < 32) mask &= left > 0 ? (1u << left) - 1u : 0u;
      const int64_t self = q % stride ? -1 : q / stride - c0;
      if (self >= 0 && self < 32) mask &= ~(1u << self);
      if (!qv) mask = 0u;
      if (PASS == 0) {
        const unsigned any = __reduce_or_sync(0xffffffffu, mask);
        if (any) {
#pragma unroll
          for (int u = 0; u < 32; ++u) {
            if (any >> u & 1u) {
              const float x = mask >> u & 1u ? v[u] : INFINITY;
#pragma unroll
              for (int w = KR - 1; w > 0; --w) kd[w] = fminf(kd[w], fmaxf(kd[w - 1], x));
              kd[0] = fminf(kd[0], x);
            }
          }
          thr = fminf(thr, kd[KR - 1]);
        }
        if ((i & 7) == 7 && qv) {  // the bound of the query's other lists
          const float mine = fmaxf(0.f, 2.f * kd[KR - 1] + nq * (1.f + KT_UP));
          if (mine < told) {
            atomicMin(reinterpret_cast<int*>(kth) + q, __float_as_int(mine));
            told = mine;
          }
          thr = fminf(thr, 0.5f * (*(volatile float*)&kth[q] - nq * (1.f + KT_UP)));
        }
      } else {
        while (mask) {
          const int c = __ffs(mask) - 1;
          mask &= mask - 1u;
          const int at = atomicAdd(&ncand[q], 1);
          if (at < KT_CAP) {
            cand[q * KT_CAP + at] = (int32_t)(c0 + c);
          } else {
            atomicOr(dense, 1);
            mask = 0u;
            thr = -INFINITY;
          }
        }
      }
    }
    if (PASS == 0 && qv) {
#pragma unroll
      for (int u = 0; u < KR; ++u)
        if (u >= KR - k) lists[((int64_t)(blockIdx.y * 2 + h) * k + (u - (KR - k))) * n + q] = kd[u];
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 9) {
    tc_fence_after();
    tmem_dealloc(S.tmem, 2 * KT_C);
  }
}

// kth[q]: T_q, from the k-th smallest upper bound of the query's sorted lists (or what a list gave already,
// which pass 0 takes without the 2 a: its lists then miss none of the k smallest bounds).
__global__ void __launch_bounds__(128) k_knn_bound(const float* __restrict__ lists, const float* __restrict__ nrm, int64_t n,
                                                   int k, int count, float* __restrict__ kth) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n) return;
  float head[2 * KT_PARTS];
  int at[2 * KT_PARTS];
#pragma unroll
  for (int l = 0; l < 2 * KT_PARTS; ++l) {
    at[l] = 0;
    head[l] = l < count ? lists[(int64_t)l * k * n + q] : INFINITY;
  }
  float v = INFINITY;
  for (int u = 0; u < k; ++u) {
    v = INFINITY;
    int from = 0;
#pragma unroll
    for (int l = 0; l < 2 * KT_PARTS; ++l)
      if (head[l] < v) {
        v = head[l];
        from = l;
      }
#pragma unroll
    for (int l = 0; l < 2 * KT_PARTS; ++l)
      if (l == from && l < count) head[l] = ++at[l] < k ? lists[((int64_t)l * k + at[l]) * n + q] : INFINITY;
  }
  kth[q] = fminf(kth[q], 2.f * v + nrm[q] * (1.f + KT_UP)) + KT_ABS;
}

// One warp per query: the distances of its candidates and the k nearest.
template <int VEC>
__global__ void __launch_bounds__(256) k_knn_exact(const float* __restrict__ X, int64_t n, int d, int k,
                                                   const int32_t* __restrict__ cand, const int* __restrict__ ncand,
                                                   int32_t* __restrict__ nbr, float* __restrict__ nd2,
                                                   const int* __restrict__ dense) {
  if (*dense) return;
  const int lane = threadIdx.x & 31;
  const int64_t q = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (q >= n) return;
  const int m = min(ncand[q], KT_CAP);
  float kd = INFINITY;
  int32_t ki = INT_MAX;
  for (int b = 0; b < m; b += 32) {
    const bool on = b + lane < m;
    const int32_t j = on ? cand[q * KT_CAP + b + lane] : INT_MAX;
    const float v = on ? knn_dist<VEC>(X + q * d, X + (int64_t)j * d, d) : INFINITY;
    const int e = min(32, m - b);
    for (int u = 0; u < e; ++u) knn_insert(kd, ki, __shfl_sync(0xffffffffu, v, u), __shfl_sync(0xffffffffu, j, u));
  }
  if (lane < k) {
    nbr[q * k + lane] = ki;
    nd2[q * k + lane] = kd;
  }
}

}  // namespace

}  // namespace snmf
