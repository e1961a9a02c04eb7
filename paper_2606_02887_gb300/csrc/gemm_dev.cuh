// CUDA-core product tile Y = A X for one CTA: FP64 and FP32 A as they are, BF16 A (full or its upper
// 128 x 128 tiles) and E4M3 A widened to FP32 while they are staged.  Used by the dense products
// (ax.cu, fp8.cu) and by the uneven batch (batch.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include "common.cuh"
#include "gram_dev.cuh"

namespace snmf {

namespace {

// How A is held: the factor type itself (row-major), BF16 (row-major), BF16 upper tiles
// (sym_tile), E4M3 codes with a power-of-two scale per 128 x 128 tile.
enum GemmA { GA_SAME = 0, GA_BF16, GA_BF16_SYM, GA_FP8 };

// The CTA tile is BM x BN with a TM x TN micro tile per thread; BK columns of A per stage.  Thread
// (tx, ty) owns rows ty + TY i and the columns of `col`.  A is staged as it lies, [row][k] with a
// row stride of BK + 16 bytes: a thread reads 16 bytes along k of each of its rows, lanes of
// different ty fall into different banks, and no transposition is needed on the way in.
template <typename T_, int KIND_, int BM_, int BN_, int TM_, int TN_, int BK_>
struct GemmCfg {
  using T = T_;
  static constexpr int KIND = KIND_, BM = BM_, BN = BN_, TM = TM_, TN = TN_, BK = BK_;
  static constexpr int TX = BN / TN, TY = BM / TM, NT = TX * TY;
  static constexpr int KV = 16 / (int)sizeof(T);             // values of 16 bytes
  static constexpr int AS = BK + KV;                         // row stride of the A stage
  static constexpr int A_ELEMS = BM * AS > BK * (BM + 4) ? BM * AS : BK * (BM + 4);
  static constexpr int STAGE = A_ELEMS + BK * BN;
  // asynchronous copies run two stages ahead; widened A goes through registers, one stage ahead
  static constexpr int STAGES = KIND == GA_SAME ? 3 : 2;
  static constexpr size_t SMEM = (size_t)STAGE * STAGES * sizeof(T);
  static constexpr int VW = TN % KV == 0 ? KV : 1;           // columns in a row of a thread
  __device__ static int col(int tx, int j) { return j / VW * (TX * VW) + tx * VW + j % VW; }
};

struct GemmA8 {
  const float* scales;
  int nt;
};

__device__ __forceinline__ float e4m3_value(uint32_t q) {
  const __half_raw h = __nv_cvt_fp8_to_halfraw((__nv_fp8_storage_t)q, __NV_E4M3);
  return __half2float(__half(h));
}

// acc[i][j] += a[i][u] x[j].  FP32: two columns per instruction (the same roundings), which leaves
// issue slots to the shared loads and the address arithmetic.
template <typename C>
__device__ __forceinline__ void fma_row(const typename C::T (&a)[C::TM][C::KV], int u, const typename C::T (&x)[C::TN],
                                        typename C::T (&acc)[C::TM][C::TN]) {
#pragma unroll
  for (int i = 0; i < C::TM; ++i) {
    if constexpr (sizeof(typename C::T) == 4 && C::TN % 2 == 0) {
      const float2 aa = make_float2(a[i][u], a[i][u]);
#pragma unroll
      for (int j = 0; j < C::TN; j += 2) {
        const float2 r = __ffma2_rn(aa, make_float2(x[j], x[j + 1]), make_float2(acc[i][j], acc[i][j + 1]));
        acc[i][j] = r.x;
        acc[i][j + 1] = r.y;
      }
    } else {
#pragma unroll
      for (int j = 0; j < C::TN; ++j) acc[i][j] = fma(a[i][u], x[j], acc[i][j]);
    }
  }
}

// acc = rows [row0, row0 + BM) x columns [col0, col0 + BN) of A X over k in [k0, k1).  A, lda: see
// GemmA (GA_BF16_SYM: lda = tiles a side; GA_FP8: a8 has the scales); na rows and columns of A
// exist.  avec / xvec: 16-byte copies of A / X are aligned and end with the row's values (k0, k1, cols
// and the pitch multiples of 16 bytes).  The widened kinds need k0 a multiple
// of BK (and, of 128 x 128 tiles, BM = 128).  Bound by the FMA pipes: 8192 x 8192 x 64 in FP32 took
// 377 us with 4 x 4 micro tiles read as scalars from a transposed stage, see ax.cu.
template <typename C, typename TA>
__device__ __forceinline__ void gemm_tile(const TA* __restrict__ A, int64_t lda, const typename C::T* __restrict__ X,
                                          int64_t ldx, int64_t na, int cols, int64_t row0, int col0, int64_t k0,
                                          int64_t k1, bool avec, bool xvec, GemmA8 a8, typename C::T* sm,
                                          typename C::T (&acc)[C::TM][C::TN]) {
  using T = typename C::T;
  constexpr int KV = C::KV, BK = C::BK, BM = C::BM, BN = C::BN, NT = C::NT, AS = C::AS;
  const int t = threadIdx.x, tx = t % C::TX, ty = t / C::TX;
#pragma unroll
  for (int i = 0; i < C::TM; ++i)
#pragma unroll
    for (int j = 0; j < C::TN; ++j) acc[i][j] = T(0);
  const int rounds = k1 > k0 ? (int)((k1 - k0 + BK - 1) / BK) : 0;
  auto copy_x = [&](int64_t k, T* xs) {
    if (xvec) {
      constexpr int NX = BK * BN / KV;
#pragma unroll
      for (int u = 0; u < (NX + NT - 1) / NT; ++u) {
        const int e = t + NT * u;
        if (NX % NT && e >= NX) break;
        const int kk = e / (BN / KV), c = e % (BN / KV) * KV;
        const bool v = k + kk < k1 && col0 + c < cols;
        cp_async<16>(xs + kk * BN + c, v ? X + (k + kk) * ldx + col0 + c : X, v);
      }
    } else if constexpr (NT % BN == 0) {  // one column of X per thread: no index arithmetic per value
      const int c = t % BN, left = (int)min((int64_t)BK, k1 - k) - t / BN;
      const bool on = col0 + c < cols;
      const T* p = X + (k + t / BN) * ldx + col0 + c;
#pragma unroll
      for (int u = 0; u < BK * BN / NT; ++u) {
        const bool v = on && u * (NT / BN) < left;
        cp_async<(int)sizeof(T)>(xs + t + NT * u, v ? p : X, v);
        p += NT / BN * ldx;
      }
    } else {
      for (int e = t; e < BK * BN; e += NT) {
        const int kk = e / BN, c = e % BN;
        const bool v = k + kk < k1 && col0 + c < cols;
        cp_async<(int)sizeof(T)>(xs + e, v ? X + (k + kk) * ldx + col0 + c : X, v);
      }
    }
  };
  auto fma_stage = [&](const T* as, const T* xs, bool tr) {
#pragma unroll
    for (int kk = 0; kk < BK; kk += KV) {
      T a[C::TM][KV];
      if (C::KIND == GA_BF16_SYM && tr) {  // the mirror tile's rows: [k][row]
#pragma unroll
        for (int i = 0; i < C::TM; ++i)
#pragma unroll
          for (int u = 0; u < KV; ++u) a[i][u] = as[(kk + u) * (BM + 4) + ty + C::TY * i];
      } else {
#pragma unroll
        for (int i = 0; i < C::TM; ++i) {
          if constexpr (sizeof(T) == 4) {
            const float4 v = *reinterpret_cast<const float4*>(as + (ty + C::TY * i) * AS + kk);
            a[i][0] = v.x; a[i][1] = v.y; a[i][2] = v.z; a[i][3] = v.w;
          } else {
            const double2 v = *reinterpret_cast<const double2*>(as + (ty + C::TY * i) * AS + kk);
            a[i][0] = v.x; a[i][1] = v.y;
          }
        }
      }
#pragma unroll
      for (int u = 0; u < KV; ++u) {
        T x[C::TN];
#pragma unroll
        for (int j = 0; j < C::TN; j += C::VW) {
          const T* p = xs + (kk + u) * BN + C::col(tx, j);
          if constexpr (C::VW == 4) {
            const float4 v = *reinterpret_cast<const float4*>(p);
            x[j] = v.x; x[j + 1] = v.y; x[j + 2] = v.z; x[j + 3] = v.w;
          } else if constexpr (C::VW == 2) {
            const double2 v = *reinterpret_cast<const double2*>(p);
            x[j] = v.x; x[j + 1] = v.y;
          } else {
            x[j] = *p;
          }
        }
        fma_row<C>(a, u, x, acc);
      }
    }
  };
  if constexpr (C::KIND == GA_SAME) {
    auto fetch = [&](int s) {
      const int64_t k = k0 + (int64_t)s * BK;
      T* as = sm + (s % C::STAGES) * C::STAGE;
      if (avec) {
        constexpr int NA = BM * BK / KV;
#pragma unroll
        for (int u = 0; u < (NA + NT - 1) / NT; ++u) {
          const int e = t + NT * u;
          if (NA % NT && e >= NA) break;
          const int m = e / (BK / KV), kk = e % (BK / KV) * KV;
          const bool v = row0 + m < na && k + kk < k1;
          cp_async<16>(as + m * AS + kk, v ? A + (row0 + m) * lda + k + kk : A, v);
        }
      } else {  // one column of the stage per thread
        static_assert(NT % BK == 0 && BM * BK % NT == 0, "whole rows of the stage");
        const int kk = t % BK, m0 = t / BK, rows = (int)min((int64_t)BM, na - row0);
        const bool on = k + kk < k1;
        const T* p = A + (row0 + m0) * lda + k + kk;
#pragma unroll
        for (int u = 0; u < BM * BK / NT; ++u) {
          const int m = m0 + u * (NT / BK);
          const bool v = on && m < rows;
          cp_async<(int)sizeof(T)>(as + m * AS + kk, v ? p : A, v);
          p += NT / BK * lda;
        }
      }
      copy_x(k, as + C::A_ELEMS);
    };
#pragma unroll
    for (int s = 0; s < C::STAGES - 1; ++s) {
      if (s < rounds) fetch(s);
      cp_async_commit();
    }
    for (int s = 0; s < rounds; ++s) {
      cp_async_wait<C::STAGES - 2>();
      __syncthreads();  // stage s is in; every thread is done with the one refilled below
      if (s + C::STAGES - 1 < rounds) fetch(s + C::STAGES - 1);
      cp_async_commit();
      const T* as = sm + (s % C::STAGES) * C::STAGE;
      fma_stage(as, as + C::A_ELEMS, false);
    }
    cp_async_wait<0>();
  } else {
    // 16 bytes of A at a time through registers: 8 BF16 values or 16 codes, widened to FP32
    constexpr int VA = C::KIND == GA_FP8 ? 16 : 8;
    constexpr int NA = BM * BK / VA, LA = (NA + NT - 1) / NT;
    uint4 ra[LA];
    bool tr = false, tr_next = false;
    float sc = 1.f, sc_next = 1.f;
    auto load = [&](int s) {
      const int64_t k = k0 + (int64_t)s * BK;
      if constexpr (C::KIND == GA_BF16_SYM) tr_next = k / 128 < row0 / 128;
      if constexpr (C::KIND == GA_FP8) sc_next = __ldg(a8.scales + row0 / 128 * a8.nt + k / 128);
#pragma unroll
      for (int u = 0; u < LA; ++u) {
        const int e = t + NT * u;
        ra[u] = make_uint4(0u, 0u, 0u, 0u);
        if (NA % NT && e >= NA) continue;
        if constexpr (C::KIND == GA_BF16_SYM) {
          const int64_t ta = row0 / 128, tb = k / 128;
          if (tr_next) {  // rows k .. of the stored mirror tile, BM values each
            const int kk = e / (BM / VA), m = e % (BM / VA) * VA;
            ra[u] = *reinterpret_cast<const uint4*>(A + (sym_tile(tb, ta, lda) << 14) + (k % 128 + kk) * 128 + m);
          } else {
            const int m = e / (BK / VA), kk = e % (BK / VA) * VA;
            ra[u] = *reinterpret_cast<const uint4*>(A + (sym_tile(ta, tb, lda) << 14) + m * 128 + k % 128 + kk);
          }
        } else {  // the pitch is padded to 16 bytes, with zeros
          const int m = e / (BK / VA), kk = e % (BK / VA) * VA;
          if (row0 + m < na && k + kk < lda) ra[u] = *reinterpret_cast<const uint4*>(A + (row0 + m) * lda + k + kk);
        }
      }
    };
    auto put = [&](T* as) {
      tr = tr_next;
      sc = sc_next;
#pragma unroll
      for (int u = 0; u < LA; ++u) {
        const int e = t + NT * u;
        if (NA % NT && e >= NA) continue;
        const uint32_t w[4] = {ra[u].x, ra[u].y, ra[u].z, ra[u].w};
        float f[VA];
        if constexpr (C::KIND == GA_FP8) {
#pragma unroll
          for (int i = 0; i < VA; ++i) f[i] = e4m3_value((w[i / 4] >> (8 * (i % 4))) & 0xFFu) * sc;
        } else {
#pragma unroll
          for (int i = 0; i < VA; ++i) f[i] = __uint_as_float(i % 2 ? w[i / 2] & 0xFFFF0000u : w[i / 2] << 16);
        }
        T* dst;
        if (C::KIND == GA_BF16_SYM && tr) dst = as + e / (BM / VA) * (BM + 4) + e % (BM / VA) * VA;
        else dst = as + e / (BK / VA) * AS + e % (BK / VA) * VA;
#pragma unroll
        for (int i = 0; i < VA; i += 4) *reinterpret_cast<float4*>(dst + i) = make_float4(f[i], f[i + 1], f[i + 2], f[i + 3]);
      }
    };
    if (rounds > 0) {
      load(0);
      put(sm);
      copy_x(k0, sm + C::A_ELEMS);
    }
    cp_async_commit();
    for (int s = 0; s < rounds; ++s) {
      T* as = sm + (s & 1) * C::STAGE;
      T* an = sm + ((s + 1) & 1) * C::STAGE;
      cp_async_wait<0>();
      __syncthreads();  // stage s is in, the other one free
      const bool tr_now = tr;
      if (s + 1 < rounds) {
        load(s + 1);
        copy_x(k0 + (int64_t)(s + 1) * BK, an + C::A_ELEMS);
      }
      cp_async_commit();
      fma_stage(as, as + C::A_ELEMS, tr_now);
      if (s + 1 < rounds) put(an);
    }
    cp_async_wait<0>();
  }
}

}  // namespace

}  // namespace snmf
