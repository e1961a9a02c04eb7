// Row kernels of an Algorithm-1 step for any rank r <= 128, FP64 or FP32, as a CTA body: block-start
// gradient, D step and relaxed update, used per restart (rowstep.cu) and per problem of the uneven
// batch (batch.cu).
//
//   RS_GRAD  g = X G - B (+ gamma LX) written to gout (and X to Xout); with Xold / Zold the BB and
//            increment inner products of an update whose X' is given; with Znext the next step's
//            Z = Proj[X - g / rho]
//   RS_D     Z = Proj[X - g / rho], g(Z) = Z G - B, D = Proj[Z - alpha g(Z)] - Z (Alg. 1 lines 2-3);
//            writes g(Z) only; NC = 2: two directions (the learned step's fallback)
//   RS_DZ    the same with Z (as X) and gamma LZ given, D written: the graph-regularised block
//   RS_U     Z and D recomputed from X, g, g(Z) with the same FMAs, X' = Proj[Z + phi beta D],
//            g(X') (Alg. 1 line 4); in place over X and g
//
// Partial layout and control steps are those of the general row kernel (RowArgs).  A step moves
// 4 + 6 arrays of n x r instead of the 6 + 8 of stored Z and D.
//
// CTA: tiles of TY MR rows of one restart, all r columns; thread (tx, ty), tx < ceil(r / 4), owns
// columns 4 tx .. of rows ty + TY p, p < MR, in the loads, the row product and the epilogue alike, so
// inputs stay in registers from the one to the other and nothing is transposed: the operand tile
// goes to shared memory row-major (stride 4 more than the columns), a thread reads 16 bytes along k
// of its rows and 16 bytes of each row of G.  Ranks between the powers of two pay for their next
// multiple of 4 only.  A CTA walks several tiles: each thread copies its own inputs of the next tile
// to shared memory (asynchronously, no barrier) as soon as it has read the current one's there, the
// operand's inputs first, B and what else the epilogue reads after it; G is read once, and one
// record of partials, in FP64 over the tiles, leaves the CTA.  For long factors HBM, the shared
// loads and the instructions around the product are within a factor of two of one another (n = 2e6, r =
// 32: block-start gradient 209 us, D step 300, update 293; a CTA per tile, without copies ahead 407, 471,
// 501; with Z and X' recomputed after the product instead of read from the operand tile and every row and
// column tested 227, 320, 316); short ones are bound by launch latency.
#pragma once

#include "rowops_dev.cuh"

namespace snmf {

namespace {

enum { RS_GRAD = 0, RS_D, RS_DZ, RS_U };

__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }

// Comparisons with zero; FP64 by the bits, since an FP64 comparison takes the FP64 pipe for 64 cycles
// of a warp (NaN is neither positive nor negative).
__device__ __forceinline__ bool positive(float t) { return t > 0.f; }
__device__ __forceinline__ bool positive(double t) {
  return (unsigned long long)__double_as_longlong(t) - 1ull < 0x7ff0000000000000ull;
}
template <typename T>
__device__ __forceinline__ bool negative(T t) { return positive(-t); }
__device__ __forceinline__ bool is_zero(float t) { return t == 0.f; }
__device__ __forceinline__ bool is_zero(double t) { return __double_as_longlong(t) << 1 == 0; }

// W consecutive values of a row
template <typename T, int W>
struct alignas(W * sizeof(T) < 16 ? W * sizeof(T) : 16) Pack {
  T v[W];
};

// explicit FMAs: the D step and the update compute the same bits
__device__ __forceinline__ float proj0(float t) { return fmaxf(t, 0.f); }  // NaN: 0, in both
__device__ __forceinline__ double proj0(double t) { return positive(t) ? t : 0.0; }
template <typename T>
__device__ __forceinline__ T zstep(T x, T g, T inv_rho) { return proj0(fma_rn(-g, inv_rho, x)); }
template <typename T>
__device__ __forceinline__ T dir(T z, T gz, T alpha) { return proj0(fma_rn(-alpha, gz, z)) - z; }
template <typename T>
__device__ __forceinline__ T upd(T z, T d, T pb) { return proj0(fma_rn(pb, d, z)); }

// rows of a thread of a full CTA: as many as the registers hold
template <typename T>
__host__ __device__ constexpr int rowstep_mr() { return sizeof(T) == 4 ? 4 : 2; }

// rows of a tile, the input arrays of a step, and the dynamic shared memory of rank r with
// `threads` threads, mr rows each and `nin` inputs
__host__ __device__ inline int rowstep_rows(int r, int threads, int mr, int w = 4) { return threads / ((r + w - 1) / w) * mr; }
inline int rowstep_inputs(int step, const RowArgs& a) {
  if (step == RS_D) return 3;  // X, g, B
  if (step == RS_U) return 4;  // X, g, g(Z), B
  int k = 2 + (a.LX != nullptr);
  if (step == RS_DZ) return k + 2;
  return k + (a.Xold ? 2 : 0) + (a.Zold ? 2 : 0);
}
template <typename T>
__host__ __device__ inline size_t rowstep_smem(int r, int threads, int mr, int nin, int w = 4) {
  const int c = (r + 3) / 4 * 4;
  return ((size_t)rowstep_rows(r, threads, mr, w) * (c + 4) + (size_t)c * c + (size_t)nin * mr * threads * w) * sizeof(T);
}

// W columns of one row of a global array: 16-byte (or W values') accesses, or single values of the w
// that exist
template <typename T, int W>
__device__ __forceinline__ void copy_pack(Pack<T, W>* dst, const T* base, int64_t off, bool on, bool vec, int w) {
  constexpr int B = W * (int)sizeof(T) < 16 ? W * (int)sizeof(T) : 16;
  if (vec) {
    const char* p = reinterpret_cast<const char*>(on ? base + off : base);
#pragma unroll
    for (int q = 0; q < (int)sizeof(Pack<T, W>); q += B) cp_async<B>(reinterpret_cast<char*>(dst) + q, p + q, on);
  } else {
#pragma unroll
    for (int q = 0; q < W; ++q) cp_async<(int)sizeof(T)>(&dst->v[q], on && q < w ? base + off + q : base, on && q < w);
  }
}
template <typename T, int W>
__device__ __forceinline__ void store_pack(T* p, const Pack<T, W>& v, bool vec, int w) {
  if (vec) {
    *reinterpret_cast<Pack<T, W>*>(p) = v;
  } else {
#pragma unroll
    for (int q = 0; q < W; ++q)
      if (q < w) p[q] = v.v[q];
  }
}

// acc[p] = (row ty + TY p of As) G[:, W tx ..], k ascending in one chain per entry; zeros when not on
template <typename T, int W, int MR>
__device__ __forceinline__ void rowstep_product(const T* As, int ls, const T* Gs, int c4, int tx, int ty, int TY,
                                                Pack<T, W> (&acc)[MR], bool on) {
#pragma unroll
  for (int p = 0; p < MR; ++p)
#pragma unroll
    for (int q = 0; q < W; ++q) acc[p].v[q] = T(0);
  if (!on) return;
  const T* ar = As + ty * ls;
  const T* gr = Gs + W * tx;
#pragma unroll 2
  for (int k = 0; k < c4; k += 4) {
    Quad<T> a[MR];
#pragma unroll
    for (int p = 0; p < MR; ++p) a[p] = *reinterpret_cast<const Quad<T>*>(ar + p * TY * ls + k);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const Pack<T, W> g = *reinterpret_cast<const Pack<T, W>*>(gr + (k + u) * c4);
#pragma unroll
      for (int p = 0; p < MR; ++p) {
        if constexpr (sizeof(T) == 4 && W == 4) {
          const float2 aa = make_float2(a[p].v[u], a[p].v[u]);
          const float2 lo = __ffma2_rn(aa, make_float2(g.v[0], g.v[1]), make_float2(acc[p].v[0], acc[p].v[1]));
          const float2 hi = __ffma2_rn(aa, make_float2(g.v[2], g.v[3]), make_float2(acc[p].v[2], acc[p].v[3]));
          acc[p].v[0] = lo.x;
          acc[p].v[1] = lo.y;
          acc[p].v[2] = hi.x;
          acc[p].v[3] = hi.y;
        } else {
#pragma unroll
          for (int q = 0; q < W; ++q) acc[p].v[q] = fma(a[p].v[u], g.v[q], acc[p].v[q]);
        }
      }
    }
  }
}

// Sums of the eight partial values over a warp: value m ends up in lanes with lane & 7 == m
// (nine shuffles instead of forty).
template <typename T>
__device__ __forceinline__ T warp_sum8(const T (&v)[8]) {
  const int lane = threadIdx.x & 31;
  T a[4], b[2], c;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const T keep = lane & 4 ? v[4 + i] : v[i], give = lane & 4 ? v[i] : v[4 + i];
    a[i] = keep + __shfl_xor_sync(0xffffffffu, give, 4);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const T keep = lane & 2 ? a[2 + i] : a[i], give = lane & 2 ? a[i] : a[2 + i];
    b[i] = keep + __shfl_xor_sync(0xffffffffu, give, 2);
  }
  {
    const T keep = lane & 1 ? b[1] : b[0], give = lane & 1 ? b[0] : b[1];
    c = keep + __shfl_xor_sync(0xffffffffu, give, 1);
  }
  c += __shfl_xor_sync(0xffffffffu, c, 8);
  c += __shfl_xor_sync(0xffffffffu, c, 16);
  return c;
}

// CTA `cta` of `per` of restart j: its tiles cta, cta + per, ... of `tiles`.  vec: every row of the
// restart starts on 16 bytes in all arrays (r and the pitch multiples of 4).  sm: rowstep_smem bytes.
template <typename T, int STEP, int NC, int MR, int W = 4>
__device__ __forceinline__ void rowstep_body(const RowArgs& a, int j, int cta, int per, int tiles, bool vec, T* sm) {
  __shared__ double shq[8][8];
  __shared__ unsigned ticket;
  const Ctl& cj = a.ctl[j];
  const bool live = cj.active && !(a.run && *a.run == 0);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double total = 0.0;  // lane m < 8: the warp's sum of value m over the tiles
  if (live) {
    const int r = a.r, TX = (r + W - 1) / W, c4 = (r + 3) / 4 * 4, ls = c4 + 4, nt = blockDim.x, TY = nt / TX;
    const int t = threadIdx.x, ty = t / TX, tx = t - ty * TX;
    T* As = sm;
    T* Gs = sm + (size_t)TY * MR * ls;
    Pack<T, W>* in = reinterpret_cast<Pack<T, W>*>(Gs + c4 * c4) + t;  // input i of row k at in[(i MR + k) nt]
    const bool on = ty < TY;  // the block may hold a few threads more than TX TY
    const int w = r - W * tx;
    const int64_t colj = (int64_t)j * r + W * tx;
    // inputs in the order of their slots
    const bool lx = (STEP == RS_GRAD || STEP == RS_DZ) && a.LX, old = STEP == RS_GRAD && a.Xold,
               zold = STEP == RS_GRAD && a.Zold;
    const int iL = 2, iO = 2 + lx, iZ = iO + (old ? 2 : 0);
    auto copy = [&](int tile, int i, const void* p) {
      const int64_t row0 = (int64_t)tile * (TY * MR) + ty;
#pragma unroll
      for (int k = 0; k < MR; ++k) {
        const int64_t row = row0 + (int64_t)k * TY;
        copy_pack<T, W>(in + (i * MR + k) * nt, (const T*)p, row * a.ld + colj, on && row < a.n, vec, w);
      }
    };
    auto fetch_operand = [&](int tile) {  // one copy group each, empty past the last tile
      if (tile < tiles) {
        copy(tile, 0, STEP == RS_U ? a.Xout : a.X);
        if (STEP == RS_D) copy(tile, 2, a.g_in);
        if (STEP == RS_U) {
          copy(tile, 2, a.gout);
          copy(tile, 3, a.gZold);
        }
      }
      cp_async_commit();
    };
    auto fetch_rest = [&](int tile) {
      if (tile < tiles) {
        copy(tile, 1, a.B);
        if (lx) copy(tile, iL, a.LX);
        if (STEP == RS_DZ) {
          copy(tile, iO, a.Wcur);
          copy(tile, iO + 1, a.gWcur);
        }
        if (old) {
          copy(tile, iO, a.Xold);
          copy(tile, iO + 1, a.gold);
        }
        if (zold) {
          copy(tile, iZ, a.Zold);
          copy(tile, iZ + 1, a.gZold);
        }
      }
      cp_async_commit();
    };
    {
      // G joins the first copy group where its rows start on 16 bytes
      const T* G = (const T*)a.G + (int64_t)j * r * r;
      if (r == c4 && !((uintptr_t)G & 15)) {
        constexpr int KV = 16 / (int)sizeof(T);
        for (int e = t * KV; e < c4 * c4; e += nt * KV) cp_async<16>(Gs + e, G + e, true);
      } else {
        for (int e = t; e < c4 * c4; e += nt) {
          const int p = e / c4, q = e - p * c4;
          Gs[e] = p < r && q < r ? G[p * r + q] : T(0);
        }
      }
    }
    if (W < 4)  // the operand's columns past r, which no thread owns
      for (int e = t; e < TY * MR * (c4 - r); e += nt) As[e / (c4 - r) * ls + r + e % (c4 - r)] = T(0);
    fetch_operand(cta);
    fetch_rest(cta);
    // while the copies are on their way: the division is ten FP64 instructions
    const T inv_rho = (T)(1.0 / cj.rho);
    const T alpha0 = (T)(NC == 1 ? cj.alpha : cj.cand_alpha[STEP == RS_U ? (cj.dsel ? 1 : 0) : 0]);
    const T alpha1 = (T)(NC == 1 ? cj.alpha : cj.cand_alpha[1]);
    const T pb = (T)cj.phibeta;
    const T gam = (T)a.gamma;
    for (int tile = cta; tile < tiles; tile += per) {
      const int64_t row0 = (int64_t)tile * (TY * MR) + ty;
      const int64_t off0 = row0 * a.ld + colj, step = (int64_t)TY * a.ld;
      T dq[8];
#pragma unroll
      for (int m = 0; m < 8; ++m) dq[m] = T(0);
      int zeros = 0;
      bool rv[MR];
#pragma unroll
      for (int k = 0; k < MR; ++k) rv[k] = on && row0 + (int64_t)k * TY < a.n;
      auto get = [&](int i, int k) { return in[(i * MR + k) * nt]; };
      // this thread's values of the operand tile; rows, columns and threads beyond the tile hold zeros in
      // every array, which add nothing to the sums
      auto operand = [&](int k) {
        Pack<T, W> v;
#pragma unroll
        for (int q = 0; q < W; ++q) v.v[q] = T(0);
        if (on) v = *reinterpret_cast<const Pack<T, W>*>(As + (ty + k * TY) * ls + W * tx);
        return v;
      };
      auto put = [&](void* p, int k, const Pack<T, W>& v) {
        if (rv[k]) store_pack<T, W>((T*)p + off0 + k * step, v, vec, w);
      };
      cp_async_wait<1>();
      Pack<T, W> x[MR], g[MR], z[MR];
#pragma unroll
      for (int k = 0; k < MR; ++k) {
        x[k] = get(0, k);
        if (STEP == RS_D || STEP == RS_U) g[k] = get(2, k);
        if (STEP == RS_U) z[k] = get(3, k);
      }
      fetch_operand(tile + per);
      // the operand tile: X, Z or X'
#pragma unroll
      for (int k = 0; k < MR; ++k) {
        Pack<T, W> op = x[k];
#pragma unroll
        for (int q = 0; q < W; ++q) {
          if (STEP == RS_D) op.v[q] = zstep(x[k].v[q], g[k].v[q], inv_rho);
          if (STEP == RS_U) {
            const T zz = zstep(x[k].v[q], g[k].v[q], inv_rho);
            op.v[q] = upd(zz, dir(zz, z[k].v[q], alpha0), pb);
          }
        }
        if (on) *reinterpret_cast<Pack<T, W>*>(As + (ty + k * TY) * ls + W * tx) = op;
      }
      __syncthreads();
      Pack<T, W> acc[MR];
      rowstep_product<T, W, MR>(As, ls, Gs, c4, tx, ty, TY, acc, on);
      cp_async_wait<1>();
      if (STEP == RS_GRAD) {
#pragma unroll
        for (int k = 0; k < MR; ++k) {
          Pack<T, W> gn, l, zn;
          const Pack<T, W> b = get(1, k);
          if (lx) l = get(iL, k);
#pragma unroll
          for (int q = 0; q < W; ++q) {
            const T xv = x[k].v[q], bv = b.v[q];
            T gv = acc[k].v[q] - bv;
            if (lx) gv += gam * l.v[q];
            gn.v[q] = gv;
            zn.v[q] = zstep(xv, gv, inv_rho);
            const T pg = positive(xv) || negative(gv) ? gv : T(0);
            dq[0] = fma_rn(pg, pg, dq[0]);
            dq[1] = fma_rn(gv - bv, xv, dq[1]);
            zeros += is_zero(xv);
          }
          if (old) {
            const Pack<T, W> xo = get(iO, k), go = get(iO + 1, k);
#pragma unroll
            for (int q = 0; q < W; ++q) {
              const T s = x[k].v[q] - xo.v[q], y = gn.v[q] - go.v[q];
              dq[2] += s * s;
              dq[3] += s * y;
              dq[4] += y * y;
            }
          }
          if (zold) {
            const Pack<T, W> zo = get(iZ, k), gz = get(iZ + 1, k);
#pragma unroll
            for (int q = 0; q < W; ++q)
              dq[5] = fma_rn(x[k].v[q] - zo.v[q], gn.v[q] + gz.v[q], dq[5]);
          }
          if (a.gout) put(a.gout, k, gn);
          if (a.Xout) put(a.Xout, k, x[k]);
          if (a.Znext) put(a.Znext, k, zn);
        }
      } else if (STEP == RS_U) {
#pragma unroll
        for (int k = 0; k < MR; ++k) {
          Pack<T, W> gn;
          const Pack<T, W> b = get(1, k);
          const Pack<T, W> xn = operand(k);
#pragma unroll
          for (int q = 0; q < W; ++q) {
            const T xv = x[k].v[q], gv = g[k].v[q], gz = z[k].v[q], bv = b.v[q];
            const T zz = zstep(xv, gv, inv_rho);
            const T xw = xn.v[q];
            const T gw = acc[k].v[q] - bv;
            gn.v[q] = gw;
            const T pg = positive(xw) || negative(gw) ? gw : T(0);
            dq[0] = fma_rn(pg, pg, dq[0]);
            dq[1] = fma_rn(gw - bv, xw, dq[1]);
            const T s = xw - xv, y = gw - gv;
            dq[2] += s * s;
            dq[3] += s * y;
            dq[4] += y * y;
            dq[5] = fma_rn(xw - zz, gw + gz, dq[5]);
            zeros += is_zero(xw);
          }
          put(a.Xout, k, xn);
          put(a.gout, k, gn);
        }
      } else {
        // RS_D / RS_DZ: g(Z), D, their inner products; then <D G, D> with D as the operand tile
        Pack<T, W> d0[MR], d1[NC == 2 ? MR : 1];
#pragma unroll
        for (int k = 0; k < MR; ++k) {
          Pack<T, W> gz, l, wc, gw;
          const Pack<T, W> b = get(1, k);
          Pack<T, W> op;
          if (STEP == RS_D) op = operand(k);
          if (STEP == RS_DZ) {
            if (lx) l = get(iL, k);
            wc = get(iO, k);
            gw = get(iO + 1, k);
          }
#pragma unroll
          for (int q = 0; q < W; ++q) {
            const T zz = STEP == RS_D ? op.v[q] : x[k].v[q];
            const T xv = STEP == RS_D ? x[k].v[q] : wc.v[q], gx = STEP == RS_D ? g[k].v[q] : gw.v[q];
            T gv = acc[k].v[q] - b.v[q];
            if (lx) gv += gam * l.v[q];
            gz.v[q] = gv;
            const T d = dir(zz, gv, alpha0);
            d0[k].v[q] = d;
            if (NC == 2) d1[NC == 2 ? k : 0].v[q] = dir(zz, gv, alpha1);
            dq[0] += gv * d;
            dq[1] += d * d;
            dq[2] = fma_rn(zz - xv, gv + gx, dq[2]);
            if (NC == 2) {
              const T e = d1[NC == 2 ? k : 0].v[q];
              dq[5] += gv * e;
              dq[6] += e * e;
            }
          }
          put(a.gZout, k, gz);
          if (STEP == RS_DZ) put(a.Dout, k, d0[k]);
        }
        fetch_rest(tile + per);
#pragma unroll
        for (int m = 0; m < NC; ++m) {
          __syncthreads();  // every thread is done with the operand tile
#pragma unroll
          for (int k = 0; k < MR; ++k)
            if (on) *reinterpret_cast<Pack<T, W>*>(As + (ty + k * TY) * ls + W * tx) = m == 0 ? d0[k] : d1[NC == 2 ? k : 0];
          __syncthreads();
          if (on) {
            rowstep_product<T, W, MR>(As, ls, Gs, c4, tx, ty, TY, acc, true);
            T qq = T(0);
#pragma unroll
            for (int k = 0; k < MR; ++k)
#pragma unroll
              for (int q = 0; q < W; ++q) qq = fma(acc[k].v[q], m == 0 ? d0[k].v[q] : d1[NC == 2 ? k : 0].v[q], qq);
            dq[m == 0 ? 4 : 7] = qq;
          }
        }
      }
      if (STEP == RS_GRAD || STEP == RS_U) {
        fetch_rest(tile + per);
        dq[1] *= T(0.5);
        dq[5] *= T(0.5);
        // the rows and columns that do not exist: all zeros, which only the count sees
#pragma unroll
        for (int k = 0; k < MR; ++k) zeros -= rv[k] ? max(0, W - w) : W;
        dq[6] = (T)zeros;
      } else {
        dq[2] *= T(0.5);
      }
      total += (double)warp_sum8(dq);
      if (tile + per < tiles) __syncthreads();  // the operand tile is written again
    }
  }
  // fixed-order CTA sums, the partial record, and the control step in the restart's last CTA
  if (lane < 8) shq[lane][wid] = total;
  __syncthreads();
  if (threadIdx.x < 8) {
    double v = 0.0;
    for (int u = 0; u < (int)(blockDim.x >> 5); ++u) v += shq[threadIdx.x][u];
    a.part[((int64_t)cta * a.b + j) * kNQ + threadIdx.x] = v;
  }
  if (!a.ctl_mode) return;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    ticket = atomicAdd(&a.counters[j], 1u);
    if (ticket == (unsigned)per - 1) a.counters[j] = 0u;  // ready for the next launch
  }
  __syncthreads();
  if (ticket == (unsigned)per - 1) control_tail<8>(a, j, 0, per, NC);
}

}  // namespace

}  // namespace snmf
