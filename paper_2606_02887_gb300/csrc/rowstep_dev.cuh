// Row kernels of an Algorithm-1 step for any rank r <= 64, FP64 or FP32, as a CTA body: block-start
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
// CTA: TY MR rows of one restart, all r columns; thread (tx, ty), tx < ceil(r / 4), owns columns
// 4 tx .. of rows ty + TY p, p < MR, in the loads, the row product and the epilogue alike, so inputs
// stay in registers from the one to the other and nothing is transposed: the operand tile goes to
// shared memory row-major (stride 4 more than the columns), a thread reads 16 bytes along k of its
// rows and 16 bytes of each row of G.  Ranks between the powers of two pay for their next
// multiple of 4 only.  Bound by HBM for long factors and by launch latency for short ones.
#pragma once

#include "rowops_dev.cuh"

namespace snmf {

namespace {

enum { RS_GRAD = 0, RS_D, RS_DZ, RS_U };

constexpr int kRowGroup = 128;  // CTAs of a restart whose partial records are summed together
// groups of a restart of `per` CTAs (0: summed at once); their records follow the CTAs' in `part`
__host__ __device__ inline int rowstep_groups(int per) { return per > 4 * kRowGroup ? (per + kRowGroup - 1) / kRowGroup : 0; }

__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }

// explicit FMAs: the D step and the update compute the same bits
template <typename T>
__device__ __forceinline__ T proj0(T t) { return t > T(0) ? t : T(0); }
template <typename T>
__device__ __forceinline__ T zstep(T x, T g, T inv_rho) { return proj0(fma_rn(-g, inv_rho, x)); }
template <typename T>
__device__ __forceinline__ T dir(T z, T gz, T alpha) { return proj0(fma_rn(-alpha, gz, z)) - z; }
template <typename T>
__device__ __forceinline__ T upd(T z, T d, T pb) { return proj0(fma_rn(pb, d, z)); }

// rows of a thread of a full CTA: as many as the registers hold
template <typename T>
__host__ __device__ constexpr int rowstep_mr() { return sizeof(T) == 4 ? 4 : 2; }

// rows of a CTA and dynamic shared memory of rank r with `threads` threads and MR rows each
__host__ __device__ inline int rowstep_rows(int r, int threads, int mr) { return threads / ((r + 3) / 4) * mr; }
template <typename T>
__host__ __device__ inline size_t rowstep_smem(int r, int threads, int mr) {
  const int c = (r + 3) / 4 * 4;
  return ((size_t)rowstep_rows(r, threads, mr) * (c + 4) + (size_t)c * c) * sizeof(T);
}

// Quad columns of one row of a global array: one or two 16-byte accesses, or single values
template <typename T>
__device__ __forceinline__ Quad<T> load_quad(const T* p, bool vec, int w) {
  Quad<T> v;
  if (vec) {
    v = *reinterpret_cast<const Quad<T>*>(p);
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) v.v[q] = q < w ? p[q] : T(0);
  }
  return v;
}
template <typename T>
__device__ __forceinline__ void store_quad(T* p, const Quad<T>& v, bool vec, int w) {
  if (vec) {
    *reinterpret_cast<Quad<T>*>(p) = v;
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q < w) p[q] = v.v[q];
  }
}

// acc[p] = (row ty + TY p of As) G[:, 4 tx ..], k ascending in one chain per entry
template <typename T, int MR>
__device__ __forceinline__ void rowstep_product(const T* As, int ls, const T* Gs, int c4, int tx, int ty, int TY,
                                                Quad<T> (&acc)[MR]) {
#pragma unroll
  for (int p = 0; p < MR; ++p) acc[p] = Quad<T>{{T(0), T(0), T(0), T(0)}};
  const T* ar = As + ty * ls;
  const T* gr = Gs + 4 * tx;
#pragma unroll 2
  for (int k = 0; k < c4; k += 4) {
    Quad<T> a[MR];
#pragma unroll
    for (int p = 0; p < MR; ++p) a[p] = *reinterpret_cast<const Quad<T>*>(ar + p * TY * ls + k);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const Quad<T> g = *reinterpret_cast<const Quad<T>*>(gr + (k + u) * c4);
#pragma unroll
      for (int p = 0; p < MR; ++p) {
        if constexpr (sizeof(T) == 4) {
          const float2 aa = make_float2(a[p].v[u], a[p].v[u]);
          const float2 lo = __ffma2_rn(aa, make_float2(g.v[0], g.v[1]), make_float2(acc[p].v[0], acc[p].v[1]));
          const float2 hi = __ffma2_rn(aa, make_float2(g.v[2], g.v[3]), make_float2(acc[p].v[2], acc[p].v[3]));
          acc[p] = Quad<T>{{lo.x, lo.y, hi.x, hi.y}};
        } else {
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[p].v[q] = fma(a[p].v[u], g.v[q], acc[p].v[q]);
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

// CTA `tile` of `per` of restart j.  vec: every row of the restart starts on 16 bytes in all arrays
// (r and the pitch multiples of 4).  sm: rowstep_smem bytes.
template <typename T, int STEP, int NC, int MR>
__device__ __forceinline__ void rowstep_body(const RowArgs& a, int j, int tile, unsigned per, bool vec, T* sm) {
  __shared__ T shq[8][8];
  __shared__ unsigned ticket;
  const Ctl& cj = a.ctl[j];
  const bool live = cj.active && !(a.run && *a.run == 0);
  T dq[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) dq[m] = T(0);
  if (live) {
    const int r = a.r, TX = (r + 3) / 4, c4 = 4 * TX, ls = c4 + 4, TY = (int)blockDim.x / TX;
    const int t = threadIdx.x, ty = t / TX, tx = t - ty * TX;
    T* As = sm;
    T* Gs = sm + (size_t)TY * MR * ls;
    const bool on = ty < TY;  // the block may hold a few threads more than TX TY
    const int w = r - 4 * tx;
    const int64_t row0 = (int64_t)tile * (TY * MR) + ty;
    const int64_t off0 = row0 * a.ld + (int64_t)j * r + 4 * tx, step = (int64_t)TY * a.ld;
    const T inv_rho = (T)(1.0 / cj.rho);
    const T alpha0 = (T)(NC == 1 ? cj.alpha : cj.cand_alpha[STEP == RS_U ? (cj.dsel ? 1 : 0) : 0]);
    const T alpha1 = (T)(NC == 1 ? cj.alpha : cj.cand_alpha[1]);
    const T pb = (T)cj.phibeta;
    const T gam = (T)a.gamma;
    bool rv[MR];
    Quad<T> x[MR], g[MR], z[MR], b[MR];
    auto get = [&](const void* p, int k) {
      Quad<T> v = {{T(0), T(0), T(0), T(0)}};
      if (rv[k]) v = load_quad((const T*)p + off0 + k * step, vec, w);
      return v;
    };
    auto put = [&](void* p, int k, const Quad<T>& v) {
      if (rv[k]) store_quad((T*)p + off0 + k * step, v, vec, w);
    };
#pragma unroll
    for (int k = 0; k < MR; ++k) rv[k] = on && row0 + (int64_t)k * TY < a.n;
    // every input of the tile in flight before the first use
#pragma unroll
    for (int k = 0; k < MR; ++k) {
      x[k] = get(STEP == RS_U ? a.Xout : a.X, k);
      if (STEP == RS_D) g[k] = get(a.g_in, k);
      if (STEP == RS_U) {
        g[k] = get(a.gout, k);
        z[k] = get(a.gZold, k);
      }
      b[k] = get(a.B, k);
    }
    {
      const T* G = (const T*)a.G + (int64_t)j * r * r;
      for (int e = t; e < c4 * c4; e += blockDim.x) {
        const int p = e / c4, q = e - p * c4;
        Gs[e] = p < r && q < r ? G[p * r + q] : T(0);
      }
    }
    // the operand tile: X, Z or X' (z: g(Z) on entry of RS_U, then X')
#pragma unroll
    for (int k = 0; k < MR; ++k) {
      Quad<T> op = x[k];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (STEP == RS_D) op.v[q] = zstep(x[k].v[q], g[k].v[q], inv_rho);
        if (STEP == RS_U) {
          const T zz = zstep(x[k].v[q], g[k].v[q], inv_rho);
          op.v[q] = upd(zz, dir(zz, z[k].v[q], alpha0), pb);
        }
      }
      if (on) *reinterpret_cast<Quad<T>*>(As + (ty + k * TY) * ls + 4 * tx) = op;
    }
    __syncthreads();
    Quad<T> acc[MR];
    if (on) rowstep_product<T, MR>(As, ls, Gs, c4, tx, ty, TY, acc);
    if (STEP == RS_GRAD) {
#pragma unroll
      for (int k = 0; k < MR; ++k) {
        if (!rv[k]) continue;
        Quad<T> gn, l, zn;
        if (a.LX) l = get(a.LX, k);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const T xv = x[k].v[q], bv = b[k].v[q];
          T gv = acc[k].v[q] - bv;
          if (a.LX) gv += gam * l.v[q];
          gn.v[q] = gv;
          zn.v[q] = zstep(xv, gv, inv_rho);
          if (q >= w) continue;
          const T pg = xv > T(0) ? gv : (gv < T(0) ? gv : T(0));
          dq[0] += pg * pg;
          dq[1] += T(0.5) * (gv - bv) * xv;
          if (xv == T(0)) dq[6] += T(1);
        }
        if (a.Xold) {
          const Quad<T> xo = get(a.Xold, k), go = get(a.gold, k);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const T s = x[k].v[q] - xo.v[q], y = gn.v[q] - go.v[q];
            if (q >= w) continue;
            dq[2] += s * s;
            dq[3] += s * y;
            dq[4] += y * y;
          }
        }
        if (a.Zold) {
          const Quad<T> zo = get(a.Zold, k), gz = get(a.gZold, k);
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (q < w) dq[5] += T(0.5) * (x[k].v[q] - zo.v[q]) * (gn.v[q] + gz.v[q]);
        }
        if (a.gout) put(a.gout, k, gn);
        if (a.Xout) put(a.Xout, k, x[k]);
        if (a.Znext) put(a.Znext, k, zn);
      }
    } else if (STEP == RS_U) {
#pragma unroll
      for (int k = 0; k < MR; ++k) {
        if (!rv[k]) continue;
        Quad<T> xn, gn;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const T xv = x[k].v[q], gv = g[k].v[q], gz = z[k].v[q], bv = b[k].v[q];
          const T zz = zstep(xv, gv, inv_rho);
          const T xw = upd(zz, dir(zz, gz, alpha0), pb);
          const T gw = acc[k].v[q] - bv;
          xn.v[q] = xw;
          gn.v[q] = gw;
          if (q >= w) continue;
          const T pg = xw > T(0) ? gw : (gw < T(0) ? gw : T(0));
          dq[0] += pg * pg;
          dq[1] += T(0.5) * (gw - bv) * xw;
          const T s = xw - xv, y = gw - gv;
          dq[2] += s * s;
          dq[3] += s * y;
          dq[4] += y * y;
          dq[5] += T(0.5) * (xw - zz) * (gw + gz);
          if (xw == T(0)) dq[6] += T(1);
        }
        put(a.Xout, k, xn);
        put(a.gout, k, gn);
      }
    } else {
      // RS_D / RS_DZ: g(Z), D, their inner products; then <D G, D> with D as the operand tile
      Quad<T> d0[MR], d1[NC == 2 ? MR : 1];
#pragma unroll
      for (int k = 0; k < MR; ++k) {
        Quad<T> gz, l, wc, gw;
        if (STEP == RS_DZ) {
          if (a.LX) l = get(a.LX, k);
          wc = get(a.Wcur, k);
          gw = get(a.gWcur, k);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const T zz = STEP == RS_D ? zstep(x[k].v[q], g[k].v[q], inv_rho) : x[k].v[q];
          const T xv = STEP == RS_D ? x[k].v[q] : wc.v[q], gx = STEP == RS_D ? g[k].v[q] : gw.v[q];
          T gv = acc[k].v[q] - b[k].v[q];
          if (STEP == RS_DZ && a.LX) gv += gam * l.v[q];
          gz.v[q] = gv;
          const bool in = rv[k] && q < w;
          const T d = in ? dir(zz, gv, alpha0) : T(0);
          d0[k].v[q] = d;
          if (NC == 2) d1[NC == 2 ? k : 0].v[q] = in ? dir(zz, gv, alpha1) : T(0);
          if (!in) continue;
          dq[0] += gv * d;
          dq[1] += d * d;
          dq[2] += T(0.5) * (zz - xv) * (gv + gx);
          if (NC == 2) {
            const T e = d1[NC == 2 ? k : 0].v[q];
            dq[5] += gv * e;
            dq[6] += e * e;
          }
        }
        put(a.gZout, k, gz);
        if (STEP == RS_DZ) put(a.Dout, k, d0[k]);
      }
#pragma unroll
      for (int m = 0; m < NC; ++m) {
        __syncthreads();  // every thread is done with the operand tile
#pragma unroll
        for (int k = 0; k < MR; ++k)
          if (on) *reinterpret_cast<Quad<T>*>(As + (ty + k * TY) * ls + 4 * tx) = m == 0 ? d0[k] : d1[NC == 2 ? k : 0];
        __syncthreads();
        if (on) {
          rowstep_product<T, MR>(As, ls, Gs, c4, tx, ty, TY, acc);
          T qq = T(0);
#pragma unroll
          for (int k = 0; k < MR; ++k)
#pragma unroll
            for (int q = 0; q < 4; ++q) qq = fma(acc[k].v[q], m == 0 ? d0[k].v[q] : d1[NC == 2 ? k : 0].v[q], qq);
          dq[m == 0 ? 4 : 7] = qq;
        }
      }
    }
  }
  // fixed-order CTA sums, the partial record, and the control step in the restart's last CTA
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  {
    const T v = warp_sum8(dq);
    if (lane < 8) shq[lane][wid] = v;
  }
  __syncthreads();
  if (threadIdx.x < 8) {
    T v = T(0);
    for (int u = 0; u < (int)(blockDim.x >> 5); ++u) v += shq[threadIdx.x][u];
    a.part[((int64_t)tile * a.b + j) * kNQ + threadIdx.x] = (double)v;
  }
  if (!a.ctl_mode) return;
  // the restart's last CTA runs its control step.  Where many CTAs make up a restart, the last of
  // each kRowGroup of them sums the group's records first (n = 2e6, r = 32: 31250 CTAs)
  auto arrive = [&](unsigned* counter, unsigned of) {
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
      ticket = atomicAdd(counter, 1u);
      if (ticket == of - 1) *counter = 0u;  // ready for the next launch
    }
    __syncthreads();
    return ticket == of - 1;
  };
  const int ng = a.gcounters ? rowstep_groups((int)per) : 0;
  if (!ng) {
    if (arrive(&a.counters[j], per)) control_tail<8>(a, j, 0, (int)per, NC);
    return;
  }
  const int grp = tile / kRowGroup, first = grp * kRowGroup, size = min(kRowGroup, (int)per - first);
  if (!arrive(&a.gcounters[(int64_t)j * ng + grp], size)) return;
  __shared__ double rec[8][8], qs[8];
  slot_sums<8>(a.part + (int64_t)first * a.b * kNQ, size, a.b, j, rec, qs);
  if (threadIdx.x < 8) a.part[((int64_t)(per + grp) * a.b + j) * kNQ + threadIdx.x] = qs[threadIdx.x];
  if (arrive(&a.counters[j], ng)) control_tail<8>(a, j, (int)per, ng, NC);
}

}  // namespace

}  // namespace snmf
