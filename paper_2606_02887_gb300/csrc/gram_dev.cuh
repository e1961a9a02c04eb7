// Gram X^T Y of a row-major factor and the power method on it, as CTA bodies: one launch per
// Gram in rowops.cu (a restart = a column range), work items of the uneven batch in batch.cu.
#pragma once

#include <math.h>

#include <type_traits>

#include "common.cuh"

namespace snmf {

namespace {

// The Gram tile is as wide as the rank needs (16, 32 or 64 columns; tiles of 64 above), so a
// rank of 10 or 20 does not pay for a 64 x 64 tile.
__host__ __device__ inline int gram_tw(int r) { return r <= 16 ? 16 : (r <= 32 ? 32 : 64); }

constexpr int kGramGroup = 16;         // chunk partials summed by one CTA at each level
constexpr int kGramStageBytes = 8192;  // one staged operand block
constexpr int kGramStages = 3;

template <typename T>
constexpr size_t gram_smem(bool same) {
  // the staging ring; after the row loop the same memory holds the 4096 tile partials
  return kGramStages * kGramStageBytes * (same ? 1 : 2) > 4096 * sizeof(T)
             ? (size_t)kGramStages * kGramStageBytes * (same ? 1 : 2)
             : 4096 * sizeof(T);
}

template <typename T>
struct alignas(16) Quad {
  T v[4];
};

__device__ __forceinline__ Quad<float> ldcg_quad(const float* p) {
  const float4 t = __ldcg(reinterpret_cast<const float4*>(p));
  return {{t.x, t.y, t.z, t.w}};
}
__device__ __forceinline__ Quad<double> ldcg_quad(const double* p) {
  const double2 a = __ldcg(reinterpret_cast<const double2*>(p)), b = __ldcg(reinterpret_cast<const double2*>(p) + 1);
  return {{a.x, a.y, b.x, b.y}};
}

// 16-, 8- or 4-byte asynchronous copy to shared memory; bytes beyond `valid` are zero
template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src, bool valid) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  const int n = valid ? BYTES : 0;
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(d), "l"(src), "n"(BYTES), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ------------------------------------------------------------------------------
// Power method (Alg. 1 line 2, Eq. (2.11)): ||G||_2 by `iters` iterations from the ones vector
// and the Rayleigh quotient.  The block holds G; row p of G v is summed by TPR adjacent lanes,
// W = P2 / TPR columns each (P2: r rounded up to a power of two), through `dot(v)`.  A fixed
// count of serial products bounds it, so an iteration is one shared read of v, the FMAs, the
// lane butterfly and one barrier: v is double buffered and G scaled by a power of two to a
// trace below one (exact; ||G|| <= trace for a Gram), so v only has to be rescaled every eighth
// iteration (it shrinks by at most 2 r each).  n = 64: 13 us with the norm taken in every
// iteration, 4 us so.
// Threads t < nact = P2 TPR take part (a multiple of 32), on barrier 1.  vs: 2 (P2 + 4 TPR)
// values, red: 2 nact / 32 values.  0 for a zero G.
// ------------------------------------------------------------------------------
__device__ __forceinline__ void bar_sync(int id, int count) {
  asm volatile("barrier.cta.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}

template <typename T>
__device__ __forceinline__ T lanes_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <typename T, int TPR, typename Dot>
__device__ __forceinline__ T power_norm(int r, int W, int nact, int iters, Dot dot, T* vs, T* red) {
  const int t = threadIdx.x, p = t / TPR, part = t % TPR;
  const int lane = t & 31, wid = t >> 5, nw = nact >> 5;
  const int len = (W + 4) * TPR;                        // columns of a part, 16 bytes apart in banks
  auto at = [&](int q) { return q + (q / W) * 4; };
  T* cur = vs;
  T* nxt = vs + len;
  if (part == 0) cur[at(p)] = p < r ? T(1) : T(0);
  bar_sync(1, nact);
  auto total = [&](T x) {  // fixed-order sum over the rows (x counts in part 0 only)
    x = lanes_sum(part == 0 ? x : T(0));
    if (lane == 0) red[wid] = x;
    bar_sync(1, nact);
    T s = T(0);
    for (int w = 0; w < nw; ++w) s += red[w];
    return s;
  };
  auto row = [&]() {
    T s = dot(cur + part * (W + 4));
#pragma unroll
    for (int o = 1; o < TPR; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
  };
  for (int it = 0; it < iters; ++it) {
    T s = row();
    // scaled by a power of two every eighth time (FP64 every 32nd: G's norm is between 1 / (2 r) and 1,
    // and neither the vector nor its square leaves the range), by the largest exponent: integer steps,
    // where a sum and a division are 17 FP64 instructions of 64 cycles
    const bool scale = sizeof(T) == 8 ? (it & 31) == 31 : (it & 7) == 7 || it == iters - 1;
    if (scale) {
      const unsigned hi = sizeof(T) == 8 ? (unsigned)__double2hiint((double)s) & 0x7fffffffu
                                         : __float_as_uint((float)s) & 0x7fffffffu;
      const unsigned m = __reduce_max_sync(0xffffffffu, hi);
      unsigned* ru = reinterpret_cast<unsigned*>(red);
      if (lane == 0) ru[wid] = m;
      bar_sync(1, nact);
      unsigned top = 0u;
      for (int w = 0; w < nw; ++w) top = max(top, ru[w]);
      if (top == 0u) return T(0);
      constexpr int MB = sizeof(T) == 8 ? 20 : 23, BIAS = sizeof(T) == 8 ? 1023 : 127;
      const int ex = min(max((int)(top >> MB), 1), 2 * BIAS - 1);  // 2^(BIAS - ex) is a normal number
      const unsigned sc = (unsigned)(2 * BIAS - ex) << MB;
      s *= sizeof(T) == 8 ? (T)__hiloint2double((int)sc, 0) : (T)__uint_as_float(sc);
    }
    if (part == 0) nxt[at(p)] = s;
    bar_sync(1, nact);
    T* x = cur;
    cur = nxt;
    nxt = x;
  }
  const T s = row(), v = cur[at(p)];
  const T num = total(v * s);
  bar_sync(1, nact);  // red read by every thread before it is written again
  const T den = total(v * v);
  return den == T(0) ? T(0) : num / den;
}

// power-of-two scale that brings a positive trace below one
__device__ __forceinline__ int trace_exponent(float tr) { return tr > 0.f && tr < INFINITY ? ilogbf(tr) + 1 : 0; }
__device__ __forceinline__ int trace_exponent(double tr) { return tr > 0.0 && tr < INFINITY ? ilogb(tr) + 1 : 0; }

__device__ __forceinline__ void set_rho(Ctl& c, double norm, double rho_scale, double rho_shift) {
  double rr = rho_scale * norm + rho_shift;  // shift: gamma ||L||_2 of a graph block
  if (!(rr > 0.0)) rr = 1.0;                 // zero Gram: unit scaling
  c.rho = rr;
}

// rho of the r x r Gram in shared memory (row stride TW, zero beyond r), r <= TW
template <typename T, int TW>
__device__ __forceinline__ void rho_in_smem(const T* Gs, int r, int iters, double rho_scale, double rho_shift, Ctl& c) {
  constexpr int W = TW / 4, NACT = 4 * TW;
  __shared__ __align__(16) T vs[2 * (TW + 16)];
  __shared__ T red[2 * NACT / 32];
  const int t = threadIdx.x;
  if (t >= NACT) return;
  const int lane = t & 31;
  T tr = T(0);
  for (int q = lane; q < r; q += 32) tr += Gs[q * TW + q];
  tr = lanes_sum(tr);
  const int e = trace_exponent(tr);
  T g[W];
#pragma unroll
  for (int u = 0; u < W; ++u) g[u] = (T)ldexp(Gs[(t >> 2) * TW + (t & 3) * W + u], -e);
  const T norm = power_norm<T, 4>(r, W, NACT, iters,
                                  [&](const T* v) {
                                    if constexpr (sizeof(T) == 8) {  // one chain: no FP64 instruction hides another
                                      T s = g[0] * v[0];
#pragma unroll
                                      for (int u = 1; u < W; ++u) s = fma(g[u], v[u], s);
                                      return s;
                                    }
                                    T s[4] = {T(0), T(0), T(0), T(0)};
#pragma unroll
                                    for (int u = 0; u < W; u += 4) {
                                      const Quad<T> x = *reinterpret_cast<const Quad<T>*>(v + u);
#pragma unroll
                                      for (int k = 0; k < 4; ++k) s[k] = fma(g[u + k], x.v[k], s[k]);
                                    }
                                    return (s[0] + s[1]) + (s[2] + s[3]);
                                  },
                                  vs, red);
  if (t == 0) set_rho(c, ldexp((double)norm, e), rho_scale, rho_shift);
}

// ------------------------------------------------------------------------------
// One chunk of rows [i_begin, i_end) of a TP x TQ tile of X^T Y: X, Y at the tile's first columns
// (wx, wy of them exist), row pitches ldx, ldy, VEC elements per copy (16 bytes when the columns and
// the pitches allow it, else single elements).  256 threads: NG = 256 M M / (TP TQ) row groups, each a
// (TP / M) x (TQ / M) grid of M x M micro tiles, M = 4 read as two 16-byte shared loads per row.  The
// groups' sums leave the row loop in shared memory; the thread returns its entries e = 4 (t + 256 u).
// NG = 1: every entry is one chain over the chunk's rows in order.
// Bound by HBM for long factors (n = 2e6, r = 32: 797 us with 152 chunks of two staged rounds
// and scalar shared reads, 177 us so) and by latency for short ones.
// ------------------------------------------------------------------------------
template <int TP, int TQ>
__host__ __device__ constexpr int tile_quads() { return TP * TQ >= 1024 ? TP * TQ / 1024 : 1; }  // 16-byte entries per thread

template <typename T, int TP, int TQ, int VEC, int M = 4>
__device__ __forceinline__ void gram_chunk(const T* __restrict__ X, const T* __restrict__ Y, int wx, int wy, int64_t ldx,
                                           int64_t ldy, int64_t i_begin, int64_t i_end, bool same, T* sm,
                                           Quad<T> (&out)[tile_quads<TP, TQ>()]) {
  constexpr int TM = TP > TQ ? TP : TQ;
  constexpr int RS = kGramStageBytes / (TM * (int)sizeof(T));  // rows per stage
  constexpr int NG = 256 * M * M / (TP * TQ), GT = 256 / NG, TX = TQ / M;
  constexpr int SX = RS * TP, SY = RS * TQ;
  const int t = threadIdx.x;
  T* Xs = sm;
  T* Ys = same ? sm : sm + kGramStages * SX;
  auto copy = [&](auto width, const T* P, int w, int64_t ld, T* dst, int64_t i0) {
    constexpr int TW = decltype(width)::value, CPR = TW / VEC, NC = (RS * CPR + 255) / 256;
#pragma unroll
    for (int m = 0; m < NC; ++m) {
      const int e = t + 256 * m, rr = e / CPR, cc = (e % CPR) * VEC;
      if (RS * CPR % 256 && e >= RS * CPR) break;
      const int64_t i = i0 + rr;
      const bool v = i < i_end && cc < w;
      cp_async<VEC * (int)sizeof(T)>(dst + rr * TW + cc, v ? P + i * ld + cc : P, v);
    }
  };
  auto fetch = [&](int64_t i0, int st) {
    copy(std::integral_constant<int, TP>{}, X, wx, ldx, Xs + st * SX, i0);
    if (!same) copy(std::integral_constant<int, TQ>{}, Y, wy, ldy, Ys + st * SY, i0);
  };
  const int rounds = (int)((i_end - i_begin + RS - 1) / RS);
#pragma unroll
  for (int s = 0; s < kGramStages - 1; ++s) {
    if (s < rounds) fetch(i_begin + (int64_t)s * RS, s);
    cp_async_commit();
  }
  struct alignas(M * sizeof(T) < 16 ? M * sizeof(T) : 16) Few {
    T v[M];
  };
  T acc[M][M];
#pragma unroll
  for (int a = 0; a < M; ++a)
#pragma unroll
    for (int c = 0; c < M; ++c) acc[a][c] = T(0);
  const int grp = t / GT, tx = (t % GT) % TX, ty = (t % GT) / TX;
  for (int k = 0; k < rounds; ++k) {
    cp_async_wait<kGramStages - 2>();
    __syncthreads();  // stage k is in; every thread is done with the stage refilled below
    if (k + kGramStages - 1 < rounds)
      fetch(i_begin + (int64_t)(k + kGramStages - 1) * RS, (k + kGramStages - 1) % kGramStages);
    cp_async_commit();
    const T* xs = Xs + (k % kGramStages) * SX + M * ty;
    const T* ys = Ys + (k % kGramStages) * SY + M * tx;
#pragma unroll 4
    for (int rr = grp; rr < RS; rr += NG) {
      const Few xa = *reinterpret_cast<const Few*>(xs + rr * TP);
      const Few yb = *reinterpret_cast<const Few*>(ys + rr * TQ);
#pragma unroll
      for (int a = 0; a < M; ++a)
#pragma unroll
        for (int c = 0; c < M; ++c) acc[a][c] = fma(xa.v[a], yb.v[c], acc[a][c]);
    }
  }
  cp_async_wait<0>();
  __syncthreads();  // the ring is free: it takes the groups' tiles
#pragma unroll
  for (int a = 0; a < M; ++a) {
    Few f;
#pragma unroll
    for (int c = 0; c < M; ++c) f.v[c] = acc[a][c];
    *reinterpret_cast<Few*>(sm + grp * TP * TQ + (M * ty + a) * TQ + M * tx) = f;
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < tile_quads<TP, TQ>(); ++u) {
    const int e = 4 * (t + 256 * u);
    if (e < TP * TQ) {
      Quad<T> s = *reinterpret_cast<const Quad<T>*>(sm + e);
#pragma unroll
      for (int g = 1; g < NG; ++g) {
        const Quad<T> v = *reinterpret_cast<const Quad<T>*>(sm + g * TP * TQ + e);
#pragma unroll
        for (int k = 0; k < 4; ++k) s.v[k] += v.v[k];
      }
      out[u] = s;
    }
  }
}

// Sum of the tiles of CTAs c = 0 .. nch - 1, each with its entries in s: true in one CTA, which holds
// the sum.  Partials go to gp (nch + ng tiles of TT values) and are summed in chunk order by the
// last CTA of each of the ng groups of 16 chunks and then, in group order, by the last group's
// (arrival counters cnt[0 .. ng], zero between launches): a fixed order, and no CTA reads many
// partials in a row, which had kept the number of chunks, and with it the CTAs, low.  ng = 0: one
// level, every chunk in order.
__host__ __device__ inline int gram_groups(int nch) { return nch > kGramGroup ? (nch + kGramGroup - 1) / kGramGroup : 0; }

template <typename T, int TT, int NE>
__device__ __forceinline__ bool sum_chunks(Quad<T> (&s)[NE], int c, int nch, int ng, T* gp, unsigned* cnt) {
  __shared__ unsigned s_ticket;
  const int t = threadIdx.x;
  const bool owns = 4 * t < TT;
  if (nch == 1) return true;
  auto publish = [&](T* dst) {
#pragma unroll
    for (int u = 0; u < NE; ++u)
      if (owns) *reinterpret_cast<Quad<T>*>(dst + 4 * (t + 256 * u)) = s[u];
    __threadfence();
    __syncthreads();
  };
  auto arrive = [&](unsigned* counter, int of) {  // CTA-uniform: the last of `of` arrivals
    if (t == 0) {
      s_ticket = atomicAdd(counter, 1u);
      if (s_ticket == (unsigned)(of - 1)) *counter = 0u;  // ready for the next launch
    }
    __syncthreads();
    const bool last = s_ticket == (unsigned)(of - 1);
    __syncthreads();
    return last;
  };
  auto sum = [&](const T* src, int m) {  // s = the m tiles at src in order, 8 loads in flight
#pragma unroll
    for (int u = 0; u < NE; ++u) {
      s[u] = Quad<T>{{T(0), T(0), T(0), T(0)}};
      if (!owns) continue;
      const T* q = src + 4 * (t + 256 * u);
      for (int k0 = 0; k0 < m; k0 += 8) {
        Quad<T> v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k)
          v[k] = k0 + k < m ? ldcg_quad(q + (int64_t)(k0 + k) * TT) : Quad<T>{{T(0), T(0), T(0), T(0)}};
#pragma unroll
        for (int k = 0; k < 8; ++k)
#pragma unroll
          for (int w = 0; w < 4; ++w) s[u].v[w] += v[k].v[w];
      }
    }
  };
  publish(gp + (int64_t)c * TT);
  const int g = c / kGramGroup, gs = min(kGramGroup, nch - g * kGramGroup);
  if (!arrive(cnt + (ng ? 1 + g : 0), ng ? gs : nch)) return false;
  __threadfence();
  sum(gp + (int64_t)(ng ? g * kGramGroup : 0) * TT, ng ? gs : nch);
  if (ng) {
    publish(gp + (int64_t)(nch + g) * TT);
    if (!arrive(cnt, ng)) return false;
    __threadfence();
    sum(gp + (int64_t)nch * TT, ng);
  }
  return true;
}

// Where a Gram tile goes: entry (p, q) of the tile is (p0 + p, q0 + q) of the r x r matrix.
template <typename T>
struct GramOut {
  double* G64;
  T* GT;  // factor-type copy with lam on the diagonal (NULL: none)
  T lam;
  int r, p0, q0;
  Ctl* rho_ctl;  // the tile is the whole Gram: rho = rho_scale ||G||_2 + rho_shift (NULL: no)
  int rho_iters;
  double rho_scale, rho_shift;
};

// CTA `c` of the nch chunks of one Gram tile (see sum_chunks).
template <typename T, int TW, int VEC, int M = 4>
__device__ __forceinline__ void gram_body(const T* X, const T* Y, int wx, int wy, int64_t ld, int64_t n, int64_t chunk,
                                          int c, int nch, int ng, bool same, T* gp, unsigned* cnt, const GramOut<T>& o,
                                          T* sm) {
  constexpr int NE = tile_quads<TW, TW>();
  const int t = threadIdx.x;
  const bool owns = 4 * t < TW * TW;
  Quad<T> s[NE];
  const int64_t i0 = (int64_t)c * chunk;
  gram_chunk<T, TW, TW, VEC, M>(X, Y, wx, wy, ld, ld, i0, min(n, i0 + chunk), same, sm, s);
  if (!sum_chunks<T, TW * TW>(s, c, nch, ng, gp, cnt)) return;
#pragma unroll
  for (int u = 0; u < NE; ++u) {
    const int e = 4 * (t + 256 * u);
    if (!owns) continue;
    if (o.rho_ctl) *reinterpret_cast<Quad<T>*>(sm + e) = s[u];
    const int p = o.p0 + e / TW;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int q = o.q0 + e % TW + k;
      if (p < o.r && q < o.r) {
        o.G64[(int64_t)p * o.r + q] = (double)s[u].v[k];
        if (o.GT) o.GT[(int64_t)p * o.r + q] = s[u].v[k] + (p == q ? o.lam : T(0));
      }
    }
  }
  if (o.rho_ctl) {
    __syncthreads();
    rho_in_smem<T, TW>(sm, o.r, o.rho_iters, o.rho_scale, o.rho_shift, *o.rho_ctl);
  }
}

}  // namespace

}  // namespace snmf
