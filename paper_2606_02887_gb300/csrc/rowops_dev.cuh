// Device bodies shared by the per-restart kernels (rowops.cu) and the grouped kernels of
// the uneven batch (batch.cu): fixed-order slot reductions, the FP64 control steps of
// Algorithm 1 and the row GEMM with its fused epilogues.  The bodies take their
// CTA coordinates as arguments, so one CTA of either launcher runs one work item.
#pragma once

#include <math.h>

#include <type_traits>

#include "common.cuh"
#include "gram_dev.cuh"
#include "mlp_dev.cuh"
#include "rowops.cuh"

namespace snmf {

namespace {

inline int cdiv(int64_t a, int64_t b) { return (int)((a + b - 1) / b); }
inline int64_t imin64(int64_t a, int64_t b) { return a < b ? a : b; }
inline int64_t imax64(int64_t a, int64_t b) { return a > b ? a : b; }

// ------------------------------------------------------------------------------
// control helpers and bodies (run by one block: a control kernel, or the last CTA of
// a producing kernel for that restart)
// ------------------------------------------------------------------------------
// Block-wide fixed-order reductions (any multiple of 32 threads up to 256): thread t sums entries t,
// t + blockDim, ... in order, then block_sum; every thread gets the same value.  `sh` holds 32
// doubles.  (One warp took 53 us for the r = 100 dot of three restarts, and 245 us for the 31250
// slots of n = 2e6.)
__device__ double reduce_slots(const double* part, int nslots, int b, int j, int q, double* sh) {
  double s = 0.0;
  const int nt = blockDim.x;
  int t = threadIdx.x;
  for (; t + 3 * nt < nslots; t += 4 * nt) {  // four loads in flight, summed in slot order
    double v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = __ldcg(part + ((int64_t)(t + u * nt) * b + j) * kNQ + q);
#pragma unroll
    for (int u = 0; u < 4; ++u) s += v[u];
  }
  for (; t < nslots; t += nt) s += __ldcg(part + ((int64_t)t * b + j) * kNQ + q);
  return block_sum(s, sh);
}

// The first NV quantities of restart j, summed over the slots into qs[NV] (shared): NV / 2 threads
// per slot read its record as 16-byte pairs.  sh: [8][NV] shared.  Ends with a barrier.
// Four warps at most: an FP64 instruction occupies its SM partition for 64 cycles whatever the lanes
// that are on, so more warps only add instructions to the shuffles and the last sum.
template <int NV>
__device__ __forceinline__ void slot_sums(const double* part, int nslots, int b, int j, double (*sh)[NV], double* qs) {
  constexpr int TPS = NV / 2;
  const int nt = min((int)blockDim.x, 128);
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5, step = nt / TPS, q = t % TPS;
  if (t < nt) {
    double s0 = 0.0, s1 = 0.0;
    auto ld = [&](int k) { return __ldcg(reinterpret_cast<const double2*>(part + ((int64_t)k * b + j) * kNQ) + q); };
    int k = t / TPS;
    for (; k + 3 * step < nslots; k += 4 * step) {
      double2 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = ld(k + u * step);
#pragma unroll
      for (int u = 0; u < 4; ++u) { s0 += v[u].x; s1 += v[u].y; }
    }
    for (; k < nslots; k += step) {
      const double2 v = ld(k);
      s0 += v.x;
      s1 += v.y;
    }
#pragma unroll
    for (int o = TPS; o < 32; o <<= 1) {
      s0 += __shfl_xor_sync(0xffffffffu, s0, o);
      s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    }
    if (lane < TPS) {
      sh[wid][2 * lane] = s0;
      sh[wid][2 * lane + 1] = s1;
    }
  }
  __syncthreads();
  if (t < NV) {
    double v = sh[0][t];
    for (int w = 1; w < nt >> 5; ++w) v += sh[w][t];
    qs[t] = v;
  }
  __syncthreads();
}

// The same by one warp (eight quantities), for a kernel whose other warps are at work.
__device__ __forceinline__ void slot_sums_warp(const double* part, int nslots, int b, int j, double* out) {
  const int lane = threadIdx.x & 31;
  double s0 = 0.0, s1 = 0.0;
  for (int k = lane >> 2; k < nslots; k += 8) {
    const double2 v = __ldcg(reinterpret_cast<const double2*>(part + ((int64_t)k * b + j) * kNQ) + (lane & 3));
    s0 += v.x;
    s1 += v.y;
  }
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) {
    s0 += __shfl_xor_sync(0xffffffffu, s0, o);
    s1 += __shfl_xor_sync(0xffffffffu, s1, o);
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) out[q] = __shfl_sync(0xffffffffu, q & 1 ? s1 : s0, q >> 1);
}

// sum_e A[e] B[e] over r*r entries; A/B FP64 matrices.
__device__ double dot_rr(const double* A, const double* B, int r, double* sh) {
  double s = 0.0;
  for (int e = threadIdx.x; e < r * r; e += blockDim.x) s += __ldcg(A + e) * __ldcg(B + e);
  return block_sum(s, sh);
}

__device__ double bb_step(const Ctl& c, const Params& P, double rho) {
  // Alg. 1 line 3 / Eq. (2.10), with the fallback 1/rho when <S,Y> <= 0
  double a;
  if (!(c.sy > 0.0)) a = 1.0 / rho;
  else a = (P.bb == 0) ? c.ss / c.sy : c.sy / c.yy;
  return fmin(P.alpha_max, fmax(P.alpha_min, a));
}

__device__ __forceinline__ bool finite_bits(double x) {
  return (__double_as_longlong(x) & 0x7ff0000000000000ll) != 0x7ff0000000000000ll;
}

__device__ void hist_reset(Ctl& c, double f) {
  c.hlen = 1;
  c.hpos = 0;
  c.fhist[0] = f;
}

__device__ void hist_push(Ctl& c, double f, int M) {
  const int cap = M > 0 ? M : 1;
  c.hpos = (c.hpos + 1) % cap;
  c.fhist[c.hpos] = f;
  if (c.hlen < cap) c.hlen++;
}

// F_k of Alg. 1 line 4 (eta averaging) or the max of the last M values; called at k > 0
// after f(X_k) has been pushed.
__device__ double reference(const Ctl& c, const Params& P) {
  if (P.memory > 0) {
    // maximum by the ordered bits (NaN left out): an FP64 comparison takes 64 cycles
    long long m = (long long)0xfff0000000000000ull ^ 0x7fffffffffffffffll;  // -inf
    for (int t = 0; t < c.hlen; ++t) {
      const long long v = __double_as_longlong(c.fhist[t]), a = v & 0x7fffffffffffffffll;
      if (a <= 0x7ff0000000000000ll) m = max(m, v < 0 ? v ^ 0x7fffffffffffffffll : v);
    }
    return __longlong_as_double(m < 0 ? m ^ 0x7fffffffffffffffll : m);
  }
  return c.f + P.eta * (c.F - c.f);
}

// Penalty block start: joint projected gradient / convergence (W block), reset of the
// block's reference (Alg. 1 line 4: F_0 = f(X_0)) and alpha_0 = 1/rho.  One thread; qs: the summed
// partials of the producing kernel (q: 0 pg2).
__device__ void pen_start_body(Ctl& c, const double* qs, int j, const Params& P, int is_w_block, int first) {
  const double pg2 = qs[0];
  if (is_w_block) {
    const double joint = sqrt(pg2 + c.pgH2);
    c.pg = joint;
    if (c.iters == 0) c.pg0 = joint;
    const bool stop = c.iters > 0 && (joint <= P.tol * c.pg0 || c.iters >= P.max_iter);
    const bool bad = !stop && !isfinite(joint);
    if (P.ring && P.ring_cap > 0) {  // statistics of the state reached by the last outer iteration
      double* rec = P.ring + ((int64_t)j * P.ring_cap + (c.iters % P.ring_cap)) * kRingVals;
      rec[0] = (double)c.iters;
      rec[1] = c.pg0 > 0.0 ? joint / c.pg0 : 0.0;
      rec[2] = joint;
      rec[3] = c.alpha;
      rec[4] = c.beta;
      rec[5] = (double)c.ls_fail;
      rec[6] = (double)c.mlp_accept;
      rec[7] = (stop || bad) ? 0.0 : 1.0;  // 1: the restart goes on
    }
    if (stop) { c.active = 0; return; }
    if (bad) { c.nan_seen = 1; c.active = 0; return; }
  } else {
    if (first) { c.pgH2 = pg2; return; }  // solve initialisation: H gradient at start
  }
  c.f = 0.0;  // block-relative objective: f(X_0) = 0
  c.F = 0.0;
  hist_reset(c, 0.0);
  c.k = 0;
  c.alpha = 1.0 / c.rho;
  for (int m = 0; m < kNCand; ++m) c.cand_alpha[m] = c.alpha;  // k = 0: every candidate is 1/rho
  c.dsel = 0;
  c.feat_ok = 0;
  c.pg_prev = sqrt(pg2);
  c.last_dec = 0.0;
}

// backtracking from beta = 1 on f(Z + beta D) - f(Z) = beta gd + beta^2/2 q against the
// reference (Alg. 1 line 4); returns beta (0 when no trial is accepted)
__device__ double backtrack(double fZ, double F, double gd, double q, const Params& P, bool* ok) {
  // beta = 1 by itself: four FP64 instructions instead of ten, and the usual end (max_ls >= 1)
  if (fZ + gd + 0.5 * q <= F + P.theta * gd) { *ok = true; return 1.0; }
  double beta = P.beta_shrink;
  for (int t = 1; t < P.max_ls; ++t) {
    const double fz = fZ + beta * gd + 0.5 * beta * beta * q;
    if (fz <= F + P.theta * beta * gd) { *ok = true; return beta; }
    beta *= P.beta_shrink;
  }
  *ok = false;
  return 0.0;
}

// Line search after the D direction (q: 0 gd, 1 dd, 2 f(Z)-f(X_k)), one thread:
// f(Z + beta D) - f(Z) = beta gd + beta^2/2 q, q = <D (H H^T + lambda I), D> + gamma <D, L D>.
// nc = 2 (learned controller): candidate 0 is the proposal, accepted only at beta = 1, else
// the plain BB direction (candidate 1) with ordinary backtracking.  The lean learned step
// (controller 3) has one candidate, the proposal, with ordinary backtracking.  nc = 9 (record mode):
// every candidate multiplier is line-searched, the best accepted decrease is recorded as
// the training label, and the plain BB candidate (index 4) is followed.
__device__ void pen_ls_body(Ctl& c, const double* qs, double q, const Params& P, int nc = 1) {
  const double gd = qs[0], dzw = qs[2];
  c.fZ = c.f + dzw;
  if (c.k > 0) c.F = reference(c, P);
  double beta = 0.0;
  bool ok = false;
  c.dsel = 0;
  if (nc == 1) {
    c.gd = gd;
    c.q = q;
    beta = backtrack(c.fZ, c.F, gd, q, P, &ok);
    if (P.controller == 3 && c.feat_ok) {  // lean learned step: the proposal, backtracked
      c.mlp_tried++;
      if (ok && beta == 1.0) c.mlp_accept++;
    }
  } else if (nc == 2) {
    // proposal: Armijo test at beta = 1 only
    const double fz1 = c.fZ + gd + 0.5 * q;
    c.mlp_tried++;
    if (fz1 <= c.F + P.theta * gd) {
      beta = 1.0;
      ok = true;
      c.mlp_accept++;
      c.gd = gd;
      c.q = q;
    } else {
      const double gd1 = qs[5], q1 = qs[7];
      c.dsel = 1;
      c.gd = gd1;
      c.q = q1;
      beta = backtrack(c.fZ, c.F, gd1, q1, P, &ok);
    }
  } else {
    // record mode: label = candidate with the best accepted decrease
    int best = 4;
    double best_dec = 0.0;
    double beta4 = 0.0;
    bool ok4 = false;
    for (int m = 0; m < nc; ++m) {
      const double gdm = m == 0 ? gd : qs[5 + 3 * (m - 1)];
      const double qm = m == 0 ? q : qs[5 + 3 * (m - 1) + 2];
      bool okm = false;
      const double bm = backtrack(c.fZ, c.F, gdm, qm, P, &okm);
      const double dec = okm ? bm * gdm + 0.5 * bm * bm * qm : 0.0;
      if (dec < best_dec) { best_dec = dec; best = m; }
      if (m == 4) { beta4 = bm; ok4 = okm; c.gd = gdm; c.q = qm; }
    }
    if (c.feat_ok && P.rec_feat) {
      const int idx = atomicAdd(P.rec_count, 1);
      if (idx < P.rec_cap) {
        for (int u = 0; u < kMlpIn; ++u) P.rec_feat[(int64_t)idx * kMlpIn + u] = c.feat[u];
        P.rec_targ[idx] = 0.5f * (float)(best - 4);  // log2 of the best multiplier
      }
    }
    beta = beta4;
    ok = ok4;
  }
  if (!ok) { beta = 0.0; c.ls_fail++; }
  if (!finite_bits(c.fZ) || !finite_bits(q) || !finite_bits(gd)) { c.nan_seen = 1; c.active = 0; }
  c.beta = beta;
  c.phibeta = P.phi * beta;
}

// After the relaxed update (q: 0 pg2, 2 ss, 3 sy, 4 yy, 5 f(X')-f(Z), 6 zero entries).
// One warp (the network): BB step of the next iteration and, with a controller, its candidates.
// Controller features (scale free): ln(BB1 rho), ln(BB2 rho), ||P grad|| ratio, objective
// decrease ratio, active-set fraction.
__device__ void pen_upd_body(Ctl& c, const double* qs, int j, const Params& P, int is_h_block, int last, int nc) {
  const double pg2 = qs[0], ss = qs[2], sy = qs[3], yy = qs[4], dwz = qs[5], zeros = qs[6];
  const double f_old = c.f;
  const double f_new = c.fZ + dwz;
  double alpha_bb;  // Alg. 1 line 3 / Eq. (2.10) with the 1/rho fallback when <S,Y> <= 0
  if (!(sy > 0.0)) alpha_bb = 1.0 / c.rho;
  else alpha_bb = (P.bb == 0) ? ss / sy : sy / yy;
  alpha_bb = fmin(P.alpha_max, fmax(P.alpha_min, alpha_bb));
  if (nc > 1) {
    // The features feed an FP32 network, so they are formed in FP32 from the FP64 sums (the
    // FP64 units of this GPU are slow, and this runs on one warp at the end of the launch).
    float phi[kMlpIn];
    const float rho = (float)c.rho;
    const float ssf = (float)ss, syf = (float)sy, yyf = (float)yy;
    const float bb1r = syf > 0.f ? ssf * rho / syf : 1.f;  // BB1 rho, BB2 rho (1 without curvature)
    const float bb2r = (syf > 0.f && yyf > 0.f) ? syf * rho / yyf : 1.f;
    const float pgf = sqrtf((float)pg2);
    const double dec = f_old - f_new;
    const float prev = (float)c.pg_prev;
    phi[0] = logf(fminf(fmaxf(bb1r, 1e-6f), 1e6f));
    phi[1] = logf(fminf(fmaxf(bb2r, 1e-6f), 1e6f));
    phi[2] = prev > 0.f ? fminf(pgf / prev, 10.f) : 1.f;
    phi[3] = fminf(fmaxf((float)dec / fmaxf(fabsf((float)c.last_dec), 1e-37f), -10.f), 10.f);
    phi[4] = (float)zeros / (float)P.nr;
    const double pg = (double)pgf;
    float mult = 1.f;
    // rollout branch (controller 4): this step's index counted over the whole solve
    const bool branch = P.controller == 4 &&
                        (int64_t)c.iters * 2 * P.inner + (int64_t)is_h_block * P.inner + c.k == P.branch_step;
    if ((nc == 2 || nc == 3) && P.controller != 4) mult = mlp_multiplier(P.mlp_w, phi);  // all lanes
    if ((threadIdx.x & 31) == 0) {
      for (int u = 0; u < kMlpIn; ++u) c.feat[u] = phi[u];
      c.feat_ok = 1;
      c.pg_prev = pg;
      c.last_dec = dec;
      if (nc == 2) {
        c.mlp_mult = mult;
        c.cand_alpha[0] = fmin(P.alpha_max, fmax(P.alpha_min, (double)mult * alpha_bb));
        c.cand_alpha[1] = alpha_bb;
      } else if (nc == 3 && P.controller == 4) {
        // rollout branch: candidate j % 9 scales the next step by 2^((c - 4) / 2); the group's
        // plain candidate records the features of the branch point, tagged with the group
        if (branch) {
          const int cand = j % kNCand;
          alpha_bb = fmin(P.alpha_max, fmax(P.alpha_min, exp2(0.5 * (cand - 4)) * alpha_bb));
          if (cand == 4 && P.rec_feat) {
            const int idx = atomicAdd(P.rec_count, 1);
            if (idx < P.rec_cap) {
              for (int u = 0; u < kMlpIn; ++u) P.rec_feat[(int64_t)idx * kMlpIn + u] = phi[u];
              P.rec_targ[idx] = (float)(j / kNCand);
            }
          }
        }
      } else if (nc == 3) {  // lean learned step: the next D uses the proposal directly
        c.mlp_mult = mult;
        alpha_bb = fmin(P.alpha_max, fmax(P.alpha_min, (double)mult * alpha_bb));
      } else {
        for (int m = 0; m < kNCand; ++m)
          c.cand_alpha[m] = fmin(P.alpha_max, fmax(P.alpha_min, exp2(0.5 * (m - 4)) * alpha_bb));
      }
    }
  }
  if ((threadIdx.x & 31) != 0) return;
  c.ss = ss; c.sy = sy; c.yy = yy;
  c.f = f_new;
  hist_push(c, c.f, P.memory);
  c.k++;
  c.alpha = alpha_bb;
  if (is_h_block) {
    c.pgH2 = pg2;
    if (last) c.iters++;
  } else if (last) {
    c.iters++;  // naive variant: the W block is the whole outer iteration
  }
  if (!finite_bits(c.f)) { c.nan_seen = 1; c.active = 0; }
}

// Final per-restart statistics of the penalty form: pax q0 = <W, A Ht>, prow q0 = ||P grad_W||^2
// at the final point; GW = W^T W, GH = Ht^T Ht, WH = W^T Ht of this restart.
__device__ void final_pen_body(Ctl& c, const double* pax, int nax, const double* prow, int nrow,
                               const double* GW, const double* GH, const double* WH, int b, int j,
                               int r, double normA2, double* sh) {
  const double wah = reduce_slots(pax, nax, b, j, 0, sh);
  const double pg2 = reduce_slots(prow, nrow, b, j, 0, sh);
  const double gwgh = dot_rr(GW, GH, r, sh);
  double trw = 0.0, trh = 0.0, trwh = 0.0;
  for (int p = threadIdx.x; p < r; p += blockDim.x) {
    trw += GW[p * r + p];
    trh += GH[p * r + p];
    trwh += WH[p * r + p];
  }
  trw = block_sum(trw, sh);
  trh = block_sum(trh, sh);
  trwh = block_sum(trwh, sh);
  if (threadIdx.x != 0) return;
  const double res2 = normA2 - 2.0 * wah + gwgh;
  c.fin_res = sqrt(fmax(res2, 0.0) / normA2);
  c.fin_f = 0.5 * res2 + 0.5 * c.lam * (trw - 2.0 * trwh + trh);
  c.fin_pg = (c.pg0 > 0.0) ? sqrt(pg2 + c.pgH2) / c.pg0 : 0.0;
}

// Fused control after a producing kernel, by one warp: modes of RowArgs::ctl_mode; qs: the summed
// partials, c: the restart's state (every lane passes; lane 0 writes).
__device__ __forceinline__ void fused_control(int mode, Ctl& c, const double* qs, int j, const Params& P, int nc) {
  if (!c.active) return;
  // candidates of the solve (3: the lean learned step, one candidate)
  const int pc = P.controller == 1 ? 2 : (P.controller == 2 ? kNCand : (P.controller >= 3 ? 3 : 1));
  const bool lead = (threadIdx.x & 31) == 0;
  switch (mode) {
    case CTL_START_W: if (lead) pen_start_body(c, qs, j, P, 1, 0); break;
    case CTL_START_H: if (lead) pen_start_body(c, qs, j, P, 0, 0); break;
    case CTL_START_INIT: if (lead) pen_start_body(c, qs, j, P, 0, 1); break;
    case CTL_LS: if (lead) pen_ls_body(c, qs, qs[4], P, nc); break;
    case CTL_UPD_W: pen_upd_body(c, qs, j, P, 0, 0, pc); break;
    case CTL_UPD_H: pen_upd_body(c, qs, j, P, 1, 0, pc); break;
    case CTL_UPD_H_LAST: pen_upd_body(c, qs, j, P, 1, 1, pc); break;
    case CTL_UPD_W_LAST_NAIVE: pen_upd_body(c, qs, j, P, 0, 1, pc); break;
    default: break;
  }
}

// The control step of restart j in the CTA that completed it: all threads sum the partial records
// [first, first + nslots) and copy the state to shared memory, one warp runs the scalar step there
// (its serial reads then cost a shared access each and not a trip to L2), and the state goes back.
template <int NV>
__device__ __forceinline__ void control_tail(const RowArgs& a, int j, int first, int nslots, int nc) {
  __shared__ double sh[8][NV], qs[NV];
  __shared__ __align__(16) uint64_t cbuf[sizeof(Ctl) / 8];
  static_assert(sizeof(Ctl) % 8 == 0, "copied in 8-byte words");
  uint64_t* g = reinterpret_cast<uint64_t*>(const_cast<Ctl*>(a.ctl + j));
  for (int e = threadIdx.x; e < (int)(sizeof(Ctl) / 8); e += blockDim.x) cbuf[e] = g[e];
  slot_sums<NV>(a.part + (int64_t)first * a.b * kNQ, nslots, a.b, j, sh, qs);
  if (threadIdx.x < 32) fused_control(a.ctl_mode, *reinterpret_cast<Ctl*>(cbuf), qs, j, a.P, nc);
  __syncthreads();
  for (int e = threadIdx.x; e < (int)(sizeof(Ctl) / 8); e += blockDim.x) g[e] = cbuf[e];
}

// ------------------------------------------------------------------------------
// Row GEMM with fused Algorithm-1 epilogues.
// ------------------------------------------------------------------------------
// CTA coordinates are arguments: restart j, row tile bx, column tile by of gy, `per` CTAs
// per restart (the partial slot of the CTA is bx * gy + by).
template <typename T, int OP, int EPI, int BM, int NC>
__device__ __forceinline__ void rowgemm_body(const RowArgs& a, int j, int bx, int by, int gy, unsigned per) {
  constexpr int MR = BM / 16;  // rows per thread
  constexpr int KC = sizeof(T) == 4 ? 64 : 32;  // K columns staged per round
  constexpr int XS_ELEMS = BM * (KC + 1);
  constexpr int DS_ELEMS = (EPI == EPI_DIR) ? BM * 65 : 1;
  constexpr int U_ELEMS = XS_ELEMS > DS_ELEMS ? XS_ELEMS : DS_ELEMS;
  constexpr int NV = NC > 1 ? 32 : 8;  // partial values written per CTA
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int64_t row0 = (int64_t)bx * BM;
  const int col0 = by * 64;  // within restart
  const int r = a.r;
  const int64_t ld = a.ld;
  const int64_t jc = (int64_t)j * r;
  __shared__ T shq[NV][8];
  __shared__ __align__(16) T ubuf[U_ELEMS];   // operand tile, later the D tile
  __shared__ T Gs[KC][64 + 1];
  T (*Xs)[KC + 1] = reinterpret_cast<T (*)[KC + 1]>(ubuf);
  T (*Ds)[65] = reinterpret_cast<T (*)[65]>(ubuf);
  const Ctl& cj = a.ctl[j];
  const bool live = cj.active && !(a.run && *a.run == 0);
  T dq[NV];
#pragma unroll
  for (int m = 0; m < NV; ++m) dq[m] = T(0);
  if (live) {
    const T* G = (const T*)a.G + (int64_t)j * r * r;
    const T inv_rho = (T)(1.0 / cj.rho);
    const T pb = (T)cj.phibeta;
    const T* X = (const T*)a.X;
    const T* gin = (const T*)a.g_in;
    const T* Zin = (const T*)a.Zin;
    const T* Din = (const T*)a.Din;
    T alph[NC];
#pragma unroll
    for (int m = 0; m < NC; ++m) alph[m] = (T)(NC == 1 ? cj.alpha : cj.cand_alpha[m]);
    auto operand = [&](int64_t i, int64_t col) -> T {
      const int64_t idx = i * ld + col;
      if (OP == OP_LOAD) return X[idx];
      if (OP == OP_ZSTEP) { T v = X[idx] - gin[idx] * inv_rho; return v > T(0) ? v : T(0); }
      T v = Zin[idx] + pb * Din[idx];
      return v > T(0) ? v : T(0);
    };
    T acc[MR][4];
#pragma unroll
    for (int p = 0; p < MR; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[p][q] = T(0);
    for (int k0 = 0; k0 < r; k0 += KC) {
      {
        // all loads of the round in flight before the shared-memory stores
        constexpr int NX = BM * KC / 256, NG = KC * 64 / 256;
        T xv_[NX], gv_[NG];
#pragma unroll
        for (int m = 0; m < NX; ++m) {
          const int e = threadIdx.x + 256 * m;
          const int rr = e / KC, kk = e % KC;
          const int64_t i = row0 + rr;
          xv_[m] = (i < a.n && k0 + kk < r) ? operand(i, jc + k0 + kk) : T(0);
        }
#pragma unroll
        for (int m = 0; m < NG; ++m) {
          const int e = threadIdx.x + 256 * m;
          const int gk = e >> 6, gc = e & 63;
          gv_[m] = (k0 + gk < r && col0 + gc < r) ? G[(int64_t)(k0 + gk) * r + col0 + gc] : T(0);
        }
#pragma unroll
        for (int m = 0; m < NX; ++m) {
          const int e = threadIdx.x + 256 * m;
          Xs[e / KC][e % KC] = xv_[m];
        }
#pragma unroll
        for (int m = 0; m < NG; ++m) {
          const int e = threadIdx.x + 256 * m;
          Gs[e >> 6][e & 63] = gv_[m];
        }
      }
      __syncthreads();
      const int kn = min(KC, r - k0);
#pragma unroll 8
      for (int kk = 0; kk < kn; ++kk) {
        T xa[MR], gb[4];
#pragma unroll
        for (int p = 0; p < MR; ++p) xa[p] = Xs[ty + 16 * p][kk];
#pragma unroll
        for (int q = 0; q < 4; ++q) gb[q] = Gs[kk][tx + 16 * q];
#pragma unroll
        for (int p = 0; p < MR; ++p)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[p][q] = fma(xa[p], gb[q], acc[p][q]);
      }
      __syncthreads();
    }
    // epilogue
    const T* B = (const T*)a.B;
    const T* LX = (const T*)a.LX;
    const T gam = (T)a.gamma;
    T gl[MR][4], xl[MR][4];  // gradient and operand of the thread's elements
    // With r <= KC the operand tile of this CTA's rows is still in shared memory.
    const bool xs_ok = r <= KC && col0 == 0;
#pragma unroll
    for (int p = 0; p < MR; ++p) {
      const int64_t i = row0 + ty + 16 * p;
      // the row's loads first: the stores below may alias inputs (Xout / Xold), so
      // keeping them apart lets all four elements' loads be in flight together
      bool vq[4];
      int64_t iq[4];
      T xq[4], bq[4], lq[4], o0[4], o1[4], o2[4], o3[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int c = col0 + tx + 16 * q;
        vq[q] = i < a.n && c < r;
        iq[q] = i * ld + jc + c;
        xq[q] = bq[q] = lq[q] = o0[q] = o1[q] = o2[q] = o3[q] = T(0);
        if (!vq[q]) continue;
        const int64_t idx = iq[q];
        xq[q] = xs_ok ? Xs[ty + 16 * p][c] : operand(i, jc + c);
        bq[q] = B[idx];
        if (LX) lq[q] = LX[idx];
        if (EPI == EPI_GRAD) {
          if (a.Xold) { o0[q] = ((const T*)a.Xold)[idx]; o1[q] = ((const T*)a.gold)[idx]; }
          if (a.Zold) { o2[q] = ((const T*)a.Zold)[idx]; o3[q] = ((const T*)a.gZold)[idx]; }
        } else if (a.Wcur) {
          o0[q] = ((const T*)a.Wcur)[idx];
          o1[q] = ((const T*)a.gWcur)[idx];
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        gl[p][q] = T(0);
        xl[p][q] = T(0);
        if (!vq[q]) continue;
        const int64_t idx = iq[q];
        const T xv = xq[q];
        T g = acc[p][q] - bq[q];
        if (LX) g += gam * lq[q];
        gl[p][q] = g;
        xl[p][q] = xv;
        if (EPI == EPI_GRAD) {
          const T pgv = xv > T(0) ? g : (g < T(0) ? g : T(0));
          dq[0] += pgv * pgv;                              // ||P grad||^2
          dq[1] += T(0.5) * (g - bq[q]) * xv;               // f - const (quadratic block)
          if (a.Xold) {
            const T sv = xv - o0[q];
            const T yv = g - o1[q];
            dq[2] += sv * sv;
            dq[3] += sv * yv;
            dq[4] += yv * yv;
          }
          if (a.Zold) dq[5] += T(0.5) * (xv - o2[q]) * (g + o3[q]);  // f(X') - f(Z), trapezoid (exact)
          if (xv == T(0)) dq[6] += T(1);                    // active (zero) entries
          if (a.gout) ((T*)a.gout)[idx] = g;
          if (a.Xout) ((T*)a.Xout)[idx] = xv;
        } else {  // EPI_DIR
          if (a.Xout) ((T*)a.Xout)[idx] = xv;
          if (a.gZout) ((T*)a.gZout)[idx] = g;
          if (a.Wcur) dq[2] += T(0.5) * (xv - o0[q]) * (g + o1[q]);  // f(Z) - f(W), trapezoid (exact)
#pragma unroll
          for (int m = 0; m < NC; ++m) {
            T d = xv - alph[m] * g;
            d = (d > T(0) ? d : T(0)) - xv;
            if (m == a.dstore) ((T*)a.Dout)[idx] = d;
            const int base = m == 0 ? 0 : 5 + 3 * (m - 1);
            dq[base] += g * d;                              // <grad f(Z), D_m>
            dq[base + 1] += d * d;                          // ||D_m||^2
            if (m == 0 && LX) dq[3] += d * lq[q];           // <D, L Z> (direct, graph)
          }
        }
      }
    }
    __syncthreads();  // the operand tile (read above) and the D tile below share memory
    if (EPI == EPI_DIR && a.want_q) {
      // <D_m G, D_m> of each candidate's line-search quadratic (restart = one column tile)
#pragma unroll 1
      for (int m = 0; m < NC; ++m) {
#pragma unroll
        for (int p = 0; p < MR; ++p)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            T d = xl[p][q] - alph[m] * gl[p][q];
            d = (d > T(0) ? d : T(0)) - xl[p][q];
            const int c = col0 + tx + 16 * q;
            const int64_t i = row0 + ty + 16 * p;
            Ds[ty + 16 * p][tx + 16 * q] = (i < a.n && c < r) ? d : T(0);
          }
        __syncthreads();
        T acc2[MR][4];
#pragma unroll
        for (int p = 0; p < MR; ++p)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc2[p][q] = T(0);
        for (int k0 = 0; k0 < r; k0 += KC) {
          if (!xs_ok) {  // else G (r <= KC) is still in shared memory from the first product
            constexpr int NG = KC * 64 / 256;
            T gv_[NG];
#pragma unroll
            for (int u = 0; u < NG; ++u) {
              const int e = threadIdx.x + 256 * u;
              const int gk = e >> 6, gc = e & 63;
              gv_[u] = (k0 + gk < r && gc < r) ? G[(int64_t)(k0 + gk) * r + gc] : T(0);
            }
#pragma unroll
            for (int u = 0; u < NG; ++u) {
              const int e = threadIdx.x + 256 * u;
              Gs[e >> 6][e & 63] = gv_[u];
            }
          }
          __syncthreads();
          const int kn = min(KC, r - k0);
#pragma unroll 8
          for (int kk = 0; kk < kn; ++kk) {
            T gb[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) gb[q] = Gs[kk][tx + 16 * q];
#pragma unroll
            for (int p = 0; p < MR; ++p) {
              const T dv = Ds[ty + 16 * p][k0 + kk];
#pragma unroll
              for (int q = 0; q < 4; ++q) acc2[p][q] = fma(dv, gb[q], acc2[p][q]);
            }
          }
          __syncthreads();
        }
        T qq = T(0);
#pragma unroll
        for (int p = 0; p < MR; ++p)
#pragma unroll
          for (int q = 0; q < 4; ++q) qq += acc2[p][q] * Ds[ty + 16 * p][tx + 16 * q];
        dq[m == 0 ? 4 : 5 + 3 * (m - 1) + 2] += qq;
        __syncthreads();
      }
    }
  }
  // one combined fixed-order reduction of the partial dots
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int m = 0; m < NV; ++m) {
    const T v = warp_sum(dq[m]);
    if (lane == 0) shq[m][wid] = v;
  }
  __syncthreads();
  if (threadIdx.x < NV) {
    T v = T(0);
#pragma unroll
    for (int w = 0; w < 8; ++w) v += shq[threadIdx.x][w];
    const int slot = bx * gy + by;
    a.part[((int64_t)slot * a.b + j) * kNQ + threadIdx.x] = (double)v;
  }
  if (a.ctl_mode) {
    // the last CTA of restart j runs its control step (all partials of j are written)
    __shared__ unsigned ticket;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) ticket = atomicAdd(&a.counters[j], 1u);
    __syncthreads();
    if (ticket == per - 1) {
      if (threadIdx.x == 0) a.counters[j] = 0u;
      control_tail<NV>(a, j, 0, (int)per, NC);
    }
  }
}

}  // namespace

}  // namespace snmf
