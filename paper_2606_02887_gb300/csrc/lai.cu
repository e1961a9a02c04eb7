// LAI-SNMPBB (Sec. 2.3, Eq. (8)): randomized eigen-sketch A ~ U E U^T and the product
// A X ~ U (E (U^T X)), U^T X formed first.
//
//   k_utx      M = E (U^T X) (k x N): CTA (row chunk, 64 x 16, 32 or 64 output tile), partials summed
//              as the Gram's (gram_dev.cuh), row l scaled by lambda_l.
//   k_rowmul   Out = In M (n x K times K x m) (+ c X2), K <= 128, in the product tiles of
//              gemm_dev.cuh.  Serves U M, Y R^-1 (CholeskyQR) and Q P (Ritz vectors).
//   k_chol     Cholesky R^T R = G (+ shift) of an l x l FP64 Gram and R^-1, one block.
//   k_jacobi   parallel cyclic Jacobi eigensolver of a symmetric l x l FP64 matrix, one block,
//              round-robin pairing (l/2 disjoint rotations per round).
//   k_select   indices of the k eigenvalues of largest magnitude, eigenvector block P_k.
#include <math.h>

#include <algorithm>
#include <string>

#include "ax_tc.cuh"
#include "gemm_dev.cuh"
#include "lai.cuh"
#include "rowops.cuh"

namespace snmf {

namespace {

inline int cdivi(int64_t a, int64_t b) { return (int)((a + b - 1) / b); }

// Bound by HBM (U and X read once): n = 2e6, k = 64, N = 32 took 757 us with two staged rounds and
// scalar shared reads in 152 CTAs.
template <typename T, int TQ, int VEC>
__global__ void __launch_bounds__(256, 3)
k_utx(const T* __restrict__ U, int k, const T* __restrict__ X, int64_t n, int N, int64_t ldx, int64_t chunk, int nch,
      int ng, T* __restrict__ part, const double* __restrict__ lam, T* __restrict__ M, unsigned* __restrict__ counters,
      const int* run) {
  extern __shared__ __align__(16) unsigned char usm[];
  if (run && *run == 0) return;
  constexpr int TT = 64 * TQ, NE = tile_quads<64, TQ>();
  const int l0 = blockIdx.y * 64, c0 = blockIdx.z * TQ, tile = blockIdx.y * gridDim.z + blockIdx.z;
  const int64_t i0 = (int64_t)blockIdx.x * chunk;
  Quad<T> s[NE];
  gram_chunk<T, 64, TQ, VEC>(U + l0, X + c0, min(64, k - l0), min(TQ, N - c0), k, ldx, i0, min(n, i0 + chunk), false,
                             reinterpret_cast<T*>(usm), s);
  if (!sum_chunks<T, TT>(s, blockIdx.x, nch, ng, part + (int64_t)tile * (nch + ng) * TT, counters + tile * (1 + ng)))
    return;
#pragma unroll
  for (int u = 0; u < NE; ++u) {
    const int e = 4 * (threadIdx.x + 256 * u);
    if (e >= TT) continue;
    const int l = l0 + e / TQ;
    if (l >= k) continue;
    const T sc = (T)lam[l];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (c0 + e % TQ + q < N) M[(int64_t)l * N + c0 + e % TQ + q] = s[u].v[q] * sc;
  }
}

template <typename T>
constexpr size_t utx_smem(int tq) {
  const size_t ring = (size_t)kGramStages * (kGramStageBytes + kGramStageBytes / 64 * tq);
  return ring > 4096 * sizeof(T) ? ring : 4096 * sizeof(T);
}

// n = 2e6, K = 64, m = 32: 445 us in 64 x 32 tiles staged one round at a time, and a finish pass.
template <typename C, int PER_SM>
__global__ void __launch_bounds__(C::NT, PER_SM)
k_rowmul(const typename C::T* __restrict__ In, int64_t ldi, int K, const typename C::T* __restrict__ Mm, int m, int64_t n,
         typename C::T* __restrict__ Out, int64_t ldo, bool avec, bool xvec, bool yvec, typename C::T c,
         const typename C::T* __restrict__ X2, const int* run) {
  using T = typename C::T;
  extern __shared__ __align__(16) unsigned char rsm[];
  if (run && *run == 0) return;
  const int64_t row0 = (int64_t)blockIdx.x * C::BM;
  const int col0 = blockIdx.y * C::BN;
  T acc[C::TM][C::TN];
  gemm_tile<C>(In, ldi, Mm, m, n, m, row0, col0, 0, K, avec, xvec, GemmA8{}, reinterpret_cast<T*>(rsm), acc);
  const int tx = threadIdx.x % C::TX, ty = threadIdx.x / C::TX;
#pragma unroll
  for (int i = 0; i < C::TM; ++i) {
    const int64_t r = row0 + ty + C::TY * i;
    if (r >= n) continue;
#pragma unroll
    for (int j = 0; j < C::TN; j += C::VW) {
      struct alignas(C::VW * sizeof(T)) Vec {
        T v[C::VW];
      };
      const int col = col0 + C::col(tx, j);
      const int64_t idx = r * ldo + col;
      if (yvec) {
        if (col >= m) continue;
        Vec y, x2;
        if (X2) x2 = *reinterpret_cast<const Vec*>(X2 + idx);
#pragma unroll
        for (int u = 0; u < C::VW; ++u) y.v[u] = X2 ? acc[i][j + u] + c * x2.v[u] : acc[i][j + u];
        *reinterpret_cast<Vec*>(Out + idx) = y;
      } else {
#pragma unroll
        for (int u = 0; u < C::VW; ++u)
          if (col + u < m) Out[idx + u] = X2 ? acc[i][j + u] + c * X2[idx + u] : acc[i][j + u];
      }
    }
  }
}

// The same in FP32 for long inputs whose rows, M and Out allow 16-byte accesses, all m <= BN columns in
// one tile: a CTA walks tiles of BM rows with M resident and a ring of three stages of BK columns of
// In that runs on over the tiles, X2 on its way during the last stage.  FMAs in the order of k_rowmul.
// Bound by HBM and, close behind, by the FMA pipes: n = 2e6, K = 64, m = 32 285 -> 217 us (1.0 GB).
template <typename C, int PER_SM>
__global__ void __launch_bounds__(C::NT, PER_SM)
k_rowmul_walk(const float* __restrict__ In, int64_t ldi, int K, const float* __restrict__ Mm, int m, int64_t n, int tiles,
              float* __restrict__ Out, int64_t ldo, float c, const float* __restrict__ X2, const int* run) {
  extern __shared__ __align__(16) unsigned char rsm[];
  if (run && *run == 0) return;
  constexpr int BM = C::BM, BN = C::BN, BK = C::BK, AS = C::AS, ST = 3, STAGE = BM * AS;
  const int t = threadIdx.x, tx = t % C::TX, ty = t / C::TX;
  const int nk = (K + BK - 1) / BK;
  float* ring = reinterpret_cast<float*>(rsm);
  float* Ms = ring + ST * STAGE;
  for (int e = t; e < nk * BK * BN; e += C::NT) {
    const int k = e / BN, q = e % BN;
    Ms[e] = k < K && q < m ? Mm[(int64_t)k * m + q] : 0.f;
  }
  const int mine = (tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x, steps = mine * nk;
  auto fetch = [&](int s) {
    if (s < steps) {
      const int64_t row0 = ((int64_t)blockIdx.x + (int64_t)(s / nk) * gridDim.x) * BM;
      const int k0 = s % nk * BK;
      float* as = ring + s % ST * STAGE;
      constexpr int NA = BM * BK / 4;
#pragma unroll
      for (int u = 0; u < NA / C::NT; ++u) {
        const int e = t + C::NT * u, r = e / (BK / 4), k = k0 + e % (BK / 4) * 4;
        const bool v = row0 + r < n && k < K;
        cp_async<16>(as + r * AS + (k - k0), v ? In + (row0 + r) * ldi + k : In, v);
      }
    }
    cp_async_commit();
  };
#pragma unroll
  for (int s = 0; s < ST - 1; ++s) fetch(s);
  float acc[C::TM][C::TN];
  for (int s = 0; s < steps; ++s) {
    const int kc = s % nk;
    const int64_t row0 = ((int64_t)blockIdx.x + (int64_t)(s / nk) * gridDim.x) * BM;
    cp_async_wait<ST - 2>();
    __syncthreads();  // stage s is in (and M); every thread is done with the stage refilled below
    fetch(s + ST - 1);
    if (kc == 0) {
#pragma unroll
      for (int i = 0; i < C::TM; ++i)
#pragma unroll
        for (int j = 0; j < C::TN; ++j) acc[i][j] = 0.f;
    }
    float4 x2[C::TM][C::TN / 4];
    if (X2 && kc == nk - 1) {
#pragma unroll
      for (int i = 0; i < C::TM; ++i)
#pragma unroll
        for (int j = 0; j < C::TN / 4; ++j) {
          const int64_t r = row0 + ty + C::TY * i;
          const int col = C::col(tx, 4 * j);
          x2[i][j] = r < n && col < m ? *reinterpret_cast<const float4*>(X2 + r * ldo + col) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    const float* as = ring + s % ST * STAGE;
    const float* xs = Ms + kc * BK * BN;
#pragma unroll
    for (int kk = 0; kk < BK; kk += 4) {
      float a[C::TM][4];
#pragma unroll
      for (int i = 0; i < C::TM; ++i) {
        const float4 v = *reinterpret_cast<const float4*>(as + (ty + C::TY * i) * AS + kk);
        a[i][0] = v.x; a[i][1] = v.y; a[i][2] = v.z; a[i][3] = v.w;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float x[C::TN];
#pragma unroll
        for (int j = 0; j < C::TN; j += 4) {
          const float4 v = *reinterpret_cast<const float4*>(xs + (kk + u) * BN + C::col(tx, j));
          x[j] = v.x; x[j + 1] = v.y; x[j + 2] = v.z; x[j + 3] = v.w;
        }
        fma_row<C>(a, u, x, acc);
      }
    }
    if (kc != nk - 1) continue;
#pragma unroll
    for (int i = 0; i < C::TM; ++i) {
      const int64_t r = row0 + ty + C::TY * i;
      if (r >= n) continue;
#pragma unroll
      for (int j = 0; j < C::TN / 4; ++j) {
        const int col = C::col(tx, 4 * j);
        if (col >= m) continue;
        float4 y = make_float4(acc[i][4 * j], acc[i][4 * j + 1], acc[i][4 * j + 2], acc[i][4 * j + 3]);
        if (X2) {
          y.x = y.x + c * x2[i][j].x;
          y.y = y.y + c * x2[i][j].y;
          y.z = y.z + c * x2[i][j].z;
          y.w = y.w + c * x2[i][j].w;
        }
        *reinterpret_cast<float4*>(Out + r * ldo + col) = y;
      }
    }
  }
  cp_async_wait<0>();
}

// Cholesky of G + shift I (l x l FP64, row-major, overwritten by R, upper) and Rinv (FP64,
// then copied to the working type).  *fail = 1 on a non-positive pivot.
template <typename T>
__global__ void k_chol(double* __restrict__ G, int l, double shift_rel, double* __restrict__ Rinv,
                       T* __restrict__ RinvT, int* __restrict__ fail) {
  __shared__ double piv;
  __shared__ double tr;
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < l; ++i) t += G[i * l + i];
    tr = t;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < l; e += blockDim.x) G[e * l + e] += shift_rel * tr;
  __syncthreads();
  for (int j = 0; j < l; ++j) {
    if (threadIdx.x == 0) {
      const double d = G[j * l + j];
      piv = d > 0.0 ? sqrt(d) : -1.0;
      if (!(d > 0.0)) *fail = 1;
    }
    __syncthreads();
    if (piv <= 0.0) return;
    for (int c = j + threadIdx.x; c < l; c += blockDim.x) G[j * l + c] = (c == j) ? piv : G[j * l + c] / piv;
    __syncthreads();
    // trailing update G[a][c] -= R[j][a] R[j][c]  (a, c > j, upper triangle)
    const int m = l - j - 1;
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
      const int a = j + 1 + e / m, c = j + 1 + e % m;
      if (c >= a) G[a * l + c] -= G[j * l + a] * G[j * l + c];
    }
    __syncthreads();
  }
  // zero the strict lower triangle (R upper)
  for (int e = threadIdx.x; e < l * l; e += blockDim.x)
    if (e / l > e % l) G[e] = 0.0;
  __syncthreads();
  // Rinv: column c solves R x = e_c (back substitution), one thread per column
  for (int c = threadIdx.x; c < l; c += blockDim.x) {
    for (int i = l - 1; i >= 0; --i) {
      double s = (i == c) ? 1.0 : 0.0;
      for (int t = i + 1; t <= c; ++t) s -= G[i * l + t] * Rinv[t * l + c];
      Rinv[i * l + c] = (i <= c) ? s / G[i * l + i] : 0.0;
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < l * l; e += blockDim.x) RinvT[e] = (T)Rinv[e];
}

// Parallel cyclic Jacobi: A (l x l FP64, symmetric, overwritten) -> eigenvalues on the
// diagonal, V (l x l FP64) eigenvectors in columns.  Round-robin pairing over m = even(l)
// indices (index l is a dummy when l is odd).  Stops when the off-diagonal norm is below
// tol times the Frobenius norm, or after max_sweeps.
__global__ void k_jacobi(double* __restrict__ A, double* __restrict__ V, int l, int max_sweeps, double tol) {
  extern __shared__ double cs[];  // [m/2] c, [m/2] s, [m/2] p, [m/2] q (as doubles)
  __shared__ double red[32];
  const int m = (l + 1) / 2 * 2, h = m / 2;
  double* C = cs;
  double* Sn = cs + h;
  int* Pp = reinterpret_cast<int*>(cs + 2 * h);
  int* Qq = Pp + h;
  for (int e = threadIdx.x; e < l * l; e += blockDim.x) V[e] = (e / l == e % l) ? 1.0 : 0.0;
  __syncthreads();
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    double off = 0.0, tot = 0.0;
    for (int e = threadIdx.x; e < l * l; e += blockDim.x) {
      const double v = A[e];
      tot += v * v;
      if (e / l != e % l) off += v * v;
    }
    off = block_sum(off, red);
    tot = block_sum(tot, red);
    if (off <= tol * tol * tot) break;
    for (int round = 0; round < m - 1; ++round) {
      for (int i = threadIdx.x; i < h; i += blockDim.x) {
        auto player = [&](int j) { return j == 0 ? 0 : ((j - 1 + round) % (m - 1)) + 1; };
        int p = player(i), q = player(m - 1 - i);
        if (p > q) { const int t = p; p = q; q = t; }
        double c = 1.0, s = 0.0;
        if (q < l) {
          const double apq = A[p * l + q];
          if (apq != 0.0) {
            const double tau = (A[q * l + q] - A[p * l + p]) / (2.0 * apq);
            const double t = (tau >= 0.0) ? 1.0 / (tau + sqrt(1.0 + tau * tau)) : -1.0 / (-tau + sqrt(1.0 + tau * tau));
            c = 1.0 / sqrt(1.0 + t * t);
            s = t * c;
          }
        }
        C[i] = c; Sn[i] = s; Pp[i] = p; Qq[i] = q;
      }
      __syncthreads();
      // columns: A <- A J, V <- V J
      for (int e = threadIdx.x; e < h * l; e += blockDim.x) {
        const int i = e / l, row = e % l;
        const int p = Pp[i], q = Qq[i];
        if (q >= l) continue;
        const double c = C[i], s = Sn[i];
        const double ap = A[row * l + p], aq = A[row * l + q];
        A[row * l + p] = c * ap - s * aq;
        A[row * l + q] = s * ap + c * aq;
        const double vp = V[row * l + p], vq = V[row * l + q];
        V[row * l + p] = c * vp - s * vq;
        V[row * l + q] = s * vp + c * vq;
      }
      __syncthreads();
      // rows: A <- J^T A
      for (int e = threadIdx.x; e < h * l; e += blockDim.x) {
        const int i = e / l, col = e % l;
        const int p = Pp[i], q = Qq[i];
        if (q >= l) continue;
        const double c = C[i], s = Sn[i];
        const double ap = A[p * l + col], aq = A[q * l + col];
        A[p * l + col] = c * ap - s * aq;
        A[q * l + col] = s * ap + c * aq;
      }
      __syncthreads();
    }
  }
}

// pick the k eigenvalues of largest |value| (ties: lower index first), write lam[k] and the
// l x k eigenvector block P (working type, row-major)
template <typename T>
__global__ void k_select(const double* __restrict__ A, const double* __restrict__ V, int l, int k,
                         double* __restrict__ lam, T* __restrict__ P, double* __restrict__ sumsq) {
  __shared__ int idx[128];
  if (threadIdx.x == 0) {
    bool used[128];
    for (int i = 0; i < l; ++i) used[i] = false;
    double s2 = 0.0;
    for (int t = 0; t < k; ++t) {
      int best = -1;
      double bv = -1.0;
      for (int i = 0; i < l; ++i)
        if (!used[i] && fabs(A[i * l + i]) > bv) { bv = fabs(A[i * l + i]); best = i; }
      used[best] = true;
      idx[t] = best;
      lam[t] = A[best * l + best];
      s2 += lam[t] * lam[t];
    }
    *sumsq = s2;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < l * k; e += blockDim.x) {
    const int row = e / k, t = e % k;
    P[e] = (T)V[row * l + idx[t]];
  }
}

template <typename T>
__global__ void k_sym(double* __restrict__ A, int l) {
  for (int e = threadIdx.x; e < l * l; e += blockDim.x) {
    const int p = e / l, q = e % l;
    if (p < q) {
      const double v = 0.5 * (A[p * l + q] + A[q * l + p]);
      A[p * l + q] = v;
      A[q * l + p] = v;
    }
  }
}

int ck(cudaError_t e, std::string& msg, const char* what) {
  if (e == cudaSuccess) return 0;
  msg = std::string(what) + ": " + cudaGetErrorString(e);
  return e == cudaErrorMemoryAllocation ? -3 : -2;
}

}  // namespace

namespace {

template <typename C, int PER_SM>
void launch_rowmul_cfg(const void* In, int64_t ldi, int K, const void* M, int m, int64_t n, void* Out, int64_t ldo,
                       const int* run, cudaStream_t s, double c, const void* X2) {
  using T = typename C::T;
  constexpr int64_t KV = C::KV, VW = C::VW;
  const bool avec = ldi % KV == 0 && K % KV == 0 && !((uintptr_t)In & 15);
  const bool xvec = m % KV == 0 && !((uintptr_t)M & 15);
  const bool yvec = ldo % VW == 0 && m % VW == 0 && !(((uintptr_t)Out | (uintptr_t)X2) & 15);
  // long inputs walk: more than two tiles for each of three CTAs per SM (n = 2e6, K = 64, m = 32 285 us
  // with a CTA per tile)
  if constexpr (sizeof(T) == 4 && C::BK == 32) {
    constexpr int kPerSm = 3;
    const int64_t tiles = cdivi(n, C::BM);
    if (avec && yvec && m <= C::BN && tiles > 2 * 152 * kPerSm) {
      const size_t smem = (3 * C::BM * C::AS + (size_t)cdivi(K, C::BK) * C::BK * C::BN) * sizeof(float);
      static SmemLimit walk;
      raise_smem_limit(walk, (const void*)k_rowmul_walk<C, kPerSm>, (3 * C::BM * C::AS + 128 * C::BN) * sizeof(float));
      k_rowmul_walk<C, kPerSm><<<152 * kPerSm, C::NT, smem, s>>>((const float*)In, ldi, K, (const float*)M, m, n, (int)tiles,
                                                                (float*)Out, ldo, (float)c, (const float*)X2, run);
      return;
    }
  }
  static SmemLimit limit;
  raise_smem_limit(limit, (const void*)k_rowmul<C, PER_SM>, C::SMEM);
  dim3 grid(cdivi(n, C::BM), cdivi(m, C::BN));
  k_rowmul<C, PER_SM><<<grid, C::NT, C::SMEM, s>>>((const T*)In, ldi, K, (const T*)M, m, n, (T*)Out, ldo, avec, xvec,
                                                   yvec, (T)c, (const T*)X2, run);
}

}  // namespace

void launch_rowmul(int tdtype, const void* In, int64_t ldi, int K, const void* M, int m, int64_t n, void* Out,
                   int64_t ldo, const int* run, cudaStream_t s, double c, const void* X2) {
  // tiles as wide as the output needs (the product's rule, see launch_ax)
#define ROWMUL(T, BM, BN, TM, TN, BK, OCC) \
  return launch_rowmul_cfg<GemmCfg<T, GA_SAME, BM, BN, TM, TN, BK>, OCC>(In, ldi, K, M, m, n, Out, ldo, run, s, c, X2)
  if (tdtype == 0) {
    if (m <= 16) ROWMUL(double, 64, 16, 4, 4, 16, 6);
    if (m <= 32) ROWMUL(double, 64, 32, 4, 4, 16, 4);
    ROWMUL(double, 64, 64, 4, 4, 16, 2);
  }
  if (m <= 16) ROWMUL(float, 128, 16, 4, 4, 32, 3);
  if (m <= 32) ROWMUL(float, 128, 32, 8, 4, 32, 3);
  ROWMUL(float, 128, 64, 8, 8, 32, 3);
#undef ROWMUL
}

namespace {

// Columns per k_utx tile (its chunks of rows: one wave of three CTAs per SM, of at least 256 rows).
int utx_tq(int N) { return N <= 16 ? 16 : (N <= 32 ? 32 : 64); }

template <typename T, int TQ, int VEC>
void launch_utx(const LaiOp& op, const void* X, int64_t n, int N, int64_t ldx, const int* run, cudaStream_t s) {
  static SmemLimit limit;
  raise_smem_limit(limit, (const void*)k_utx<T, TQ, VEC>, utx_smem<T>(TQ));
  dim3 grid(op.nch, cdivi(op.k, 64), cdivi(N, TQ));
  k_utx<T, TQ, VEC><<<grid, 256, utx_smem<T>(TQ), s>>>((const T*)op.U, op.k, (const T*)X, n, N, ldx, op.chunk, op.nch,
                                                       op.ng, (T*)op.xpart, op.lam, (T*)op.M, op.counters, run);
}

}  // namespace

int lai_apply(const LaiOp& op, int tdtype, const Dims& d, const void* X, void* Y, double c, const void* X2,
              const void* P1, const void* P2, double* part, const int* run, cudaStream_t s) {
  const int N = d.N, v = tdtype == 0 ? 2 : 4;
  const bool vec = op.k % v == 0 && N % v == 0 && d.ld % v == 0 && !((uintptr_t)X & 15);
#define UTX(T, TQ, V) launch_utx<T, TQ, V>(op, X, d.n, N, d.ld, run, s)
#define UTX_T(T, V)                                           \
  if (utx_tq(N) == 16) { if (vec) UTX(T, 16, V); else UTX(T, 16, 1); } \
  else if (utx_tq(N) == 32) { if (vec) UTX(T, 32, V); else UTX(T, 32, 1); } \
  else { if (vec) UTX(T, 64, V); else UTX(T, 64, 1); }
  if (tdtype == 0) { UTX_T(double, 2) } else { UTX_T(float, 4) }
#undef UTX_T
#undef UTX
  // the dots are of the product before c X2: with them the finish pass adds it
  const bool dots = P1 || P2;
  launch_rowmul(tdtype, op.U, op.k, op.k, op.M, N, d.n, Y, d.ld, run, s, c, dots ? nullptr : X2);
  if (!dots) return cdivi(d.n, kRowTile);
  return launch_ax_finish_impl(tdtype, d, Y, nullptr, 1, c, X2, P1, P2, part, 0, run, s);
}

// product of the input operator with an n x cols block (ld = cols), for the sketch
static int sketch_product(const AxArgs& A, int td, int64_t n, int cols, const void* X, void* Y, void* ws,
                          size_t ws_elems, void* xh, void* xl, int* err, cudaStream_t s) {
  Dims d;
  d.n = n; d.r = cols; d.b = 1; d.N = cols; d.ld = cols;
  int splits;
  if (A.kind == AX_DENSE && A.a_dtype == 2) {
    splits = launch_ax_tc(A.A, n, (const float*)X, cols, cols, xh, xl, (float*)Y, (float*)ws, ws_elems, err,
                          2000000000LL, s, nullptr, 2, A.sym);
    if (splits < 1) return -1;
  } else {
    // A dense product's sums in one order whatever its tiles are (as gram_plan_sketch): K in powers of two
    // until 64 x 64 tiles would be two CTAs per SM, at least 256 columns each, or in one piece without the room.
    ProdTune order;
    const int64_t tiles = (int64_t)cdivi(cols, 64) * cdivi(n, 64);
    int64_t sp = 1;
    while (tiles * sp < 2 * 152 && n / (2 * sp) >= 256) sp *= 2;
    if ((size_t)sp * (size_t)n * (size_t)cols > ws_elems) sp = 1;
    order.splits = (int)sp;
    order.kchunk = ((n + sp - 1) / sp + 15) / 16 * 16;
    splits = launch_ax(A, td, n, cols, cols, X, Y, ws, ws_elems, nullptr, s, A.kind == AX_DENSE ? &order : nullptr);
  }
  return splits;
}

int lai_build(LaiOp& op, const AxArgs& A, int td, int64_t n, int k, int ell, int power_iters, uint64_t seed,
              int maxN, cudaStream_t s, std::string& msg) {
  lai_free(op);
  const size_t esz = td == 0 ? 8 : 4;
  const size_t blk = (size_t)n * ell;
  void *Y = nullptr, *Q = nullptr, *ws = nullptr, *xh = nullptr, *xl = nullptr, *RinvT = nullptr, *Pk = nullptr;
  double *G = nullptr, *Rinv = nullptr, *V = nullptr, *part = nullptr, *sums = nullptr;
  void* gpart = nullptr;
  unsigned* counters = nullptr;
  int *fail = nullptr, *err = nullptr;
  int rc = 0;
  auto cleanup = [&]() {
    cudaFree(Y); cudaFree(Q); cudaFree(ws); cudaFree(xh); cudaFree(xl); cudaFree(RinvT); cudaFree(Pk);
    cudaFree(G); cudaFree(Rinv); cudaFree(V); cudaFree(gpart); cudaFree(part); cudaFree(sums);
    cudaFree(counters); cudaFree(fail); cudaFree(err);
  };
#define LCK(call)                                   \
  do {                                              \
    rc = ck((call), msg, #call);                    \
    if (rc) { cleanup(); return rc; }               \
  } while (0)
  const size_t ws_elems = (A.kind == AX_DENSE) ? 4 * blk : 0;
  LCK(cudaMalloc(&Y, blk * esz));
  LCK(cudaMalloc(&Q, blk * esz));
  if (ws_elems) LCK(cudaMalloc(&ws, ws_elems * esz));
  if (A.kind == AX_DENSE && A.a_dtype == 2) {
    LCK(cudaMalloc(&xh, (size_t)ell * tc_ld(n) * 2));
    LCK(cudaMalloc(&xl, (size_t)ell * tc_ld(n) * 2));
  }
  const GramPlan gp = gram_plan_sketch(n, ell);
  LCK(cudaMalloc(&G, (size_t)ell * ell * sizeof(double)));
  LCK(cudaMalloc(&Rinv, (size_t)ell * ell * sizeof(double)));
  LCK(cudaMalloc(&V, (size_t)ell * ell * sizeof(double)));
  LCK(cudaMalloc(&RinvT, (size_t)ell * ell * esz));
  LCK(cudaMalloc(&Pk, (size_t)ell * k * esz));
  LCK(cudaMalloc(&gpart, gp.part_elems * esz));
  LCK(cudaMalloc(&part, (size_t)1024 * sizeof(double)));
  LCK(cudaMalloc(&sums, 4 * sizeof(double)));
  LCK(cudaMalloc(&counters, gp.counters * sizeof(unsigned)));
  LCK(cudaMemsetAsync(counters, 0, gp.counters * sizeof(unsigned), s));
  LCK(cudaMalloc(&fail, sizeof(int)));
  LCK(cudaMemsetAsync(fail, 0, sizeof(int), s));
  LCK(cudaMalloc(&err, sizeof(int)));
  LCK(cudaMemsetAsync(err, 0, sizeof(int), s));
  Dims dl;
  dl.n = n; dl.r = ell; dl.b = 1; dl.N = ell; dl.ld = ell;

  // Omega (Gaussian, Philox) -> Q; Y = A Omega
  launch_philox_gaussian(td, Q, n, ell, seed, s);
  auto product = [&](const void* X, void* Out) -> int {
    const int sp = sketch_product(A, td, n, ell, X, Out, ws, ws_elems, xh, xl, err, s);
    if (sp < 0) { msg = "sketch product failed"; return -2; }
    if (sp > 1) launch_ax_finish_impl(td, dl, Out, ws, sp, 0.0, nullptr, nullptr, nullptr, part, 0, nullptr, s);
    return 0;
  };
  // Q <- orth(Y) by CholeskyQR2 (first pass with a tiny diagonal shift)
  auto cholqr = [&](void* Yb, void* Qb) -> int {
    for (int pass = 0; pass < 2; ++pass) {
      const void* src = pass == 0 ? Yb : Qb;
      launch_gram(td, src, src, dl, gp, 0, gpart, nullptr, nullptr, G, nullptr, -1, 0.0, counters, s);
      if (td == 0)
        k_chol<double><<<1, 256, 0, s>>>(G, ell, pass == 0 ? 1e-14 : 0.0, Rinv, (double*)RinvT, fail);
      else
        k_chol<float><<<1, 256, 0, s>>>(G, ell, pass == 0 ? 1e-7 : 0.0, Rinv, (float*)RinvT, fail);
      // Qb = src Rinv (via Yb when reading Qb: multiply into Yb then swap contents)
      void* dst = pass == 0 ? Qb : Yb;
      launch_rowmul(td, src, ell, ell, RinvT, ell, n, dst, ell, nullptr, s);
      if (pass == 1) {
        if (cudaMemcpyAsync(Qb, Yb, blk * esz, cudaMemcpyDeviceToDevice, s) != cudaSuccess) return -2;
      }
    }
    return 0;
  };
  if ((rc = product(Q, Y))) { cleanup(); return rc; }
  if ((rc = cholqr(Y, Q))) { cleanup(); return rc; }
  for (int it = 0; it < power_iters; ++it) {
    if ((rc = product(Q, Y))) { cleanup(); return rc; }
    if ((rc = cholqr(Y, Q))) { cleanup(); return rc; }
  }
  // T = Q^T (A Q), symmetrised; eigendecomposition; U = Q P_k
  if ((rc = product(Q, Y))) { cleanup(); return rc; }
  launch_gram(td, Q, Y, dl, gp, 0, gpart, nullptr, nullptr, G, nullptr, -1, 0.0, counters, s);
  k_sym<double><<<1, 256, 0, s>>>(G, ell);
  const int h = (ell + 1) / 2;
  k_jacobi<<<1, 256, 4 * h * sizeof(double), s>>>(G, V, ell, 40, 1e-13);
  LCK(cudaMalloc(&op.lam, (size_t)k * sizeof(double)));
  LCK(cudaMalloc(&op.U, (size_t)n * k * esz));
  if (td == 0) k_select<double><<<1, 256, 0, s>>>(G, V, ell, k, op.lam, (double*)Pk, sums);
  else k_select<float><<<1, 256, 0, s>>>(G, V, ell, k, op.lam, (float*)Pk, sums);
  launch_rowmul(td, Q, ell, ell, Pk, k, n, op.U, k, nullptr, s);
  double host_sums = 0.0;
  int host_fail = 0, host_err = 0;
  LCK(cudaMemcpyAsync(&host_sums, sums, sizeof(double), cudaMemcpyDeviceToHost, s));
  LCK(cudaMemcpyAsync(&host_fail, fail, sizeof(int), cudaMemcpyDeviceToHost, s));
  LCK(cudaMemcpyAsync(&host_err, err, sizeof(int), cudaMemcpyDeviceToHost, s));
  LCK(cudaStreamSynchronize(s));
  LCK(cudaGetLastError());
  if (host_fail || host_err) {
    msg = host_fail ? "CholeskyQR: non-positive pivot (sketch rank deficient)" : "sketch product wait timed out";
    cleanup();
    lai_free(op);
    return -2;
  }
  op.k = k;
  op.n = n;
  op.normA2 = host_sums;
  op.maxN = maxN;
  const int tq = utx_tq(maxN);
  const int64_t tiles = (int64_t)cdivi(k, 64) * cdivi(maxN, tq);
  int64_t nch = std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 3 * 152 / tiles));
  op.chunk = ((n + nch - 1) / nch + 31) / 32 * 32;
  op.nch = (int)((n + op.chunk - 1) / op.chunk);
  op.ng = gram_groups(op.nch);
  LCK(cudaMalloc(&op.xpart, (size_t)tiles * (op.nch + op.ng) * 64 * tq * esz));
  LCK(cudaMalloc(&op.M, (size_t)k * maxN * esz));
  LCK(cudaMalloc(&op.counters, (size_t)tiles * (1 + op.ng) * sizeof(unsigned)));
  LCK(cudaMemsetAsync(op.counters, 0, (size_t)tiles * (1 + op.ng) * sizeof(unsigned), s));
  LCK(cudaStreamSynchronize(s));
  cleanup();
  return 0;
#undef LCK
}

// SVD start of Sec. 4.1 guideline (4) from the eigen-sketch of a symmetric A (k = r): the
// singular values of A are |lambda| with left vectors U and right vectors U sign(lambda), so
// |U E^1/2| and |E^1/2 P^T|^T are both |U| |lambda|^1/2 (column-wise).  Written to every one of
// the b restart column blocks of W (n x r b, ld r b).
namespace {
template <typename T>
__global__ void k_svd_start(const T* __restrict__ U, const double* __restrict__ lam, int64_t n, int r, int b,
                            T* __restrict__ W) {
  const int64_t total = n * (int64_t)r;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / r;
    const int c = (int)(e % r);
    const T v = (T)(fabs((double)U[e]) * sqrt(fabs(lam[c])));
    for (int j = 0; j < b; ++j) W[i * (int64_t)r * b + (int64_t)j * r + c] = v;
  }
}
}  // namespace

void launch_svd_start(int tdtype, const LaiOp& op, int64_t n, int r, int b, void* W, cudaStream_t s) {
  const int blocks = (int)std::min<int64_t>((n * r + 255) / 256, 152 * 8);
  if (tdtype == 0) k_svd_start<double><<<blocks, 256, 0, s>>>((const double*)op.U, op.lam, n, r, b, (double*)W);
  else k_svd_start<float><<<blocks, 256, 0, s>>>((const float*)op.U, op.lam, n, r, b, (float*)W);
}

void lai_free(LaiOp& op) {
  cudaFree(op.U); cudaFree(op.lam); cudaFree(op.xpart); cudaFree(op.M); cudaFree(op.counters);
  op = LaiOp{};
}

}  // namespace snmf
