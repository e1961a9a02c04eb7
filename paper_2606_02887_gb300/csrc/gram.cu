// r x r Gram X_j^T Y_j of each restart j (Eq. (2.1): H H^T, and the Z^T D, D^T D products of the
// line-search polynomial) and rho = ||G||_2 by the power method (Alg. 1 line 2, Eq. (2.11)).
#include <algorithm>

#include "common.cuh"
#include "gram_dev.cuh"
#include "rowops.cuh"

namespace snmf {

namespace {

// Gram of one restart's columns: CTA (chunk, restart x tile), see gram_body.
template <typename T, int TW, int VEC, int M = 4>
__global__ void __launch_bounds__(256, 3)
k_gram(const T* __restrict__ X, const T* __restrict__ Y, int64_t n, int r, int64_t ld, GramPlan pl,
       T* __restrict__ gpart, const Ctl* __restrict__ ctl, const int* run, double* __restrict__ G64,
       T* __restrict__ GT, T lam, unsigned* __restrict__ counters, Ctl* __restrict__ rho_ctl, int rho_iters,
       double rho_scale, double rho_shift) {
  extern __shared__ __align__(16) unsigned char gsm[];
  const int j = blockIdx.y / (pl.ntile * pl.ntile), tile = blockIdx.y % (pl.ntile * pl.ntile);
  if ((run && *run == 0) || (ctl && !ctl[j].active)) return;
  GramOut<T> o;
  o.r = r;
  o.p0 = tile / pl.ntile * TW;
  o.q0 = tile % pl.ntile * TW;
  o.G64 = G64 + (int64_t)j * r * r;
  o.GT = GT ? GT + (int64_t)j * r * r : nullptr;
  o.lam = lam;
  o.rho_ctl = rho_ctl ? rho_ctl + j : nullptr;
  o.rho_iters = rho_iters;
  o.rho_scale = rho_scale;
  o.rho_shift = rho_shift;
  gram_body<T, TW, VEC, M>(X + (int64_t)j * r + o.p0, Y + (int64_t)j * r + o.q0, min(TW, r - o.p0), min(TW, r - o.q0), ld,
                        n, pl.chunk, blockIdx.x, pl.nch, pl.ng, X == Y && o.p0 == o.q0,
                        gpart + (int64_t)blockIdx.y * (pl.nch + pl.ng) * (TW * TW), counters + (int64_t)blockIdx.y * (1 + pl.ng),
                        o, reinterpret_cast<T*>(gsm));
}

// rho = rho_scale ||G||_2 + rho_shift of a Gram in memory, one block per restart.  PT is the
// arithmetic type (double in FP64 precision, float otherwise).
// r <= 64: the Gram's own power method on a copy of G in shared memory.  Larger ranks: 1024
// threads, TPR per row with EPT columns each, RG of them in registers and (FP32, r > 128) the
// rest in shared memory; FP64 of r > 128 reads G from L2 in every product, and scales the sums by the
// power of two instead of G's entries (the same bits: as many ldexp as entries were half of its time).
// n = 100: 276 us with 256 threads that read G from shared memory and took the norm in every iteration.
template <typename PT, int TW>
__global__ void __launch_bounds__(256) k_rho(const double* __restrict__ G64, int r, int iters, double rho_scale,
                                             double rho_shift, Ctl* __restrict__ ctl) {
  __shared__ __align__(16) PT Gs[TW * TW];
  Ctl& c = ctl[blockIdx.x];
  if (!c.active) return;
  const double* G = G64 + (int64_t)blockIdx.x * r * r;
  for (int e = threadIdx.x; e < TW * TW; e += 256) {
    const int p = e / TW, q = e % TW;
    Gs[e] = p < r && q < r ? (PT)__ldcg(G + p * r + q) : PT(0);
  }
  __syncthreads();
  rho_in_smem<PT, TW>(Gs, r, iters, rho_scale, rho_shift, c);
}

template <typename PT, int TPR, int EPT, int RG, bool SMEM>
__global__ void __launch_bounds__(1024) k_rho_wide(const double* __restrict__ G64, int r, int iters, double rho_scale,
                                                   double rho_shift, Ctl* __restrict__ ctl) {
  extern __shared__ __align__(16) unsigned char rho_raw[];
  __shared__ __align__(16) PT vs[2 * (EPT + 4) * TPR];
  __shared__ PT red[64];
  PT* rest = reinterpret_cast<PT*>(rho_raw);  // SMEM: column RG + u of thread t at [u][t]
  Ctl& c = ctl[blockIdx.x];
  if (!c.active) return;
  const double* G = G64 + (int64_t)blockIdx.x * r * r;
  const int t = threadIdx.x, p = t / TPR, q0 = t % TPR * EPT;
  PT tr = PT(0);
  for (int q = t & 31; q < r; q += 32) tr += (PT)__ldcg(G + q * r + q);
  tr = lanes_sum(tr);
  const int e = trace_exponent(tr);
  auto raw = [&](int u) { return p < r && q0 + u < r ? __ldcg(G + (int64_t)(q0 + u) * r + p) : 0.0; };
  auto entry = [&](int u) { return (PT)ldexp(raw(u), -e); };
  PT g[RG > 0 ? RG : 1];
#pragma unroll
  for (int u = 0; u < RG; ++u) g[u] = entry(u);
  if (SMEM)
    for (int u = RG; u < EPT; ++u) rest[(u - RG) * 1024 + t] = entry(u);
  const PT norm = power_norm<PT, TPR>(r, EPT, 1024, iters,
                                      [&](const PT* v) {
                                        PT s[4] = {PT(0), PT(0), PT(0), PT(0)};
#pragma unroll
                                        for (int u = 0; u < RG; u += 4) {
                                          const Quad<PT> x = *reinterpret_cast<const Quad<PT>*>(v + u);
#pragma unroll
                                          for (int k = 0; k < 4; ++k) s[k] = fma(g[u + k], x.v[k], s[k]);
                                        }
#pragma unroll 2
                                        for (int u = RG; u < EPT; u += 4) {
                                          const Quad<PT> x = *reinterpret_cast<const Quad<PT>*>(v + u);
#pragma unroll
                                          for (int k = 0; k < 4; ++k)
                                            s[k] = fma(SMEM ? rest[(u - RG + k) * 1024 + t] : (PT)raw(u + k), x.v[k], s[k]);
                                        }
                                        const PT sum = (s[0] + s[1]) + (s[2] + s[3]);
                                        return RG == 0 && !SMEM ? (PT)ldexp(sum, -e) : sum;
                                      },
                                      vs, red);
  if (t == 0) set_rho(c, ldexp((double)norm, e), rho_scale, rho_shift);
}

}  // namespace

GramPlan gram_plan(int tdtype, int64_t n, int r, int b) {
  GramPlan pl;
  pl.tw = gram_tw(r);
  pl.ntile = r <= 64 ? 1 : (r + 63) / 64;
  const int64_t tiles = (int64_t)b * pl.ntile * pl.ntile;
  // one wave of three CTAs per SM over the tiles, chunks of at least 64 rows (32 in FP64, whose pipes
  // are slow); up to 32 chunks fit one level of 16 partials (n = 1000, r = 20: 16 chunks 10 us,
  // one chunk 50 us)
  const int64_t least = tdtype == 0 ? 32 : 64;
  int64_t nch = std::min<int64_t>((n + least - 1) / least, 3 * 152 / tiles);
  if (nch > kGramGroup && nch <= 2 * kGramGroup) nch = kGramGroup;
  if (nch < 1) nch = 1;
  pl.chunk = ((n + nch - 1) / nch + 31) / 32 * 32;
  pl.nch = (int)((n + pl.chunk - 1) / pl.chunk);
  pl.ng = gram_groups(pl.nch);
  pl.part_elems = (size_t)tiles * (pl.nch + pl.ng) * pl.tw * pl.tw;
  pl.counters = (size_t)tiles * (1 + pl.ng);
  return pl;
}

GramPlan gram_plan_sketch(int64_t n, int ell) {
  // one chain per entry: 2 x 2 micro tiles in a 32-wide tile (a sketch of 18 columns, FP64 n = 500: 5.60 ms with
  // the 64-wide tile for every width, 2.94 so)
  GramPlan pl;
  pl.micro = ell <= 32 ? 2 : 4;
  pl.tw = 16 * pl.micro;
  pl.ntile = (ell + 63) / 64;
  const int64_t tiles = (int64_t)pl.ntile * pl.ntile;
  const int64_t nch = std::max<int64_t>(1, std::min<int64_t>(152 / tiles, n / 512));
  pl.chunk = (n + nch - 1) / nch;
  pl.nch = (int)((n + pl.chunk - 1) / pl.chunk);
  pl.ng = 0;
  pl.part_elems = (size_t)tiles * pl.nch * pl.tw * pl.tw;
  pl.counters = (size_t)tiles;
  return pl;
}

template <typename T, int TW, int VEC, int M = 4>
static void launch_gram_t(const void* X, const void* Y, const Dims& d, const GramPlan& pl, void* gpart, const Ctl* ctl,
                          const int* run, double* G64, void* GT, double lam, unsigned* counters, Ctl* rho_ctl,
                          int rho_iters, double rho_scale, double rho_shift, cudaStream_t s) {
  static SmemLimit limit;
  raise_smem_limit(limit, (const void*)k_gram<T, TW, VEC, M>, gram_smem<T>(false));
  const size_t smem = gram_smem<T>(X == Y && pl.ntile == 1);
  dim3 grid(pl.nch, d.b * pl.ntile * pl.ntile);
  k_gram<T, TW, VEC, M><<<grid, 256, smem, s>>>((const T*)X, (const T*)Y, d.n, d.r, d.ld, pl, (T*)gpart, ctl, run, G64,
                                             (T*)GT, (T)lam, counters, rho_ctl, rho_iters, rho_scale, rho_shift);
}

void launch_gram(int tdtype, const void* X, const void* Y, const Dims& d, const GramPlan& pl, int pair, void* gpart,
                 const Ctl* ctl, const int* run, double* G64, void* GT, int tpair, double lam_shift, unsigned* counters,
                 cudaStream_t s, Ctl* rho_ctl, int rho_iters, double rho_scale, double rho_shift) {
  if (pl.ntile > 1) rho_ctl = nullptr;  // launch_rho
  G64 += (int64_t)pair * d.b * d.r * d.r;
  if (pair != tpair) GT = nullptr;
  // 16-byte copies when every restart's rows start on 16 bytes
  const int v = tdtype == 0 ? 2 : 4;
  const bool vec = d.r % v == 0 && d.ld % v == 0 && !((uintptr_t)X & 15) && !((uintptr_t)Y & 15);
#define GRAM(T, ...)                                                                                               \
  launch_gram_t<T, __VA_ARGS__>(X, Y, d, pl, gpart, ctl, run, G64, GT, lam_shift, counters, rho_ctl, rho_iters, rho_scale, \
                          rho_shift, s)
#define GRAM_T(T, V)                            \
  if (pl.micro == 2) {                          \
    if (vec) GRAM(T, 32, V, 2); else GRAM(T, 32, 1, 2); \
  } else if (pl.tw == 16) {                     \
    if (vec) GRAM(T, 16, V); else GRAM(T, 16, 1); \
  } else if (pl.tw == 32) {                     \
    if (vec) GRAM(T, 32, V); else GRAM(T, 32, 1); \
  } else {                                      \
    if (vec) GRAM(T, 64, V); else GRAM(T, 64, 1); \
  }
  if (tdtype == 0) { GRAM_T(double, 2) } else { GRAM_T(float, 4) }
#undef GRAM_T
#undef GRAM
}

void launch_rho(int tdtype, const double* G64, const Dims& d, int iters, double scale, Ctl* ctl, cudaStream_t s,
                double shift) {
#define RHO_ARGS G64, d.r, iters, scale, shift, ctl
#define RHO(PT)                                                            \
  if (d.r <= 16) k_rho<PT, 16><<<d.b, 256, 0, s>>>(RHO_ARGS);              \
  else if (d.r <= 32) k_rho<PT, 32><<<d.b, 256, 0, s>>>(RHO_ARGS);         \
  else if (d.r <= 64) k_rho<PT, 64><<<d.b, 256, 0, s>>>(RHO_ARGS);         \
  else if (d.r <= 128) k_rho_wide<PT, 8, 16, 16, false><<<d.b, 1024, 0, s>>>(RHO_ARGS);
  if (tdtype == 0) {
    RHO(double) else k_rho_wide<double, 4, 64, 0, false><<<d.b, 1024, 0, s>>>(RHO_ARGS);
  } else {
    RHO(float) else {
      static SmemLimit limit;
      raise_smem_limit(limit, (const void*)k_rho_wide<float, 4, 64, 32, true>, 128 * 1024);
      k_rho_wide<float, 4, 64, 32, true><<<d.b, 1024, 128 * 1024, s>>>(RHO_ARGS);
    }
  }
#undef RHO
#undef RHO_ARGS
}

}  // namespace snmf
