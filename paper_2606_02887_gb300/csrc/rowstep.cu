// Launchers of the row kernels of rowstep_dev.cuh over the restarts of a handle.
#include <algorithm>

#include "common.cuh"
#include "rowops.cuh"
#include "rowstep_dev.cuh"

namespace snmf {

namespace {

template <typename T, int STEP, int NC, int MR, int W>
__global__ void __launch_bounds__(256, 2) k_rowstep(RowArgs a, int tiles, bool vec) {
  extern __shared__ __align__(16) unsigned char rsm[];
  rowstep_body<T, STEP, NC, MR, W>(a, blockIdx.y, blockIdx.x, gridDim.x, tiles, vec, reinterpret_cast<T*>(rsm));
}

template <typename T, int STEP, int NC, int MR, int W>
void launch_t(const RowArgs& a, const RowStepPlan& pl, cudaStream_t s) {
  static SmemLimit limit;  // the most over the ranks: r = 128 with 256 threads and every input
  raise_smem_limit(limit, (const void*)k_rowstep<T, STEP, NC, MR, W>,
                   rowstep_smem<T>(sizeof(T) == 8 && MR > 1 ? 64 : 128, 256, MR, 7, W));
  uintptr_t all = 0;
  for (const void* p : {a.X, a.g_in, a.B, a.LX, (const void*)a.Xout, (const void*)a.gout, (const void*)a.Dout,
                        (const void*)a.gZout, a.Xold, a.gold, a.Zold, a.gZold, a.Wcur, a.gWcur, (const void*)a.Znext})
    all |= (uintptr_t)p;
  const bool vec = W == 1 || (a.r % 4 == 0 && a.ld % 4 == 0 && !(all & 15));
  dim3 grid((unsigned)pl.slots, (unsigned)a.b);
  k_rowstep<T, STEP, NC, MR, W>
      <<<grid, pl.threads, rowstep_smem<T>(a.r, pl.threads, MR, rowstep_inputs(STEP, a), W), s>>>(a, pl.tiles, vec);
}

}  // namespace

RowStepPlan rowstep_plan(int tdtype, int64_t n, int r, int b) {
  // 4 (FP64: 2) rows per thread of 128 or (r > 32) 256 threads; one row, and half the threads, while that
  // still makes no more than two CTAs per SM (n = 1000, r = 20: 84 CTAs of 12 rows; the general
  // kernel had 32 of 32)
  // Above r = 64 always 256 threads (G is copied by them) and one row each in FP64, whose G takes up
  // to 128 KB of the shared memory.
  const int big = (r + 3) / 4 > 8 ? 256 : 128;
  RowStepPlan pl{big, tdtype == 0 ? rowstep_mr<double>() : rowstep_mr<float>(), 4, 0, 0, 0};
  // FP64, an instruction of a warp taking 64 cycles of its SM partition: one column per thread while
  // threads of four columns would be fewer than a warp for each of the 608 partitions (n = 500, r = 10
  // in 24 CTAs of two warps with four columns each: D step 13.0 us, update 13.4)
  if (tdtype == 0 && n * r * b < 4 * 608 * 32 && r <= 64) {
    pl.w = 1;
    pl.mr = 1;
    pl.threads = r > 32 ? 256 : 128;
  }
  for (const auto& o : {std::pair<int, int>{big / 2, 1}, std::pair<int, int>{big, 1}}) {
    const int64_t rows = rowstep_rows(r, o.first, o.second);
    if (pl.w == 1 || (r > 64 && o.first < big)) continue;
    if (r > 64 && tdtype == 0) {
      pl.mr = 1;
      break;
    }
    if ((n + rows - 1) / rows * b <= 2 * 152) {
      pl.threads = o.first;
      pl.mr = o.second;
      break;
    }
  }
  pl.rows = rowstep_rows(r, pl.threads, pl.mr, pl.w);
  pl.tiles = (int)((n + pl.rows - 1) / pl.rows);
  // 512 threads per SM (r > 64: 256, the shared memory holds one CTA) over the restarts, each CTA as
  // many tiles as the next one
  const int most = std::max(1, (152 * ((r > 64 ? 256 : 512) / pl.threads) + b - 1) / b);
  const int each = (pl.tiles + most - 1) / most;
  pl.slots = (pl.tiles + each - 1) / each;
  return pl;
}

#define ROWSTEP(T, STEP, NC)                                    \
  do {                                                          \
    if (pl.mr == 1) launch_t<T, STEP, NC, 1, 4>(a, pl, s);      \
    else launch_t<T, STEP, NC, rowstep_mr<T>(), 4>(a, pl, s);   \
  } while (0)
#define ROWSTEP_T(STEP, NC)                                     \
  do {                                                          \
    if (pl.w == 1) launch_t<double, STEP, NC, 1, 1>(a, pl, s);  \
    else if (tdtype == 0) ROWSTEP(double, STEP, NC);            \
    else ROWSTEP(float, STEP, NC);                              \
  } while (0)

void launch_rowstep_grad(int tdtype, const RowArgs& a, const RowStepPlan& pl, cudaStream_t s) { ROWSTEP_T(RS_GRAD, 1); }

void launch_rowstep_d(int tdtype, const RowArgs& a, const RowStepPlan& pl, int nc, cudaStream_t s) {
  if (nc == 2) ROWSTEP_T(RS_D, 2);
  else ROWSTEP_T(RS_D, 1);
}

void launch_rowstep_dz(int tdtype, const RowArgs& a, const RowStepPlan& pl, cudaStream_t s) { ROWSTEP_T(RS_DZ, 1); }

void launch_rowstep_update(int tdtype, const RowArgs& a, const RowStepPlan& pl, int nc, cudaStream_t s) {
  if (nc == 2) ROWSTEP_T(RS_U, 2);
  else ROWSTEP_T(RS_U, 1);
}

#undef ROWSTEP_T
#undef ROWSTEP

}  // namespace snmf
