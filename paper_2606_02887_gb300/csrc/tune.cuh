// Launch configuration of the A*X product kernels chosen by the autotuner (tune.cu), and
// its JSON cache keyed by device.
#pragma once

#include <stdint.h>

#include <string>

namespace snmf {

// Zero fields keep the built-in heuristic of the kernel's launcher.
struct ProdTune {
  int splits = 0;   // split-K slices
  int stages = 0;   // tcgen05 product: shared-memory ring stages
  int per_sm = 0;   // tcgen05 product: CTAs planned per SM (sets the default split count)
  int bn = 0;       // tcgen05 product: output columns per CTA tile (multiple of 16, <= 256)
  int row_bm = 0;   // row kernels of a step (FP32): rows per CTA
  int row_tc = 0;   // the step's row products on the tensor cores (r = 64): 1 rowtc.cu, 2 rowtma.cu
  int64_t kchunk = 0;  // CUDA-core product: columns of A per split, a multiple of 16 (not in the cache)
};

struct TuneEntry {
  ProdTune cfg;
  double ms = 0.0;  // measured mean time of one product (CUDA events)
};

// "<device name>/<SM count>" of the current device ("" when it cannot be queried).
std::string tune_device_key();
// Cache lookup / store in the JSON file at `path` (NULL or empty: an in-process cache
// only).  The file maps device keys to shape keys ("dense/<dtype>/n<n>/r<r>/N<N>") to entries.  A file
// of the format's first version was timed with other tiles of the CUDA-core product (64 x 64 for every
// size), which says nothing about how to split K for the present ones: the `splits` of its FP64 and
// FP32 entries are left to the built-in rule (0).
bool tune_lookup(const char* path, const std::string& dev, const std::string& key, TuneEntry* out);
bool tune_store(const char* path, const std::string& dev, const std::string& key, const TuneEntry& e);

}  // namespace snmf
