// One launch over several trees (multi.cu, multi_level.cu): per-call arguments.
#pragma once

#include "fst_internal.h"

namespace fst {

constexpr int kMaxMulti = FST_MAX_MULTI;

struct MultiIO {
  const float* q;
  const float* qd;
  const float* qdd;
  const float* tau;
  float* poses;
  float* tau_out;
  float* M;
  float* qdd_out;
  int64_t B;
};

// Work items: segment s covers items [seg_start[s], seg_start[s+1]), one
// tile of environments each, of operator seg_op[s] (a Role) on tree
// seg_model[s].
struct MultiArgs {
  ModelView mv[kMaxMulti];
  MultiIO io[kMaxMulti];
  int seg_start[4 * kMaxMulti + 1];
  unsigned char seg_model[4 * kMaxMulti];
  unsigned char seg_op[4 * kMaxMulti];
  int n_items;
  int max_rows;          // staged input rows of the widest item
  size_t model_bytes;    // shared memory reserved for the largest tree
  int* counter;          // generic form: device work counter (reset before each launch)
};

// The generic form (multi.cu): one environment per thread, `block` per item.
cudaError_t launch_multi(const MultiArgs& a, int max_n, int block, cudaStream_t s);
// The form in tiles (multi_level.cu): one block per item of 32 environments;
// smem: the largest multi_tile_smem of its (tree, operator) pairs.
size_t multi_tile_smem(const ModelView& mv, int role, int slots);
cudaError_t launch_multi_tiles(const MultiArgs& a, size_t smem, int block, cudaStream_t s);

}  // namespace fst

struct fst_multi {
  std::vector<const fst_model*> models;
  int* counter = nullptr;
  int device = -1;
  int block = 64;
  int variant = FST_VARIANT_AUTO;  // or FST_VARIANT_GENERIC, FST_VARIANT_LEVEL
};
