// The level-parallel form of the persistent launch over several trees
// (multi.cu has the work list's description and the generic form).
#include "launch.h"
#include "level.cuh"
#include "multi.h"

namespace fst {
namespace {

// The same work list run with the level-parallel bodies (level.cuh): an item
// is 32 environments (one per lane) of one operator on one tree, and the
// block's warps split each of the tree's levels. Shared memory: the largest
// tree's model, the staged input rows, then the per-body state of the
// largest (tree, operator) pair. ABA runs in its lean form (aba_level_lean:
// 12 floats per body and a few contribution slots instead of 59 floats per
// body), so that the block's shared memory, sized for the largest pair, is
// not set by ABA.
__global__ void __launch_bounds__(256) multi_level_kernel(MultiArgs a) {
  extern __shared__ float4 smem[];
  __shared__ int s_item;
  float* tile = reinterpret_cast<float*>(reinterpret_cast<char*>(smem) + a.model_bytes);
  const int lane = threadIdx.x & 31;
  int cur = -1;
  SmemModel sm{nullptr, nullptr, 0};
  for (;;) {
    if (threadIdx.x == 0) s_item = atomicAdd(a.counter, 1);
    __syncthreads();
    const int item = s_item;
    __syncthreads();  // every thread has read s_item before thread 0 can overwrite it for the next item
    if (item >= a.n_items) break;
    int sg = 0;
    while (item >= a.seg_start[sg + 1]) ++sg;
    const int m = a.seg_model[sg];
    const int op = a.seg_op[sg];
    const ModelView& mv = a.mv[m];
    const MultiIO& io = a.io[m];
    if (m != cur) {
      sm = stage_model(mv, smem);  // synchronises the block
      cur = m;
    }
    const int64_t B = io.B;
    const int64_t e = (int64_t)(item - a.seg_start[sg]) * kLaneEnvs + lane;
    const bool act = e < B;
    stage_block_rows(tile, io.q, mv.nq, B, e);
    if (op == ROLE_RNEA) {
      stage_block_rows(tile + mv.nq * kLaneEnvs, io.qd, mv.nv, B, e);
      stage_block_rows(tile + (mv.nq + mv.nv) * kLaneEnvs, io.qdd, mv.nv, B, e);
    } else if (op == ROLE_ABA) {
      stage_block_rows(tile + mv.nq * kLaneEnvs, io.qd, mv.nv, B, e);
      stage_block_rows(tile + (mv.nq + mv.nv) * kLaneEnvs, io.tau, mv.nv, B, e);
    }
    cp_async_wait_all();
    __syncthreads();
    const Col cq{tile + lane, kLaneEnvs};
    const Col c1{tile + mv.nq * kLaneEnvs + lane, kLaneEnvs};
    const Col c2{tile + (mv.nq + mv.nv) * kLaneEnvs + lane, kLaneEnvs};
    float* state = tile + a.max_rows * kLaneEnvs;
    switch (op) {
      case ROLE_ABA:
        aba_level_lean(sm, world_accel(mv), cq, c1, c2, LaneState{state, kAbaLeanBodyFloats},
                       LaneState{state + kAbaLeanBodyFloats * mv.n * kLaneEnvs, kAbaLeanSlotFloats},
                       io.qdd_out, B, e, act);
        break;
      case ROLE_CRBA:
        crba_level(sm, cq, mv.nv, LaneState{state, kCrbaState}, io.M, B, e, act);
        break;
      case ROLE_RNEA:
        rnea_level(sm, world_accel(mv), cq, c1, c2, LaneState{state, kRneaState}, io.tau_out, B, e, act);
        break;
      default:
        fk_level(sm, cq, LaneState{state, kFkState}, io.poses, B, e, act);
        break;
    }
    __syncthreads();  // everyone is done with this item's shared memory
  }
}

}  // namespace

cudaError_t launch_multi_level(const MultiArgs& a, size_t state_bytes, int block, cudaStream_t s) {
  const size_t sh = a.model_bytes + (size_t)a.max_rows * kLaneEnvs * sizeof(float) + state_bytes;
  if (sh > kLevelSmemLimit) return cudaErrorInvalidConfiguration;
  cudaError_t err = cudaMemsetAsync(a.counter, 0, sizeof(int), s);
  if (err != cudaSuccess) return err;
  prepare(multi_level_kernel, sh);
  const int grid = persistent_grid(multi_level_kernel, block, sh, a.n_items);
  multi_level_kernel<<<grid, block, sh, s>>>(a);
  return cudaGetLastError();
}

}  // namespace fst
