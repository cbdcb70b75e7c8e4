// The mixed-tree launch in tiles (fst_multi_eval): the work list of multi.cu,
// one block per item of 32 environments x one operator x one tree, its warps
// sharing the bodies (level.cuh).
//
// The blocks are ordered heaviest first and the hardware hands them out in
// that order, which balances the SMs as the generic form's persistent grid
// does with its atomic work counter, but needs no counter to reset, no
// occupancy query and no second barrier per item. Shared memory is sized for
// the largest (tree, operator) pair, all in their lean forms: 71 KB for the
// 23-body tree's ABA, so three blocks an SM. Bound by the latency of the longest
// items (that tree's ABA, 11 levels three times over). Five trees, 7936
// environments: 70 us in the generic form, 19 here; a whole call 70.7 -> 30 us,
// which is the host's part.
#include "launch.h"
#include "level.cuh"
#include "multi.h"

namespace fst {
namespace {

__global__ void __launch_bounds__(256) multi_tile_kernel(const __grid_constant__ MultiArgs a) {
  extern __shared__ float4 smem[];
  const int item = blockIdx.x, lane = threadIdx.x & 31;
  int sg = 0;
  while (item >= a.seg_start[sg + 1]) ++sg;
  const int op = a.seg_op[sg];
  const ModelView& mv = a.mv[a.seg_model[sg]];
  const MultiIO& io = a.io[a.seg_model[sg]];
  pdl_launch();
  stage_model_begin(mv, smem);
  pdl_wait();
  float* const tile = smem_tile(smem, mv.n);
  const int64_t B = io.B;
  const int64_t e = (int64_t)(item - a.seg_start[sg]) * kLaneEnvs + lane;
  const bool act = e < B;
  int rows = mv.nq;
  stage_block_rows(tile, io.q, mv.nq, B, e);
  if (op == ROLE_RNEA || op == ROLE_ABA) {
    stage_block_rows(tile + rows * kLaneEnvs, io.qd, mv.nv, B, e);
    stage_block_rows(tile + (rows + mv.nv) * kLaneEnvs, op == ROLE_ABA ? io.tau : io.qdd, mv.nv, B, e);
    rows += 2 * mv.nv;
  }
  const SmemModel sm = stage_model_end(mv, smem);
  const Col cq{tile + lane, kLaneEnvs};
  const Col c1{tile + mv.nq * kLaneEnvs + lane, kLaneEnvs};
  const Col c2{tile + (mv.nq + mv.nv) * kLaneEnvs + lane, kLaneEnvs};
  float* const state = tile + rows * kLaneEnvs;
  switch (op) {
    case ROLE_ABA:
      aba_level_lean<true, true>(sm, world_accel(mv), cq, c1, c2, LaneState{state, kAbaLeanBodyFloats},
                     LaneState{state + kAbaLeanBodyFloats * mv.n * kLaneEnvs, kAbaLeanSlotFloats}, io.qdd_out, B, e,
                     act);
      break;
    case ROLE_CRBA:
      crba_level_lean(sm, [&](const BodyC& c, const BodyI& bi) { return joint_X(c, bi, cq); }, mv.nv,
                      LaneState{state, kCrbaLeanBodyFloats},
                      LaneState{state + kCrbaLeanBodyFloats * mv.n * kLaneEnvs, kCrbaLeanSlotFloats}, io.M, B, e, act);
      break;
    case ROLE_RNEA:
      rnea_level<true, true, true>(sm, world_accel(mv), cq, c1, c2, LaneState{state, kRneaLeanFloats}, io.tau_out, B,
                                   e, act);
      break;
    default:
      fk_level<true>(sm, cq, LaneState{state, kFkState}, io.poses, B, e, act);
      break;
  }
}

}  // namespace

size_t multi_tile_smem(const ModelView& mv, int role, int slots) {
  size_t f = mv.nq;
  if (role == ROLE_ABA)
    f += 2 * (size_t)mv.nv + (size_t)kAbaLeanBodyFloats * mv.n + (size_t)kAbaLeanSlotFloats * slots;
  else if (role == ROLE_CRBA)
    f += (size_t)kCrbaLeanBodyFloats * mv.n + (size_t)kCrbaLeanSlotFloats * slots;
  else if (role == ROLE_RNEA)
    f += 2 * (size_t)mv.nv + (size_t)kRneaLeanFloats * mv.n;
  else
    f += (size_t)kFkState * mv.n;
  return smem_bytes(mv.n) + f * kLaneEnvs * sizeof(float);
}

cudaError_t launch_multi_tiles(const MultiArgs& a, size_t smem, int block, cudaStream_t s) {
  if (smem > kLevelSmemLimit) return cudaErrorInvalidConfiguration;
  prepare(multi_tile_kernel, smem);
  return launch_pdl(multi_tile_kernel, (unsigned)a.n_items, block, smem, s, a);
}

}  // namespace fst
