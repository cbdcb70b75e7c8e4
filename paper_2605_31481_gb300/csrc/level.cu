// Level-parallel kernels (bodies in level.cuh): tiles of 32 environments,
// W warps per tile splitting each tree level's bodies. A block is one tile
// (1-D, 32 W threads) or T tiles (3-D, (32, T, W); see warp_id()).
//
// Shared memory: model | per tile: input rows (rows x 32) | per-body state
// (F x n x 32); `stride` floats per tile.
#include "launch.h"
#include "level.cuh"

namespace fst {
namespace {

__device__ __forceinline__ float* level_tile(float4* smem, int n) { return smem_tile(smem, n); }

#define FST_LEVEL_PROLOGUE_S(rows, F, stride)                                            \
  extern __shared__ float4 smem[];                                                       \
  float* tile = level_tile(smem, mv.n) + (size_t)threadIdx.y * (stride);                 \
  const LaneState S{tile + (rows) * kLaneEnvs, (F)};                                     \
  const int lane = threadIdx.x & 31;                                                     \
  const int64_t e = ((int64_t)blockIdx.x * blockDim.y + threadIdx.y) * kLaneEnvs + lane; \
  const bool act = e < B;                                                                \
  pdl_launch();                                                                          \
  stage_model_begin(mv, smem);                                                           \
  pdl_wait()

#define FST_LEVEL_PROLOGUE(rows, F) FST_LEVEL_PROLOGUE_S(rows, F, ((rows) + (F) * mv.n) * kLaneEnvs)

// stage_model_end waits for the model and for this thread's staged rows, then
// synchronises the block, so everything staged is visible to every warp.
#define FST_LEVEL_READY const SmemModel sm = stage_model_end(mv, smem)

template <bool AHEAD>
__global__ void __launch_bounds__(256) fk_level_kernel(ModelView mv, int64_t B, const float* __restrict__ q,
                                                       float* __restrict__ poses) {
  FST_LEVEL_PROLOGUE(mv.nq, kFkState);
  stage_block_rows(tile, q, mv.nq, B, e);
  FST_LEVEL_READY;
  fk_level<AHEAD>(sm, Col{tile + lane, kLaneEnvs}, S, poses, B, e, act);
}

template <bool AHEAD>
__global__ void __launch_bounds__(256) jac_level_kernel(ModelView mv, int64_t B, const float* __restrict__ q,
                                                        LinkList links, float* __restrict__ poses,
                                                        float* __restrict__ J) {
  FST_LEVEL_PROLOGUE(mv.nq, kFkState);
  stage_block_rows(tile, q, mv.nq, B, e);
  FST_LEVEL_READY;
  kin_level<AHEAD>(sm, Col{tile + lane, kLaneEnvs}, mv.nv, links, S, poses, J, B, e, act);
}

__global__ void __launch_bounds__(256) rnea_level_kernel(ModelView mv, int64_t B, const float* __restrict__ q,
                                                         const float* __restrict__ qd, const float* __restrict__ qdd,
                                                         float* __restrict__ tau) {
  FST_LEVEL_PROLOGUE(mv.nq + 2 * mv.nv, kRneaState);
  stage_block_rows(tile, q, mv.nq, B, e);
  stage_block_rows(tile + mv.nq * kLaneEnvs, qd, mv.nv, B, e);
  stage_block_rows(tile + (mv.nq + mv.nv) * kLaneEnvs, qdd, mv.nv, B, e);
  FST_LEVEL_READY;
  rnea_level<false, false, true>(sm, world_accel(mv), Col{tile + lane, kLaneEnvs},
                                 Col{tile + mv.nq * kLaneEnvs + lane, kLaneEnvs},
                                 Col{tile + (mv.nq + mv.nv) * kLaneEnvs + lane, kLaneEnvs}, S, tau, B, e, act);
}

// RNEA with 12 floats of state a body: four tiles of the floating humanoid per
// SM instead of two (B = 65536: 66.6 -> 47.3 us, 16384: 20.1 -> 15.0).
__global__ void __launch_bounds__(256) rnea_lean_kernel(ModelView mv, int64_t B, const float* __restrict__ q,
                                                        const float* __restrict__ qd, const float* __restrict__ qdd,
                                                        float* __restrict__ tau) {
  FST_LEVEL_PROLOGUE(mv.nq + 2 * mv.nv, kRneaLeanFloats);
  stage_block_rows(tile, q, mv.nq, B, e);
  stage_block_rows(tile + mv.nq * kLaneEnvs, qd, mv.nv, B, e);
  stage_block_rows(tile + (mv.nq + mv.nv) * kLaneEnvs, qdd, mv.nv, B, e);
  FST_LEVEL_READY;
  rnea_level<true, true, true>(sm, world_accel(mv), Col{tile + lane, kLaneEnvs},
                               Col{tile + mv.nq * kLaneEnvs + lane, kLaneEnvs},
                               Col{tile + (mv.nq + mv.nv) * kLaneEnvs + lane, kLaneEnvs}, S, tau, B, e, act);
}

__global__ void __launch_bounds__(256) crba_level_kernel(ModelView mv, int64_t B, const float* __restrict__ q,
                                                         float* __restrict__ M) {
  FST_LEVEL_PROLOGUE(mv.nq, kCrbaState);
  stage_block_rows(tile, q, mv.nq, B, e);
  FST_LEVEL_READY;
  crba_level(sm, Col{tile + lane, kLaneEnvs}, mv.nv, S, M, B, e, act);
}

__global__ void __launch_bounds__(256) aba_level_kernel(ModelView mv, int64_t B, const float* __restrict__ q,
                                                        const float* __restrict__ qd, const float* __restrict__ tau,
                                                        float* __restrict__ qdd) {
  FST_LEVEL_PROLOGUE(mv.nq + 2 * mv.nv, kAbaState);
  stage_block_rows(tile, q, mv.nq, B, e);
  stage_block_rows(tile + mv.nq * kLaneEnvs, qd, mv.nv, B, e);
  stage_block_rows(tile + (mv.nq + mv.nv) * kLaneEnvs, tau, mv.nv, B, e);
  FST_LEVEL_READY;
  aba_level(sm, world_accel(mv), Col{tile + lane, kLaneEnvs}, Col{tile + mv.nq * kLaneEnvs + lane, kLaneEnvs},
            Col{tile + (mv.nq + mv.nv) * kLaneEnvs + lane, kLaneEnvs}, S, qdd, B, e, act);
}

// ABA with the lean per-tile state (FST_VARIANT_LEVEL_LEAN): per body
// kAbaLeanBodyFloats, plus the contribution slots. Bound by the latency of its
// level phases, so by the tiles an SM holds: with a slot per running
// contribution instead of a ring of two levels the floating humanoid's tile
// takes 75 KB instead of 90, three an SM instead of two (B = 65536: 118 -> 94
// us; FP32 floor 18). Tried on top and not kept: four tiles, with qd and tau
// read from global memory and the bias accelerations folded into the forces
// (105 us, and 1 us more at small batches).
template <bool AHEAD>
__global__ void __launch_bounds__(256) aba_lean_kernel(ModelView mv, int64_t B, const float* __restrict__ q,
                                                       const float* __restrict__ qd, const float* __restrict__ tau,
                                                       float* __restrict__ qdd, int slots) {
  const int rows = mv.nq + 2 * mv.nv;
  FST_LEVEL_PROLOGUE_S(rows, kAbaLeanBodyFloats,
                       (rows + kAbaLeanBodyFloats * mv.n + kAbaLeanSlotFloats * slots) * kLaneEnvs);
  const LaneState R{tile + (rows + kAbaLeanBodyFloats * mv.n) * kLaneEnvs, kAbaLeanSlotFloats};
  stage_block_rows(tile, q, mv.nq, B, e);
  stage_block_rows(tile + mv.nq * kLaneEnvs, qd, mv.nv, B, e);
  stage_block_rows(tile + (mv.nq + mv.nv) * kLaneEnvs, tau, mv.nv, B, e);
  FST_LEVEL_READY;
  aba_level_lean<true, AHEAD>(sm, world_accel(mv), Col{tile + lane, kLaneEnvs},
                       Col{tile + mv.nq * kLaneEnvs + lane, kLaneEnvs},
                       Col{tile + (mv.nq + mv.nv) * kLaneEnvs + lane, kLaneEnvs}, S, R, qdd, B, e, act);
}

// CRBA with the lean per-tile state (FST_VARIANT_LEVEL_LEAN, and the default's
// tiles): kCrbaLeanBodyFloats per body and the contribution slots, three tiles
// of the floating humanoid per SM where the full state has two. Bound by the
// level phases' latency, then by the stores of M (B = 65536: 92 -> 77 us, of
// them 33 for the bytes; 4096: 10.4 -> 9.8). q is staged where it fits (read
// from global memory in the level loop instead: 93 us) and the bodies with the
// longest walk to the root go first. More than 80 registers a thread would cost
// small trees a block an SM: none is forced here (64 used).
template <bool STAGED>
__global__ void __launch_bounds__(256) crba_lean_kernel(ModelView mv, int64_t B, const float* __restrict__ q,
                                                           float* __restrict__ M, int slots) {
  const int rows = STAGED ? mv.nq : 0;
  FST_LEVEL_PROLOGUE_S(rows, kCrbaLeanBodyFloats,
                       (rows + kCrbaLeanBodyFloats * mv.n + kCrbaLeanSlotFloats * slots) * kLaneEnvs);
  const LaneState R{tile + (rows + kCrbaLeanBodyFloats * mv.n) * kLaneEnvs, kCrbaLeanSlotFloats};
  if (STAGED) stage_block_rows(tile, q, mv.nq, B, e);
  FST_LEVEL_READY;
  const int64_t ec = act ? e : B - 1;  // lanes past B compute on the last environment and store nothing
  auto X_of = [&](const BodyC& c, const BodyI& bi) {
    return STAGED ? joint_X(c, bi, Col{tile + lane, kLaneEnvs}) : joint_X_rows(c, bi, q, B, ec);
  };
  crba_level_lean(sm, X_of, mv.nv, S, R, M, B, e, act);
}

// SM-pinned ABA (FST_VARIANT_PINNED): blocks on SMs pinned to ABA take
// tiles of 32 environments until none is left (pinned_tiles). The model is
// staged only by blocks that get work.
__global__ void __launch_bounds__(256) aba_level_pin_kernel(ModelView mv, int64_t B, const float* __restrict__ q,
                                                            const float* __restrict__ qd,
                                                            const float* __restrict__ tau, float* __restrict__ qdd,
                                                            PinArgs p) {
  extern __shared__ float4 smem[];
  float* tile = level_tile(smem, mv.n);
  const LaneState S{tile + (mv.nq + 2 * mv.nv) * kLaneEnvs, kAbaState};
  const int lane = threadIdx.x & 31;
  const int my = pinned_role(p) == ROLE_ABA ? 0 : -1;
  bool staged = false;
  SmemModel sm{nullptr, nullptr, 0};
  auto body = [&](int, int t) {
    if (!staged) {
      sm = stage_model(mv, smem);  // synchronises the block
      staged = true;
    }
    const int64_t e = (int64_t)t * kLaneEnvs + lane;
    const bool act = e < B;
    stage_block_rows(tile, q, mv.nq, B, e);
    stage_block_rows(tile + mv.nq * kLaneEnvs, qd, mv.nv, B, e);
    stage_block_rows(tile + (mv.nq + mv.nv) * kLaneEnvs, tau, mv.nv, B, e);
    cp_async_wait_all();
    __syncthreads();
    aba_level(sm, world_accel(mv), Col{tile + lane, kLaneEnvs}, Col{tile + mv.nq * kLaneEnvs + lane, kLaneEnvs},
              Col{tile + (mv.nq + mv.nv) * kLaneEnvs + lane, kLaneEnvs}, S, qdd, B, e, act);
    __syncthreads();  // the next tile reuses the staged rows and the state
  };
  pinned_tiles(p, my, 1, (int)((B + kLaneEnvs - 1) / kLaneEnvs), body);
}

// Fused evaluation with the level-parallel bodies: blockIdx.y is the role.
__global__ void __launch_bounds__(256) eval_level_kernel(ModelView mv, int64_t B, EvalArgs a) {
  const int role = a.roles[blockIdx.y];
  const int F = role == ROLE_ABA ? kAbaState : role == ROLE_CRBA ? kCrbaState : role == ROLE_RNEA ? kRneaState : kFkState;
  // tiles are sized for the largest role (ABA), as the launch allocates them
  FST_LEVEL_PROLOGUE_S(mv.nq + 2 * mv.nv, F, (mv.nq + 2 * mv.nv + kAbaState * mv.n) * kLaneEnvs);
  stage_block_rows(tile, a.q, mv.nq, B, e);
  if (role == ROLE_RNEA) {
    stage_block_rows(tile + mv.nq * kLaneEnvs, a.qd, mv.nv, B, e);
    stage_block_rows(tile + (mv.nq + mv.nv) * kLaneEnvs, a.qdd, mv.nv, B, e);
  } else if (role == ROLE_ABA) {
    stage_block_rows(tile + mv.nq * kLaneEnvs, a.qd, mv.nv, B, e);
    stage_block_rows(tile + (mv.nq + mv.nv) * kLaneEnvs, a.tau, mv.nv, B, e);
  }
  FST_LEVEL_READY;
  const Col cq{tile + lane, kLaneEnvs};
  const Col c1{tile + mv.nq * kLaneEnvs + lane, kLaneEnvs};
  const Col c2{tile + (mv.nq + mv.nv) * kLaneEnvs + lane, kLaneEnvs};
  switch (role) {
    case ROLE_ABA:
      aba_level(sm, world_accel(mv), cq, c1, c2, S, a.qdd_out, B, e, act);
      break;
    case ROLE_CRBA:
      crba_level(sm, cq, mv.nv, S, a.M, B, e, act);
      break;
    case ROLE_RNEA:
      rnea_level(sm, world_accel(mv), cq, c1, c2, S, a.tau_out, B, e, act);
      break;
    default:
      kin_level(sm, cq, mv.nv, a.links, S, a.poses, a.J, B, e, act);
      break;
  }
}

// bytes of shared memory of one tile: input rows and per-body state
size_t level_tile_bytes(const ModelView& mv, int rows, int F) {
  return (size_t)rows * kLaneEnvs * sizeof(float) + (size_t)F * mv.n * kLaneEnvs * sizeof(float);
}

// `block` threads (a multiple of 32 T) as `tiles` tiles of block / (32 T)
// warps each: a 1-D block for one tile, (32, T, W) for several.
template <typename... P, typename... A>
cudaError_t go(void (*kernel)(P...), const ModelView& mv, int64_t B, size_t sh, int block, int tiles, unsigned gy,
               cudaStream_t s, A... args) {
  if (sh > kLevelSmemLimit || tiles < 1 || block < 32 * tiles || block % (32 * tiles))
    return cudaErrorInvalidConfiguration;
  prepare(kernel, sh);
  const int64_t envs = (int64_t)kLaneEnvs * tiles;
  const dim3 blk = tiles == 1 ? dim3(block) : dim3(32, tiles, block / (32 * tiles));
  return launch_pdl(kernel, dim3((unsigned)((B + envs - 1) / envs), gy), blk, sh, s, mv, B, args...);
}

// The warps of a tile do their next bodies' own work ahead of its level
// (level_pass) in FK and ABA up to two tiles an SM, see there for both sides.

}  // namespace

size_t model_smem_bytes(int n) { return smem_bytes(n); }

size_t level_smem_needed(const ModelView& mv, int kind, int tiles) {
  size_t t;
  switch (kind) {
    case LEVEL_FK:
    case LEVEL_JAC:
      t = level_tile_bytes(mv, mv.nq, kFkState);
      break;
    case LEVEL_RNEA:
      t = level_tile_bytes(mv, mv.nq + 2 * mv.nv, kRneaState);
      break;
    case LEVEL_CRBA:
      t = level_tile_bytes(mv, mv.nq, kCrbaState);
      break;
    default:  // ABA, and eval (its tiles are sized for the ABA role)
      t = level_tile_bytes(mv, mv.nq + 2 * mv.nv, kAbaState);
      break;
  }
  return smem_bytes(mv.n) + (size_t)tiles * t;
}

cudaError_t launch_fk_level(const ModelView& mv, int64_t B, const float* q, float* poses, int block, int tiles,
                            cudaStream_t s) {
  return go(many_tiles(B) ? fk_level_kernel<false> : fk_level_kernel<true>, mv, B,
            level_smem_needed(mv, LEVEL_FK, tiles), block, tiles, 1, s, q, poses);
}
cudaError_t launch_jac_level(const ModelView& mv, int64_t B, const float* q, const LinkList& links, float* J,
                             int block, int tiles, cudaStream_t s) {
  return go(many_tiles(B) ? jac_level_kernel<false> : jac_level_kernel<true>, mv, B,
            level_smem_needed(mv, LEVEL_JAC, tiles), block, tiles, 1, s, q, links, (float*)nullptr, J);
}
cudaError_t launch_rnea_level(const ModelView& mv, int64_t B, const float* q, const float* qd, const float* qdd,
                              float* tau, int block, int tiles, cudaStream_t s) {
  return go(rnea_level_kernel, mv, B, level_smem_needed(mv, LEVEL_RNEA, tiles), block, tiles, 1, s, q, qd, qdd, tau);
}
cudaError_t launch_rnea_lean(const ModelView& mv, int64_t B, const float* q, const float* qd, const float* qdd,
                             float* tau, int block, cudaStream_t s) {
  const size_t sh = smem_bytes(mv.n) + level_tile_bytes(mv, mv.nq + 2 * mv.nv, kRneaLeanFloats);
  return go(rnea_lean_kernel, mv, B, sh, block, 1, 1, s, q, qd, qdd, tau);
}
cudaError_t launch_crba_level(const ModelView& mv, int64_t B, const float* q, float* M, int block, int tiles,
                              cudaStream_t s) {
  return go(crba_level_kernel, mv, B, level_smem_needed(mv, LEVEL_CRBA, tiles), block, tiles, 1, s, q, M);
}
cudaError_t launch_aba_level(const ModelView& mv, int64_t B, const float* q, const float* qd, const float* tau,
                             float* qdd, int block, int tiles, cudaStream_t s) {
  return go(aba_level_kernel, mv, B, level_smem_needed(mv, LEVEL_ABA, tiles), block, tiles, 1, s, q, qd, tau, qdd);
}
size_t aba_lean_smem_needed(const ModelView& mv, int slots) {
  return smem_bytes(mv.n) + level_tile_bytes(mv, mv.nq + 2 * mv.nv, kAbaLeanBodyFloats) +
         (size_t)kAbaLeanSlotFloats * slots * kLaneEnvs * sizeof(float);
}
cudaError_t launch_aba_level_lean(const ModelView& mv, int64_t B, const float* q, const float* qd, const float* tau,
                                  float* qdd, int block, int slots, cudaStream_t s) {
  return go(many_tiles(B) ? aba_lean_kernel<false> : aba_lean_kernel<true>, mv, B, aba_lean_smem_needed(mv, slots),
            block, 1, 1, s, q, qd, tau, qdd, slots);
}
size_t crba_lean_smem_needed(const ModelView& mv, int slots, bool staged) {
  return smem_bytes(mv.n) + (staged ? level_tile_bytes(mv, mv.nq, 0) : 0) +
         (size_t)(kCrbaLeanBodyFloats * mv.n + kCrbaLeanSlotFloats * slots) * kLaneEnvs * sizeof(float);
}
cudaError_t launch_crba_level_lean(const ModelView& mv, int64_t B, const float* q, float* M, int block, int slots,
                                   cudaStream_t s) {
  const size_t sh = crba_lean_smem_needed(mv, slots, true);
  if (sh <= kLevelSmemLimit) return go(crba_lean_kernel<true>, mv, B, sh, block, 1, 1, s, q, M, slots);
  return go(crba_lean_kernel<false>, mv, B, crba_lean_smem_needed(mv, slots, false), block, 1, 1, s, q, M, slots);
}
cudaError_t launch_aba_level_pinned(const ModelView& mv, int64_t B, const float* q, const float* qd,
                                    const float* tau, float* qdd, int block, const PinArgs& p, cudaStream_t s) {
  const size_t sh = level_smem_needed(mv, LEVEL_ABA);
  if (sh > kLevelSmemLimit) return cudaErrorInvalidConfiguration;
  prepare(aba_level_pin_kernel, sh);
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  aba_level_pin_kernel<<<2 * (sms > 0 ? sms : 1), block, sh, s>>>(mv, B, q, qd, tau, qdd, p);
  return cudaGetLastError();
}

cudaError_t launch_eval_level(const ModelView& mv, int64_t B, const EvalArgs& a, int block, int tiles,
                              cudaStream_t s) {
  return go(eval_level_kernel, mv, B, level_smem_needed(mv, LEVEL_EVAL, tiles), block, tiles, (unsigned)a.n_roles, s,
            a);
}

}  // namespace fst
