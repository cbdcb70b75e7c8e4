// Kernels of aligned.cuh: tiles of 32 environments (one per lane), one tile
// per block, the block's warps sharing the bodies.
//
// Shared memory: model | input rows x 32 | per-body state x 32 | (forward
// dynamics) the tree-sparse mass matrix and its index lists.
#include "aligned.cuh"
#include "launch.h"

namespace fst {
namespace {

#define FST_TILE                                                 \
  extern __shared__ float4 smem[];                               \
  float* const tile = smem_tile(smem, mv.n);                     \
  const int lane = threadIdx.x & 31;                             \
  const int64_t e = (int64_t)blockIdx.x * kLaneEnvs + lane;      \
  const bool act = e < B;                                        \
  pdl_launch();                                                  \
  stage_model_begin(mv, smem);                                   \
  pdl_wait()

__device__ __forceinline__ Col tile_col(float* tile, int row) {
  return Col{tile + row * kLaneEnvs + (threadIdx.x & 31), kLaneEnvs};
}

// Dense derivatives of inverse dynamics. Bound by the latency of its phases
// (one tile of the humanoid, 159 KB, per SM: 21 barriers, each behind the
// dependent loads and arithmetic of one body), not by its stores. The kernel
// that it replaces as the default swept one tangent per degree of freedom
// through the whole tree in one thread per environment, nv times the
// recursions' work and their state in local memory: floating humanoid,
// B = 2048: 418 -> 21.5 us; quadruped, B = 4096: 61.6 -> 14 us.
template <int T>
__global__ void __launch_bounds__(T) rnea_derivs_aligned_kernel(ModelView mv, int64_t B, const float* __restrict__ q,
                                                                  const float* __restrict__ qd,
                                                                  const float* __restrict__ qdd,
                                                                  float* __restrict__ dq, float* __restrict__ dqd) {
  FST_TILE;
  stage_block_rows(tile, q, mv.nq, B, e);
  stage_block_rows(tile + mv.nq * kLaneEnvs, qd, mv.nv, B, e);
  stage_block_rows(tile + (mv.nq + mv.nv) * kLaneEnvs, qdd, mv.nv, B, e);
  const SmemModel sm = stage_model_end(mv, smem);
  const LaneState S{tile + (mv.nq + 2 * mv.nv) * kLaneEnvs, kDerivState};
  rnea_derivs_aligned<false>(sm, world_accel(mv), tile_col(tile, 0), tile_col(tile, mv.nq),
                             tile_col(tile, mv.nq + mv.nv), mv.nv, S, TreeMat{}, dq, dqd, B, e, act);
}

// Forward-dynamics derivatives in one launch: qdd by the lean level-parallel
// ABA, the inverse dynamics' derivatives and M there, then
//   d qdd / d q = -M^-1 d tau / d q,  d qdd / d qd = -M^-1 d tau / d qd,  M^-1
// by the tree-sparse factorisation. The right-hand sides pass through the
// output arrays (L2); a warp solves two columns at a time in shared memory
// that the per-body state no longer needs. Latency-bound: a chain of about 60
// short phases per tile. One thread per environment with a dense Cholesky and
// its solves in global memory took 364 us for legged12 at B = 1000 (now 25)
// and 2300 us for the floating humanoid at B = 2048 (now 139).
__global__ void __launch_bounds__(512) aba_derivs_aligned_kernel(ModelView mv, int64_t B, const float* __restrict__ q,
                                                                 const float* __restrict__ qd,
                                                                 const float* __restrict__ tau, float* qdd, float* dq,
                                                                 float* dqd, float* Minv, int entries,
                                                                 int dof_depth, int state_floats) {
  FST_TILE;
  const int nv = mv.nv, W = n_warps(), w = warp_id();
  const int rows = mv.nq + 3 * nv;
  float* const state = tile + rows * kLaneEnvs;
  float* const hbase = state + (size_t)state_floats * kLaneEnvs;
  int* const lists = reinterpret_cast<int*>(hbase + entries * kLaneEnvs);  // off | dep | order | level | anc
  stage_block_rows(tile, q, mv.nq, B, e);
  stage_block_rows(tile + mv.nq * kLaneEnvs, qd, nv, B, e);
  stage_block_rows(tile + (mv.nq + nv) * kLaneEnvs, tau, nv, B, e);
  const DofLists* dl = reinterpret_cast<const DofLists*>(mv.topo + 1);
  for (int k = threadIdx.x; k < nv; k += blockDim.x) {
    cp_async4(lists + k, dl->off + k);
    cp_async4(lists + nv + k, dl->dep + k);
    cp_async4(lists + 2 * nv + k, dl->order + k);
  }
  for (int k = threadIdx.x; k <= dof_depth; k += blockDim.x) cp_async4(lists + 3 * nv + k, dl->level + k);
  int* const anc = lists + 4 * nv + 1;
  for (int k = threadIdx.x; k < entries; k += blockDim.x) cp_async4(anc + k, dl->anc + k);
  const SmemModel sm = stage_model_end(mv, smem);
  const Col cq = tile_col(tile, 0), cqd = tile_col(tile, mv.nq);
  float* const qcol = tile + (mv.nq + 2 * nv) * kLaneEnvs + lane;  // qdd
  aba_level_lean<false, true>(sm, world_accel(mv), cq, cqd, tile_col(tile, mv.nq + nv), LaneState{state, kAbaLeanBodyFloats},
                 LaneState{state + kAbaLeanBodyFloats * mv.n * kLaneEnvs, kAbaLeanSlotFloats}, qdd, B, e, act,
                 qcol);
  const TreeMat H{hbase, lists, lists + nv, anc};
  rnea_derivs_aligned<true>(sm, world_accel(mv), cq, cqd, Col{qcol, kLaneEnvs}, nv, LaneState{state, kDerivState}, H,
                            dq, dqd, B, e, act);
  __syncthreads();  // M and the right-hand sides are complete; the state is free
  tree_factor(H, lists + 2 * nv, lists + 3 * nv, dof_depth);
  // items: column c of both derivatives, then columns c and c + 1 of M^-1
  float* const x = state + (size_t)w * 2 * nv * kLaneEnvs + lane;
  const int ld = nv * kLaneEnvs;
  const int n_d = dq || dqd ? nv : 0;
  const int64_t col = B, row = (int64_t)nv * B;
  for (int it = w; it < n_d + (nv + 1) / 2; it += W) {
    const bool d = it < n_d;
    const int c0 = d ? it : 2 * (it - n_d);
    float* const p0 = d ? (dq ? dq + c0 * col + e : nullptr) : Minv + c0 * col + e;
    float* const p1 = d ? (dqd ? dqd + c0 * col + e : nullptr) : (c0 + 1 < nv ? p0 + col : nullptr);
    if (d) {
#pragma unroll 4
      for (int r = 0; r < nv; ++r) {
        x[r * kLaneEnvs] = act && p0 ? -p0[r * row] : 0.f;
        x[ld + r * kLaneEnvs] = act && p1 ? -p1[r * row] : 0.f;
      }
    } else {
      for (int r = 0; r < nv; ++r) {
        x[r * kLaneEnvs] = r == c0 ? 1.f : 0.f;
        x[ld + r * kLaneEnvs] = r == c0 + 1 ? 1.f : 0.f;
      }
    }
    tree_solve<2>(H, nv, x, ld);
    if (!act) continue;
#pragma unroll 4
    for (int r = 0; r < nv; ++r) {
      if (p0) p0[r * row] = x[r * kLaneEnvs];
      if (p1) p1[r * row] = x[ld + r * kLaneEnvs];
    }
  }
}

// The adjoint of inverse dynamics and the identification loss with its
// gradient. Bound by latency: shared memory holds one tile of the humanoid
// (172 KB) or two of the quadruped per SM (see rnea_vjp_lean_kernel). The one-thread-per-environment
// kernel ran all sweeps in series with their state in local memory and 50
// shuffles per body for the parameter gradient: humanoid, B = 4096: 70 -> 16
// us; arm, B = 8192, loss and gradient: 16.0 -> 12.0 us (the specialised
// kernel against this one).
template <int MODE>
__global__ void __launch_bounds__(512) rnea_vjp_aligned_kernel(ModelView mv, int64_t B, const float* __restrict__ q,
                                                               const float* __restrict__ qd,
                                                               const float* __restrict__ qdd, const float* tb,
                                                               float* qbar, float* qdbar, float* qddbar,
                                                               float* partial) {
  FST_TILE;
  const int nv = mv.nv, P = mv.n * 10 + (MODE == VJP_LOSS ? 1 : 0);
  stage_block_rows(tile, q, mv.nq, B, e);
  stage_block_rows(tile + mv.nq * kLaneEnvs, qd, nv, B, e);
  stage_block_rows(tile + (mv.nq + nv) * kLaneEnvs, qdd, nv, B, e);
  stage_block_rows(tile + (mv.nq + 2 * nv) * kLaneEnvs, tb, nv, B, e);
  const SmemModel sm = stage_model_end(mv, smem);
  const LaneState S{tile + (mv.nq + 3 * nv) * kLaneEnvs, kVjpState};
  float* const th = partial ? partial + (int64_t)blockIdx.x * P : nullptr;
  const VjpAligned o{qbar, qdbar, qddbar, th, 1.f};
  float loss = rnea_vjp_aligned<MODE>(sm, world_accel(mv), tile_col(tile, 0), tile_col(tile, mv.nq),
                                      tile_col(tile, mv.nq + nv), tile + (mv.nq + 2 * nv) * kLaneEnvs + lane, S, o, B,
                                      e, act);
  if (MODE == VJP_LOSS) {
    __shared__ float wsum[16];
    loss = act ? loss : 0.f;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, off);
    if (lane == 0) wsum[warp_id()] = loss;
    __syncthreads();
    if (threadIdx.x == 0) {
      float s = 0.f;
      for (int k = 0; k < n_warps(); ++k) s += wsum[k];
      th[P - 1] = s;
    }
  }
}

// The same with the lean state, blockDim.y tiles per block over one copy of
// the model: two tiles of the humanoid an SM instead of one, four of the
// quadruped instead of two. Adjoint with the parameter gradient, B = 65536:
// humanoid 320 us in one thread per environment, 161 in rnea_vjp_aligned_kernel,
// 123 here (133 before a body's own terms and its sums for theta's gradient were
// formed ahead of its level; 16384 39.1 -> 36.2); quadruped 80 -> 60. A short
// chain gains nothing (arm7 B = 16384 15.4 against 17.2), so trees of up to 8
// bodies keep the other form.
__global__ void __launch_bounds__(512) rnea_vjp_lean_kernel(ModelView mv, int64_t B, const float* __restrict__ q,
                                                            const float* __restrict__ qd,
                                                            const float* __restrict__ qdd,
                                                            const float* __restrict__ tb, float* qbar, float* qdbar,
                                                            float* qddbar, float* partial) {
  extern __shared__ float4 smem[];
  const int64_t t = (int64_t)blockIdx.x * blockDim.y + threadIdx.y;
  const int64_t e = t * kLaneEnvs + (threadIdx.x & 31);
  pdl_launch();
  stage_model_begin(mv, smem);
  pdl_wait();
  const SmemModel sm = stage_model_end(mv, smem);
  if (t * kLaneEnvs >= B) return;  // a whole tile past the end, its warps alone share its barrier
  const LaneState S{smem_tile(smem, mv.n) + (size_t)threadIdx.y * kVjpLeanState * mv.n * kLaneEnvs, kVjpLeanState};
  const VjpAligned o{qbar, qdbar, qddbar, partial ? partial + t * mv.n * 10 : nullptr, 1.f};
  rnea_vjp_lean(sm, world_accel(mv), q, qd, qdd, tb, S, o, B, e, e < B);
}

// The ABA adjoint in one launch: lambda = M^-1 qddbar by the lean
// level-parallel ABA at rest and without gravity, then minus the adjoint of
// inverse dynamics at (q, qd, qdd) for the cotangent lambda, in body axes (see
// rnea_vjp_aligned). Quadruped, B = 5001: 17.0 us (19.9 in root axes), the
// specialised one-thread-per-environment kernel 41.9; humanoid, 65536: 288.
__global__ void __launch_bounds__(512) aba_vjp_aligned_kernel(ModelView mv, int64_t B, const float* __restrict__ q,
                                                              const float* __restrict__ qd,
                                                              const float* __restrict__ qdd,
                                                              const float* __restrict__ qddbar, float* qbar,
                                                              float* qdbar, float* taubar, float* partial) {
  FST_TILE;
  const int nv = mv.nv;
  // rows: q | qd | qdd | qddbar | lambda | one row of zeros
  stage_block_rows(tile, q, mv.nq, B, e);
  stage_block_rows(tile + mv.nq * kLaneEnvs, qd, nv, B, e);
  stage_block_rows(tile + (mv.nq + nv) * kLaneEnvs, qdd, nv, B, e);
  stage_block_rows(tile + (mv.nq + 2 * nv) * kLaneEnvs, qddbar, nv, B, e);
  const int rows = mv.nq + 4 * nv + 1;
  float* const zero = tile + (rows - 1) * kLaneEnvs + lane;
  if (threadIdx.x < 32) *zero = 0.f;
  const SmemModel sm = stage_model_end(mv, smem);
  float* const state = tile + rows * kLaneEnvs;
  float* const lam = tile + (mv.nq + 3 * nv) * kLaneEnvs + lane;
  const Col cq = tile_col(tile, 0);
  aba_level_lean<false, true>(sm, sv_zero(), cq, Col{zero, 0}, tile_col(tile, mv.nq + 2 * nv), LaneState{state, kAbaLeanBodyFloats},
                 LaneState{state + kAbaLeanBodyFloats * mv.n * kLaneEnvs, kAbaLeanSlotFloats}, taubar, B, e, act,
                 lam);
  const VjpAligned o{qbar, qdbar, nullptr, partial ? partial + (int64_t)blockIdx.x * mv.n * 10 : nullptr, -1.f};
  rnea_vjp_aligned<VJP_GIVEN, true>(sm, world_accel(mv), cq, tile_col(tile, mv.nq), tile_col(tile, mv.nq + nv), lam,
                              LaneState{state, kVjpState}, o, B, e, act);
}

// Bound by the latency of two sweeps over the levels (fixed humanoid, B = 3000:
// 46 -> 9 us; the general kernel staged 12 cotangent rows a body and swept the
// bodies one by one), three tiles of the humanoid
// per SM (floating humanoid, B = 65536: 305 -> 57 us, 75 MB read).
__global__ void __launch_bounds__(256) fk_vjp_tile_kernel(ModelView mv, int64_t B, const float* __restrict__ q,
                                                          const float* __restrict__ pbar, float* __restrict__ qbar) {
  FST_TILE;
  stage_block_rows(tile, q, mv.nq, B, e);
  const SmemModel sm = stage_model_end(mv, smem);
  fk_vjp_tile(sm, tile_col(tile, 0), pbar, LaneState{tile + mv.nq * kLaneEnvs, kFkVjpState}, qbar, B, e, act);
}

// The store variant's forward: RNEA that also leaves its state on the tape.
__global__ void __launch_bounds__(256) rnea_store_tile_kernel(ModelView mv, int64_t B, const float* __restrict__ q,
                                                              const float* __restrict__ qd,
                                                              const float* __restrict__ qdd, float* __restrict__ tau,
                                                              float* tape) {
  FST_TILE;
  stage_block_rows(tile, q, mv.nq, B, e);
  stage_block_rows(tile + mv.nq * kLaneEnvs, qd, mv.nv, B, e);
  stage_block_rows(tile + (mv.nq + mv.nv) * kLaneEnvs, qdd, mv.nv, B, e);
  const SmemModel sm = stage_model_end(mv, smem);
  rnea_level(sm, world_accel(mv), tile_col(tile, 0), tile_col(tile, mv.nq), tile_col(tile, mv.nq + mv.nv),
             LaneState{tile + (mv.nq + 2 * mv.nv) * kLaneEnvs, kRneaState}, tau, B, e, act, nullptr, tape);
}

// ---- fused evaluation ----------------------------------------------------------
// blockIdx.y picks the operator of a block, blockIdx.x its tile; the bodies
// are those of the per-operator kernels, so the results are theirs bit for
// bit. Blocks of the heaviest operator come first. EXT (a kernel of its own,
// so that the plain one keeps its registers): the RNEA adjoint beside tau, and
// M and J in the packed layouts.
// Bound by the ABA blocks' latency at B = 4096 (quadruped, five operators: 13.3
// us; the specialised fused kernel that the default took before 31.3, its
// roles' straight-line code refetched by every SM) and by shared memory, two
// to four tiles an SM, at larger batches (humanoid, B = 16384: 164 -> 72 us).
template <bool EXT, bool LEAN>
__global__ void __launch_bounds__(256) eval_tile_kernel(ModelView mv, int64_t B, EvalArgs a) {
  FST_TILE;
  const int role = a.roles[blockIdx.y], nv = mv.nv;
  const bool vjp = EXT && role == ROLE_RNEA && (a.rnea_flags & EVAL_RNEA_VJP);
  stage_block_rows(tile, a.q, mv.nq, B, e);
  int rows = mv.nq;
  if (role == ROLE_RNEA || role == ROLE_ABA) {
    stage_block_rows(tile + rows * kLaneEnvs, a.qd, nv, B, e);
    stage_block_rows(tile + (rows + nv) * kLaneEnvs, role == ROLE_ABA ? a.tau : a.qdd, nv, B, e);
    if (vjp && !(a.rnea_flags & EVAL_TBAR_IS_TAU))
      stage_block_rows(tile + (rows + 2 * nv) * kLaneEnvs, a.tau_bar, nv, B, e);
    rows += (vjp ? 3 : 2) * nv;
  }
  const SmemModel sm = stage_model_end(mv, smem);
  float* const state = tile + rows * kLaneEnvs;
  const Col cq = tile_col(tile, 0), c1 = tile_col(tile, mv.nq), c2 = tile_col(tile, mv.nq + nv);
  auto X_of = [&](const BodyC& c, const BodyI& bi) { return joint_X(c, bi, cq); };
  const LaneState R{state + kCrbaLeanBodyFloats * mv.n * kLaneEnvs, kCrbaLeanSlotFloats};
  switch (role) {
    case ROLE_ABA:
      aba_level_lean<true, !LEAN>(sm, world_accel(mv), cq, c1, c2, LaneState{state, kAbaLeanBodyFloats},
                     LaneState{state + kAbaLeanBodyFloats * mv.n * kLaneEnvs, kAbaLeanSlotFloats}, a.qdd_out, B,
                     e, act);
      break;
    case ROLE_CRBA:
      if (EXT && a.packed)
        crba_level_lean<true>(sm, X_of, nv, LaneState{state, kCrbaLeanBodyFloats}, R, a.M, B, e, act);
      else
        crba_level_lean(sm, X_of, nv, LaneState{state, kCrbaLeanBodyFloats}, R, a.M, B, e, act);
      break;
    case ROLE_RNEA:
      if (!vjp || a.tau_out || (a.rnea_flags & EVAL_TBAR_IS_TAU))
        rnea_level<LEAN, LEAN && !EXT, true>(
            sm, world_accel(mv), cq, c1, c2, LaneState{state, LEAN ? kRneaLeanFloats : kRneaState}, a.tau_out, B, e, act,
            vjp && (a.rnea_flags & EVAL_TBAR_IS_TAU) ? tile + (mv.nq + 2 * nv) * kLaneEnvs + lane : nullptr);
      if (vjp)  // rnea_level ends with a barrier: the cotangent is complete and the state free
        rnea_vjp_aligned<VJP_GIVEN>(sm, world_accel(mv), cq, c1, c2, tile + (mv.nq + 2 * nv) * kLaneEnvs + lane,
                                    LaneState{state, kVjpState}, VjpAligned{a.qbar, a.qdbar, a.qddbar, nullptr, 1.f},
                                    B, e, act);
      break;
    default:
      kin_level<!LEAN>(sm, cq, nv, a.links, LaneState{state, kFkState}, a.poses, a.J, B, e, act,
                EXT && a.packed ? &a.pj : nullptr);
      break;
  }
}

size_t floats32(size_t f) { return f * kLaneEnvs * sizeof(float); }

// Per-body state that also holds the lean ABA's (run before it in the same space).
size_t state_with_aba(int n, int slots, int per_body) {
  const size_t a = (size_t)kAbaLeanBodyFloats * n + kAbaLeanSlotFloats * slots, b = (size_t)per_body * n;
  return a > b ? a : b;
}

// Threads per block: one warp per two or three bodies while the tiles fill the
// SMs, more when they do not.
int aligned_block(int n, int64_t tiles) {
  if (n >= 16) return tiles <= 2 * kSms ? 512 : 256;
  return tiles <= 2 * kSms ? 256 : 128;
}

}  // namespace

size_t rnea_derivs_aligned_smem(const ModelView& mv) {
  return smem_bytes(mv.n) + floats32((size_t)mv.nq + 2 * mv.nv + (size_t)kDerivState * mv.n);
}

size_t rnea_vjp_aligned_smem(const ModelView& mv) {
  return smem_bytes(mv.n) + floats32((size_t)mv.nq + 3 * mv.nv + (size_t)kVjpState * mv.n);
}

size_t aba_vjp_aligned_smem(const ModelView& mv, int slots) {
  return smem_bytes(mv.n) + floats32((size_t)mv.nq + 4 * mv.nv + 1 + state_with_aba(mv.n, slots, kVjpState));
}

// The forward-dynamics derivatives' solve phase keeps two columns per warp in
// the state's space: the block is as large as that allows (0: not one warp).
// 16 warps while no SM has a second tile to run (legged12 B = 1000 30.3 -> 26.8
// us, humanoid29 B = 2048 180 -> 146).
static int aba_derivs_threads(const ModelView& mv, int slots, int64_t tiles) {
  const size_t st = state_with_aba(mv.n, slots, kDerivState);
  int t = tiles <= kSms ? 512 : aligned_block(mv.n, tiles);
  while (t >= 32 && (size_t)(t / 32) * 2 * mv.nv > st) t /= 2;
  return t >= 32 ? t : 0;
}

size_t aba_derivs_aligned_smem(const ModelView& mv, int slots, int entries) {
  if (!aba_derivs_threads(mv, slots, 1)) return kLevelSmemLimit + 1;
  return smem_bytes(mv.n) +
         floats32((size_t)mv.nq + 3 * mv.nv + state_with_aba(mv.n, slots, kDerivState) + entries) +
         ((size_t)4 * mv.nv + 1 + entries) * sizeof(int);
}

size_t eval_tile_smem(const ModelView& mv, int role, bool vjp, bool lean, int slots) {
  size_t f = mv.nq;
  if (role == ROLE_ABA)
    f += 2 * (size_t)mv.nv + (size_t)kAbaLeanBodyFloats * mv.n + (size_t)kAbaLeanSlotFloats * slots;
  else if (role == ROLE_CRBA)
    f += (size_t)kCrbaLeanBodyFloats * mv.n + (size_t)kCrbaLeanSlotFloats * slots;
  else if (role == ROLE_RNEA)
    f += (vjp ? 3 : 2) * (size_t)mv.nv + (size_t)(vjp ? kVjpState : lean ? kRneaLeanFloats : kRneaState) * mv.n;
  else
    f += (size_t)kFkState * mv.n;
  return smem_bytes(mv.n) + floats32(f);
}

size_t fk_vjp_tile_smem(const ModelView& mv) {
  return smem_bytes(mv.n) + floats32((size_t)mv.nq + (size_t)kFkVjpState * mv.n);
}

cudaError_t launch_fk_vjp_tile(const ModelView& mv, int64_t B, const float* q, const float* pbar, float* qbar,
                               int block, cudaStream_t s) {
  const size_t sh = fk_vjp_tile_smem(mv);
  prepare(fk_vjp_tile_kernel, sh);
  return launch_pdl(fk_vjp_tile_kernel, grid_for(B, kLaneEnvs), block, sh, s, mv, B, q, pbar, qbar);
}

cudaError_t launch_rnea_store_tile(const ModelView& mv, int64_t B, const float* q, const float* qd, const float* qdd,
                                   float* tau, float* tape, int block, cudaStream_t s) {
  const size_t sh = level_smem_needed(mv, LEVEL_RNEA);
  prepare(rnea_store_tile_kernel, sh);
  return launch_pdl(rnea_store_tile_kernel, grid_for(B, kLaneEnvs), block, sh, s, mv, B, q, qd, qdd, tau, tape);
}

cudaError_t launch_eval_tile(const ModelView& mv, int64_t B, const EvalArgs& a, bool lean, size_t smem, int block,
                             cudaStream_t s) {
  const dim3 grid(grid_for(B, kLaneEnvs), a.n_roles);
  auto go = [&](auto* k) {
    prepare(k, smem);
    return launch_pdl(k, grid, block, smem, s, mv, B, a);
  };
  if (a.rnea_flags || a.packed) return lean ? go(eval_tile_kernel<true, true>) : go(eval_tile_kernel<true, false>);
  return lean ? go(eval_tile_kernel<false, true>) : go(eval_tile_kernel<false, false>);
}

cudaError_t launch_rnea_derivs_aligned(const ModelView& mv, int64_t B, const float* q, const float* qd,
                                       const float* qdd, float* dq, float* dqd, cudaStream_t s) {
  const size_t sh = rnea_derivs_aligned_smem(mv);
  const unsigned tiles = grid_for(B, kLaneEnvs);
  auto go = [&](auto* k, int threads) {
    prepare(k, sh);
    return launch_pdl(k, tiles, threads, sh, s, mv, B, q, qd, qdd, dq, dqd);
  };
  // 24 warps where an SM has one tile and the tree work for them (humanoid29 B =
  // 2048: 21.0 -> 19.7 us, legged18 B = 2700 11.0 -> 10.3).
  if (mv.n > 16 && tiles <= kSms) return go(rnea_derivs_aligned_kernel<768>, 768);
  return go(rnea_derivs_aligned_kernel<512>, aligned_block(mv.n, tiles));
}

cudaError_t launch_aba_derivs_aligned(const ModelView& mv, int64_t B, const float* q, const float* qd,
                                      const float* tau, float* qdd, float* dq, float* dqd, float* Minv, int slots,
                                      int entries, int dof_depth, cudaStream_t s) {
  const size_t sh = aba_derivs_aligned_smem(mv, slots, entries);
  const unsigned tiles = grid_for(B, kLaneEnvs);
  prepare(aba_derivs_aligned_kernel, sh);
  return launch_pdl(aba_derivs_aligned_kernel, tiles, aba_derivs_threads(mv, slots, tiles), sh, s, mv, B, q, qd,
                    tau, qdd, dq, dqd, Minv, entries, dof_depth, (int)state_with_aba(mv.n, slots, kDerivState));
}

cudaError_t launch_rnea_vjp_aligned(const ModelView& mv, int64_t B, const float* q, const float* qd, const float* qdd,
                                    const float* tbar, float* qbar, float* qdbar, float* qddbar, float* thbar,
                                    float* scratch, cudaStream_t s) {
  const size_t sh = rnea_vjp_aligned_smem(mv);
  const unsigned tiles = grid_for(B, kLaneEnvs);
  float* const partial = thbar ? scratch : nullptr;
  // Where more tiles wait than the SMs take, the lean state, in as many tiles
  // per block as double the tiles per SM.
  const size_t model = smem_bytes(mv.n), lean = floats32((size_t)kVjpLeanState * mv.n);
  const int T = model + 2 * lean <= kLevelSmemLimit && 2 * (model + lean + 1024) > kLevelSmemLimit ? 2 : 1;
  cudaError_t err;
  if (tiles > 2 * kSms && mv.n > 8) {
    const int W = mv.n > 16 ? 8 : 4;
    prepare(rnea_vjp_lean_kernel, model + T * lean);
    err = launch_pdl(rnea_vjp_lean_kernel, (tiles + T - 1) / T, dim3(32, T, W), model + T * lean, s, mv, B, q, qd, qdd,
                     tbar, qbar, qdbar, qddbar, partial);
  } else {
    prepare(rnea_vjp_aligned_kernel<VJP_GIVEN>, sh);
    err = launch_pdl(rnea_vjp_aligned_kernel<VJP_GIVEN>, tiles, aligned_block(mv.n, tiles), sh, s, mv, B, q, qd,
                     qdd, tbar, qbar, qdbar, qddbar, partial);
  }
  if (err == cudaSuccess && thbar) err = launch_partial_reduce(scratch, (int)tiles, mv.n * 10, thbar, s);
  return err;
}

cudaError_t launch_loss_grad_aligned(const ModelView& mv, int64_t B, const float* q, const float* qd, const float* qdd,
                                     const float* tau_meas, float* loss_theta, float* qbar, float* qdbar,
                                     float* scratch, cudaStream_t s) {
  const size_t sh = rnea_vjp_aligned_smem(mv);
  const unsigned tiles = grid_for(B, kLaneEnvs);
  prepare(rnea_vjp_aligned_kernel<VJP_LOSS>, sh);
  cudaError_t err = launch_pdl(rnea_vjp_aligned_kernel<VJP_LOSS>, tiles, aligned_block(mv.n, tiles), sh, s, mv,
                               B, q, qd, qdd, tau_meas, qbar, qdbar, nullptr, scratch);
  if (err == cudaSuccess) err = launch_partial_reduce(scratch, (int)tiles, mv.n * 10 + 1, loss_theta, s);
  return err;
}

cudaError_t launch_aba_vjp_aligned(const ModelView& mv, int64_t B, const float* q, const float* qd, const float* qdd,
                                   const float* qddbar, float* qbar, float* qdbar, float* taubar, float* thbar,
                                   float* scratch, int slots, cudaStream_t s) {
  const size_t sh = aba_vjp_aligned_smem(mv, slots);
  const unsigned tiles = grid_for(B, kLaneEnvs);
  prepare(aba_vjp_aligned_kernel, sh);
  cudaError_t err = launch_pdl(aba_vjp_aligned_kernel, tiles, aligned_block(mv.n, tiles), sh, s, mv, B, q, qd,
                               qdd, qddbar, qbar, qdbar, taubar, thbar ? scratch : nullptr);
  if (err == cudaSuccess && thbar) err = launch_partial_reduce(scratch, (int)tiles, mv.n * 10, thbar, s);
  return err;
}

}  // namespace fst
