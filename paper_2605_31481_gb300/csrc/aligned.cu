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
  const bool act = e < B

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
__global__ void __launch_bounds__(512) rnea_derivs_aligned_kernel(ModelView mv, int64_t B, const float* __restrict__ q,
                                                                  const float* __restrict__ qd,
                                                                  const float* __restrict__ qdd,
                                                                  float* __restrict__ dq, float* __restrict__ dqd) {
  FST_TILE;
  stage_block_rows(tile, q, mv.nq, B, e);
  stage_block_rows(tile + mv.nq * kLaneEnvs, qd, mv.nv, B, e);
  stage_block_rows(tile + (mv.nq + mv.nv) * kLaneEnvs, qdd, mv.nv, B, e);
  const SmemModel sm = stage_model(mv, smem);
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
// its solves in global memory took 364 us for legged12 at B = 1000 (now 31)
// and 2300 us for the floating humanoid at B = 2048 (now 147).
__global__ void __launch_bounds__(512) aba_derivs_aligned_kernel(ModelView mv, int64_t B, const float* __restrict__ q,
                                                                 const float* __restrict__ qd,
                                                                 const float* __restrict__ tau, float* qdd, float* dq,
                                                                 float* dqd, float* Minv, int maxw, int entries,
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
  const SmemModel sm = stage_model(mv, smem);
  const Col cq = tile_col(tile, 0), cqd = tile_col(tile, mv.nq);
  float* const qcol = tile + (mv.nq + 2 * nv) * kLaneEnvs + lane;  // qdd
  aba_level_lean(sm, world_accel(mv), cq, cqd, tile_col(tile, mv.nq + nv), LaneState{state, kAbaLeanBodyFloats},
                 LaneState{state + kAbaLeanBodyFloats * mv.n * kLaneEnvs, kAbaLeanRingFloats}, maxw, qdd, B, e, act,
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

size_t floats32(size_t f) { return f * kLaneEnvs * sizeof(float); }

// Per-body state that also holds the lean ABA's (run before it in the same space).
size_t state_with_aba(int n, int maxw, int per_body) {
  const size_t a = (size_t)kAbaLeanBodyFloats * n + 2 * kAbaLeanRingFloats * maxw, b = (size_t)per_body * n;
  return a > b ? a : b;
}

// Threads per block: a caller's setting, else one warp per two or three
// bodies while the tiles fill the SMs, more when they do not.
int aligned_block(int set, int n, int64_t tiles) {
  if (set) return set;
  if (n >= 16) return tiles <= 304 ? 512 : 256;
  return tiles <= 304 ? 256 : 128;
}

}  // namespace

size_t rnea_derivs_aligned_smem(const ModelView& mv) {
  return smem_bytes(mv.n) + floats32((size_t)mv.nq + 2 * mv.nv + (size_t)kDerivState * mv.n);
}

// The forward-dynamics derivatives' solve phase keeps two columns per warp in
// the state's space: the block is as large as that allows (0: not one warp).
static int aba_derivs_threads(const ModelView& mv, int maxw, int set, int64_t tiles) {
  const size_t st = state_with_aba(mv.n, maxw, kDerivState);
  int t = aligned_block(set, mv.n, tiles);
  while (t >= 32 && (size_t)(t / 32) * 2 * mv.nv > st) t /= 2;
  return t >= 32 ? t : 0;
}

size_t aba_derivs_aligned_smem(const ModelView& mv, int maxw, int entries) {
  if (!aba_derivs_threads(mv, maxw, 32, 1)) return kLevelSmemLimit + 1;
  return smem_bytes(mv.n) +
         floats32((size_t)mv.nq + 3 * mv.nv + state_with_aba(mv.n, maxw, kDerivState) + entries) +
         ((size_t)4 * mv.nv + 1 + entries) * sizeof(int);
}

cudaError_t launch_rnea_derivs_aligned(const ModelView& mv, int64_t B, const float* q, const float* qd,
                                       const float* qdd, float* dq, float* dqd, int block, cudaStream_t s) {
  const size_t sh = rnea_derivs_aligned_smem(mv);
  const unsigned tiles = grid_for(B, kLaneEnvs);
  prepare(rnea_derivs_aligned_kernel, sh);
  rnea_derivs_aligned_kernel<<<tiles, aligned_block(block, mv.n, tiles), sh, s>>>(mv, B, q, qd, qdd, dq, dqd);
  return cudaGetLastError();
}

cudaError_t launch_aba_derivs_aligned(const ModelView& mv, int64_t B, const float* q, const float* qd,
                                      const float* tau, float* qdd, float* dq, float* dqd, float* Minv, int maxw,
                                      int entries, int dof_depth, int block, cudaStream_t s) {
  const size_t sh = aba_derivs_aligned_smem(mv, maxw, entries);
  const unsigned tiles = grid_for(B, kLaneEnvs);
  prepare(aba_derivs_aligned_kernel, sh);
  aba_derivs_aligned_kernel<<<tiles, aba_derivs_threads(mv, maxw, block, tiles), sh, s>>>(
      mv, B, q, qd, tau, qdd, dq, dqd, Minv, maxw, entries, dof_depth, (int)state_with_aba(mv.n, maxw, kDerivState));
  return cudaGetLastError();
}

}  // namespace fst
