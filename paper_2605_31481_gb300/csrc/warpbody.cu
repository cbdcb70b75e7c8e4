// Kernels of warpbody.cuh: one tile of 32 environments per block, one warp
// per body.
//
// Bound by the chain of levels at 3 to 4 cycles an instruction of one warp;
// registers hold one or two tiles an SM, so the tile kernels of aligned.cu take
// over once a third tile waits. ABA adjoint, B = 4096, against those: arm 17.0 ->
// 11.9 us, quadruped 15.2 -> 14.2 (15.8 with M^-1 and the sweep in root axes).
#include "launch.h"
#include "warpbody.cuh"

namespace fst {
namespace {

#define FST_WB_TILE                                         \
  extern __shared__ float smem_f[];                         \
  const int lane = threadIdx.x & 31;                        \
  const int64_t e = (int64_t)blockIdx.x * kLaneEnvs + lane; \
  const bool act = e < B;                                   \
  const int64_t ec = act ? e : B - 1;                       \
  const Me me(t);                                           \
  (void)ec;                                                 \
  pdl_launch();                                             \
  pdl_wait()

template <int T, int MINB, int MODE>
__global__ void __launch_bounds__(T, MINB) wb_vjp_kernel(const __grid_constant__ WarpTree t, ModelView mv, int64_t B,
                                                         const float* __restrict__ q, const float* __restrict__ qd,
                                                         const float* __restrict__ qdd, const float* __restrict__ tb,
                                                         float* qbar, float* qdbar, float* qddbar, float* partial) {
  FST_WB_TILE;
  const int P = mv.n * 10 + (MODE == VJP_LOSS ? 1 : 0);
  float* const th = partial ? partial + (int64_t)blockIdx.x * P : nullptr;
  float loss = vjp_warp<MODE>(me, t, mv, q, qd, qdd, own_v(me, tb, B, ec), LaneState{smem_f, kWbVjpFloats},
                              VjpAligned{qbar, qdbar, qddbar, th, 1.f}, B, e, act);
  if (MODE == VJP_LOSS) {  // the tile's loss: lanes, then warps in order
    __shared__ float wsum[32];
    loss = act ? loss : 0.f;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, off);
    if (lane == 0) wsum[threadIdx.x >> 5] = loss;
    __syncthreads();
    if (threadIdx.x == 0) {
      float s = 0.f;
      for (int k = 0; k < t.n; ++k) s += wsum[k];
      th[P - 1] = s;
    }
  }
}

// lambda = M^-1 qddbar at rest, then minus the adjoint of inverse dynamics for it.
template <int T, int MINB>
__global__ void __launch_bounds__(T, MINB) wb_aba_vjp_kernel(const __grid_constant__ WarpTree t, ModelView mv,
                                                             int64_t B, const float* __restrict__ q,
                                                             const float* __restrict__ qd,
                                                             const float* __restrict__ qdd,
                                                             const float* __restrict__ qddbar, float* qbar,
                                                             float* qdbar, float* taubar, float* partial) {
  FST_WB_TILE;
  const LaneState S{smem_f, kWbVjpFloats};
  const Own lam = minv_warp(me, t, mv, q, qddbar, S, taubar, B, e, act);
  __syncthreads();  // the last level has read its parents' accelerations
  float* const th = partial ? partial + (int64_t)blockIdx.x * mv.n * 10 : nullptr;
  vjp_warp<VJP_GIVEN, true>(me, t, mv, q, qd, qdd, lam, S, VjpAligned{qbar, qdbar, nullptr, th, -1.f}, B, e, act);
}

size_t wb_smem(int n, int floats) { return (size_t)n * floats * kLaneEnvs * sizeof(float); }

// Instantiates a kernel for the smallest block that holds a warp per body;
// two blocks per SM keep the registers to 128 (n <= 8), 80 (n <= 12) and, with
// spills that cost more than the second block brings, not at all above.
#define FST_WB_GO(KERNEL, ...)                                        \
  do {                                                                \
    const size_t sh_ = wb_smem(t.n, kWbVjpFloats);                    \
    auto go_ = [&](auto* k_) {                                        \
      prepare(k_, sh_);                                               \
      return launch_pdl(k_, grid_for(B, kLaneEnvs), 32 * t.n, sh_, s, t, mv, B, __VA_ARGS__); \
    };                                                                \
    if (t.n <= 8) return go_(KERNEL(256, 2));                         \
    if (t.n <= 12) return go_(KERNEL(384, 2));                        \
    return go_(KERNEL(512, 1));                                       \
  } while (0)

cudaError_t go_vjp(const WarpTree& t, const ModelView& mv, int64_t B, const float* q, const float* qd,
                   const float* qdd, const float* tbar, float* qbar, float* qdbar, float* qddbar, float* partial,
                   cudaStream_t s) {
#define K(T, M) (wb_vjp_kernel<T, M, VJP_GIVEN>)
  FST_WB_GO(K, q, qd, qdd, tbar, qbar, qdbar, qddbar, partial);
#undef K
}
cudaError_t go_loss(const WarpTree& t, const ModelView& mv, int64_t B, const float* q, const float* qd,
                    const float* qdd, const float* tau_meas, float* qbar, float* qdbar, float* partial,
                    cudaStream_t s) {
#define K(T, M) (wb_vjp_kernel<T, M, VJP_LOSS>)
  FST_WB_GO(K, q, qd, qdd, tau_meas, qbar, qdbar, (float*)nullptr, partial);
#undef K
}
cudaError_t go_aba_vjp(const WarpTree& t, const ModelView& mv, int64_t B, const float* q, const float* qd,
                       const float* qdd, const float* qddbar, float* qbar, float* qdbar, float* taubar,
                       float* partial, cudaStream_t s) {
#define K(T, M) (wb_aba_vjp_kernel<T, M>)
  FST_WB_GO(K, q, qd, qdd, qddbar, qbar, qdbar, taubar, partial);
#undef K
}

}  // namespace

cudaError_t launch_wb_rnea_vjp(const WarpTree& t, const ModelView& mv, int64_t B, const float* q, const float* qd,
                               const float* qdd, const float* tbar, float* qbar, float* qdbar, float* qddbar,
                               float* thbar, float* scratch, cudaStream_t s) {
  cudaError_t err = go_vjp(t, mv, B, q, qd, qdd, tbar, qbar, qdbar, qddbar, thbar ? scratch : nullptr, s);
  if (err == cudaSuccess && thbar) err = launch_partial_reduce(scratch, (int)grid_for(B, kLaneEnvs), mv.n * 10, thbar, s);
  return err;
}

cudaError_t launch_wb_loss_grad(const WarpTree& t, const ModelView& mv, int64_t B, const float* q, const float* qd,
                                const float* qdd, const float* tau_meas, float* loss_theta, float* qbar, float* qdbar,
                                float* scratch, cudaStream_t s) {
  cudaError_t err = go_loss(t, mv, B, q, qd, qdd, tau_meas, qbar, qdbar, scratch, s);
  if (err == cudaSuccess)
    err = launch_partial_reduce(scratch, (int)grid_for(B, kLaneEnvs), mv.n * 10 + 1, loss_theta, s);
  return err;
}

cudaError_t launch_wb_aba_vjp(const WarpTree& t, const ModelView& mv, int64_t B, const float* q, const float* qd,
                              const float* qdd, const float* qddbar, float* qbar, float* qdbar, float* taubar,
                              float* thbar, float* scratch, cudaStream_t s) {
  cudaError_t err = go_aba_vjp(t, mv, B, q, qd, qdd, qddbar, qbar, qdbar, taubar, thbar ? scratch : nullptr, s);
  if (err == cudaSuccess && thbar) err = launch_partial_reduce(scratch, (int)grid_for(B, kLaneEnvs), mv.n * 10, thbar, s);
  return err;
}

}  // namespace fst
