// Level-parallel operator bodies: one block serves 32 environments (one per
// lane) and its W warps split the bodies of each tree level between them.
//
// This is the paper's level-parallel propagation (Sec. 3.3: all bodies of
// one depth are independent given their parents) mapped onto warps instead
// of batched tensor ops: warp w handles bodies level_body[k] with
// k = level_start[l] + w, + W, ... and the block synchronises once per level.
// The per-body sweep state lives in shared memory as [body][field][lane]
// (lane-contiguous, so every access is conflict-free), because a body's
// parent or children may belong to another warp. Leaf-to-root passes are
// gathers, not scatters: each body leaves its contribution to the parent in
// its own slots and the parent adds its children's after the level barrier,
// so no atomics are needed (the paper keeps these passes sequential for the
// same reason, Sec. 3.3). A body adds its children's from the last to the
// first, the order in which a single thread's sweep from the last body to the
// first meets them: the two forms then round alike, and a call gives the same
// bits in either.
//
// Every warp runs the same loops with the same trip counts, so all warps
// meet every __syncthreads(); padding lanes (environments past B) compute on
// zeros and store nothing to global memory.
#pragma once

#include "ops.cuh"

namespace fst {

constexpr int kLaneEnvs = 32;

struct LaneState {
  float* base;  // [body][F][32]
  int F;
  __device__ __forceinline__ float* at(int i, int f) const {
    return base + ((i * F + f) << 5) + (threadIdx.x & 31);
  }
  __device__ __forceinline__ SV sv(int i, int f) const {
    const float* p = at(i, f);
    return SV{f3{p[0], p[32], p[64]}, f3{p[96], p[128], p[160]}};
  }
  __device__ __forceinline__ void put(int i, int f, SV v) const {
    float* p = at(i, f);
    p[0] = v.w.x;
    p[32] = v.w.y;
    p[64] = v.w.z;
    p[96] = v.v.x;
    p[128] = v.v.y;
    p[160] = v.v.z;
  }
  __device__ __forceinline__ void get_n(int i, int f, float* out, int n) const {
    const float* p = at(i, f);
    for (int k = 0; k < n; ++k) out[k] = p[k << 5];
  }
  __device__ __forceinline__ void put_n(int i, int f, const float* in, int n) const {
    float* p = at(i, f);
    for (int k = 0; k < n; ++k) p[k << 5] = in[k];
  }
  __device__ __forceinline__ Xf X(int i, int f) const {
    Xf x;
    const float* p = at(i, f);
#pragma unroll
    for (int k = 0; k < 9; ++k) x.R[k] = p[k << 5];
#pragma unroll
    for (int k = 0; k < 3; ++k) x.t[k] = p[(9 + k) << 5];
    return x;
  }
  __device__ __forceinline__ void putX(int i, int f, const Xf& x) const {
    float* p = at(i, f);
#pragma unroll
    for (int k = 0; k < 9; ++k) p[k << 5] = x.R[k];
#pragma unroll
    for (int k = 0; k < 3; ++k) p[(9 + k) << 5] = x.t[k];
  }
  __device__ __forceinline__ Sym6 sym(int i, int f) const {
    Sym6 s;
    const float* p = at(i, f);
#pragma unroll
    for (int k = 0; k < 6; ++k) s.A[k] = p[k << 5];
#pragma unroll
    for (int k = 0; k < 9; ++k) s.Bk[k] = p[(6 + k) << 5];
#pragma unroll
    for (int k = 0; k < 6; ++k) s.C[k] = p[(15 + k) << 5];
    return s;
  }
  __device__ __forceinline__ void putsym(int i, int f, const Sym6& s) const {
    float* p = at(i, f);
#pragma unroll
    for (int k = 0; k < 6; ++k) p[k << 5] = s.A[k];
#pragma unroll
    for (int k = 0; k < 9; ++k) p[(6 + k) << 5] = s.Bk[k];
#pragma unroll
    for (int k = 0; k < 6; ++k) p[(15 + k) << 5] = s.C[k];
  }
  __device__ __forceinline__ In10 in10(int i, int f) const {
    float t[10];
    get_n(i, f, t, 10);
    return in_load(t);
  }
  __device__ __forceinline__ void putin(int i, int f, const In10& I) const {
    const float t[10] = {I.m, I.h.x, I.h.y, I.h.z, I.I[0], I.I[1], I.I[2], I.I[3], I.I[4], I.I[5]};
    put_n(i, f, t, 10);
  }
};

// floats of per-body state per environment
constexpr int kFkState = kFkStateFloats;
constexpr int kRneaState = kRneaStateFloats;   // v 6 | a 6 | f 6 | X 12
constexpr int kCrbaState = kCrbaStateFloats;   // X 12 | Ic 10 | contribution 10
constexpr int kAbaState = kAbaStateFloats;    // X 12 | va 6 | c 6 | IA 21 | pA 6 | U 6 | invD | u

// Warps of one tile of 32 environments (lane = threadIdx.x & 31). A 1-D
// block of 32 W threads is one tile of W warps. A 3-D block (32, T, W) holds
// T tiles (threadIdx.y) of W warps (threadIdx.z) each; its hardware warp k
// belongs to tile k mod T, so each tile's first warp (the one that owns the
// first body of every level, the busiest) sits on its own SM sub-partition.
__device__ __forceinline__ int warp_id() { return (threadIdx.x >> 5) + (blockDim.x >> 5) * threadIdx.z; }
__device__ __forceinline__ int n_warps() { return (blockDim.x >> 5) * blockDim.z; }

// Stages `rows` rows of this tile's 32 environments (zeros past B);
// call from every thread, then cp_async_wait_all() and __syncthreads().
__device__ __forceinline__ void stage_block_rows(float* tile, const float* __restrict__ src, int rows, int64_t B,
                                                 int64_t e) {
  const int W = n_warps(), w = warp_id(), lane = threadIdx.x & 31;
  for (int r = w; r < rows; r += W) {
    float* d = tile + (r << 5) + lane;
    if (e < B)
      cp_async4(d, src + (int64_t)r * B + e);
    else
      *d = 0.f;
  }
}

// Loop over the bodies of level l that belong to this warp (every W-th one,
// starting at the warp's index). With a run-time topology this is a strided
// loop; with a compile-time one it is unrolled over the whole level with a
// cheap round-robin ownership test, so each body's constants fold into its
// code and each warp executes only its own bodies.
#ifdef FST_FIXED_TOPOLOGY
#define FST_FOR_MY_BODIES(tp, l, k)                                                          \
  _Pragma("unroll") for (int k = (tp).level_begin(l), own_ = 0; k < (tp).level_begin((l) + 1); \
                         ++k, own_ = (own_ + 1 == W ? 0 : own_ + 1)) if (own_ == w)
#else
#define FST_FOR_MY_BODIES(tp, l, k) for (int k = (tp).level_begin(l) + w; k < (tp).level_begin((l) + 1); k += W)
#endif

// A pass over the levels, root to leaf or (UP) leaf to root, with a barrier
// after each: dep(o) with o = loc(i) for each body i, where loc reads only what
// is known before the pass. With AHEAD body k of the level order is warp k mod
// W's, so that the bodies of neighbouring levels are different warps', and a warp
// whose level has not come yet does the loc of its next body meanwhile: what is
// left on the chain of levels is dep. Without it each level starts at warp 0.
// A tile's time is that chain's as long as an SM has few tiles (us without ->
// with, humanoid29 B = 4096: FK 5.0 -> 4.6, RNEA 9.0 -> 8.3, CRBA 10.6 -> 9.8, ABA
// 14.6 -> 13.6; arm7 ABA 12.6 -> 11.1; legged12 B = 1000 d qdd 26.7 -> 23.6). Where
// many tiles wait it still pays for CRBA and the lean RNEA (humanoid29 B = 65536
// 79.8 -> 76.8 and 49.0 -> 47.3), but the lean ABA's registers (109 instead of 77)
// then cost more than the shorter chain saves (91.6 -> 96).
struct BlockBarrier {
  __device__ __forceinline__ void operator()() const { __syncthreads(); }
};
template <bool UP, bool AHEAD, class TP, class Loc, class Dep, class Bar = BlockBarrier>
__device__ __forceinline__ void level_pass(const TP& tp, const Loc& loc, const Dep& dep, const Bar& barrier = Bar()) {
  const int W = n_warps(), w = warp_id(), D = tp.depth();
  if (!AHEAD) {
    FST_UNROLL
    for (int s = 0; s < D; ++s) {
      FST_FOR_MY_BODIES(tp, UP ? D - 1 - s : s, k) dep(loc(tp.level_body(k)));
      barrier();
    }
    return;
  }
  const int n = tp.n();
  decltype(loc(0)) mine;
  bool have = false;
  int j = w;  // position in the order of the pass
  int end = UP ? n - tp.level_begin(D - 1) : tp.level_begin(1);
  for (int s = 0; s < D; ++s) {
    for (;;) {
      if (!have && j < n) {
        mine = loc(tp.level_body(UP ? n - 1 - j : j));
        have = true;
      }
      if (j >= end) break;
      dep(mine);
      have = false;
      j += W;
      if (j >= end) break;
    }
    const int next = s + 1 < D ? s + 1 : s;
    end = UP ? n - tp.level_begin(D - 1 - next) : tp.level_begin(next + 1);
    barrier();
  }
}


// ---- forward kinematics -------------------------------------------------------
template <bool AHEAD = false, class TP>
__device__ __forceinline__ void fk_level(const TP& tp, const Col& q, const LaneState& S, float* __restrict__ poses,
                                         int64_t B, int64_t e, bool act) {
  struct Own {
    int i, parent;
    Xf X;
  };
  level_pass<false, AHEAD>(
      tp,
      [&](int i) {
        const BodyI bi = tp.I(i);
        return Own{i, bi.parent, joint_X(tp.C(i), bi, q)};
      },
      [&](const Own& o) {
        Xf P = o.X;
        if (o.parent >= 0) {
          const Xf Pp = S.X(o.parent, 0);
          compose(Pp.R, Pp.t, o.X, P.R, P.t);
        }
        S.putX(o.i, 0, P);
        if (poses && act) {
          float* out = poses + (int64_t)o.i * 12 * B + e;
#pragma unroll
          for (int c = 0; c < 9; ++c) out[(int64_t)c * B] = P.R[c];
#pragma unroll
          for (int c = 0; c < 3; ++c) out[(int64_t)(9 + c) * B] = P.t[c];
        }
      });
}

// Jacobians after fk_level: one (link, body) column per work item; columns
// of bodies off a link's support path are written as zeros. (Clearing the
// tile's rows first and writing only the support-path columns, as
// crba_level does for M, was measured slower here: the columns are cheap to
// write, and the clear adds L2 writes.)
// Packed (PK non-null, see PackedJ): only the columns on the support path.
template <class TP>
__device__ __forceinline__ void jac_columns(const TP& tp, int nv, const LinkList& links, const LaneState& S,
                                           float* __restrict__ J, int64_t B, int64_t e, bool act,
                                           const PackedJ* PK = nullptr) {
  const int W = n_warps(), w = warp_id();
  const int n = tp.n();
  for (int item = w; item < links.n * n; item += W) {
    const int l = item / n, k = item % n;
    const BodyI bk = tp.I(k);
    if (nv_of(bk.type) == 0 || !act) continue;
    const bool on_path = (tp.C(links.idx[l]).anc >> k) & 1ull;
    int64_t first = (int64_t)l * 6 * nv;
    int stride = nv, col = bk.vi;
    if (PK) {
      if (!on_path) continue;
      first = PK->off[l];
      stride = PK->cols[l];
      col = 0;
      for (int j = bk.parent; j >= 0; j = tp.I(j).parent) col += nv_of(tp.I(j).type);
    }
    const Xf P = S.X(k, 0);
    jac_column(tp, k, P.R, P.t, on_path, stride, col, J + first * B + e, B);
  }
}

// FK, then the Jacobian columns of `links` when J is given.
template <bool AHEAD = false, class TP>
__device__ __forceinline__ void kin_level(const TP& tp, const Col& q, int nv, const LinkList& links,
                                          const LaneState& S, float* __restrict__ poses, float* __restrict__ J,
                                          int64_t B, int64_t e, bool act, const PackedJ* PK = nullptr) {
  fk_level<AHEAD>(tp, q, S, poses, B, e, act);
  if (J) jac_columns(tp, nv, links, S, J, B, e, act, PK);
}

// ---- RNEA -----------------------------------------------------------------------
// tau goes to global memory (may be null) and, if tau_col is not null, also to
// that shared-memory column (rows of 32). With a tape, the forward state of
// every body is left there for the store variant of the adjoint (tape_store's
// layout). LEAN keeps 12 floats a body instead of 30: the force is formed on
// the way back from v and a, which it then replaces, and the joint transform is
// evaluated again instead of stored. That lengthens the chain (quadruped, B =
// 4096: 7.4 -> 8 us) and lets twice the tiles share an SM; the arithmetic and
// so the bits are the same.
// SPEND (with LEAN): the staged rows are the sweep's to overwrite: a joint's sine
// and 1 - cosine replace its q and qd until the way back has used them
// (humanoid B = 65536: 50.2 -> 49.0 us).
template <bool LEAN = false, bool SPEND = false, bool AHEAD = false, class TP>
__device__ __forceinline__ void rnea_level(const TP& tp, SV a0, const Col& q, const Col& qd, const Col& qdd,
                                           const LaneState& S, float* __restrict__ tau, int64_t B, int64_t e,
                                           bool act, float* tau_col = nullptr, float* tape = nullptr) {
  const int W = n_warps(), w = warp_id();
  enum { V_ = 0, A_ = 6, C_ = LEAN ? 0 : 12, X_ = 18 };  // v 6 | a 6 | force, then its contribution 6 | X 12
  auto force = [&](int i, SV v, SV a) {
    const In10 I = in_load(tp.theta(i));
    return in_mul(I, a) + crf(v, in_mul(I, v));
  };
  struct Moved {
    int i, parent;
    Xf X;
    SV vJ;
    ScaledSV aJ;
  };
  level_pass<false, AHEAD>(
      tp,
      [&](int i) {
        const BodyC& c = tp.C(i);
        const BodyI bi = tp.I(i);
        float omc = 0.f;
        if (SPEND && bi.type == FST_JOINT_REVOLUTE) {
          const SinOmc t = sin_omc(q[bi.qi]);
          *q.spent(bi.qi) = t.s;
          omc = t.omc;
        }
        Moved m;
        m.i = i;
        m.parent = bi.parent;
        m.X = joint_X<SPEND>(c, bi, q, &omc);
        m.vJ = S_times(c, bi, qd);
        m.aJ = S_scaled(c, bi, qdd);
        if (SPEND && bi.type == FST_JOINT_REVOLUTE) *qd.spent(bi.vi) = omc;
        return m;
      },
      [&](const Moved& m) {
        const int i = m.i;
        const Xf& X = m.X;
        SV vi, ai;
        if (m.parent < 0) {
          vi = m.vJ;
          ai = m.aJ.add_to(X_motion(X, a0));
        } else {
          vi = X_motion(X, S.sv(m.parent, V_)) + m.vJ;
          ai = m.aJ.add_to(X_motion(X, S.sv(m.parent, A_))) + crm(vi, m.vJ);
        }
        S.put(i, V_, vi);
        S.put(i, A_, ai);
        if (!LEAN) S.putX(i, X_, X);
        if (!LEAN && !AHEAD) S.put(i, C_, force(i, vi, ai));
        if (tape && act) {
          float* p = tape + (int64_t)i * 30 * B + e;
          const float r[24] = {X.R[0], X.R[1], X.R[2], X.R[3], X.R[4], X.R[5], X.R[6], X.R[7],
                               X.R[8], X.t[0], X.t[1], X.t[2], vi.w.x, vi.w.y, vi.w.z, vi.v.x,
                               vi.v.y, vi.v.z, ai.w.x, ai.w.y, ai.w.z, ai.v.x, ai.v.y, ai.v.z};
#pragma unroll
          for (int c2 = 0; c2 < 24; ++c2) p[(int64_t)c2 * B] = r[c2];
        }
      });
  struct Own {
    int i, ch, ch_end;
    BodyI b;
    SV F;
    Xf X;
  };
  level_pass<true, AHEAD>(
      tp,
      [&](int i) {
        Own o;
        o.i = i;
        o.b = tp.I(i);
        o.ch = tp.child_begin(i);
        o.ch_end = tp.child_begin(i + 1);
        o.F = LEAN || AHEAD ? force(i, S.sv(i, V_), S.sv(i, A_)) : S.sv(i, C_);
        if (o.b.parent >= 0) o.X = LEAN ? joint_X<SPEND>(tp.C(i), o.b, q, qd.p + o.b.vi * qd.ld) : S.X(i, X_);
        return o;
      },
      [&](const Own& o) {
        SV F = o.F;
        for (int ch = o.ch_end - 1; ch >= o.ch; --ch) F = F + S.sv(tp.child(ch), C_);
        if (act && tau) ST_store(tp.C(o.i), o.b, F, tau, B, e);
        if (tau_col) ST_store(tp.C(o.i), o.b, F, tau_col, kLaneEnvs, 0);
        if (tape && act) {
          float* p = tape + ((int64_t)o.i * 30 + 24) * B + e;
          const float r[6] = {F.w.x, F.w.y, F.w.z, F.v.x, F.v.y, F.v.z};
#pragma unroll
          for (int c2 = 0; c2 < 6; ++c2) p[(int64_t)c2 * B] = r[c2];
        }
        if (o.b.parent >= 0) S.put(o.i, C_, XT_force(o.X, F));
      });
}

// ---- CRBA -----------------------------------------------------------------------
// Zeros rows [0, rows) of a [rows][B] array for the tile's 32 environments
// e0 .. e0 + 31, shared among the tile's W warps (w = this warp). A full tile
// of a 16-byte aligned array with B a multiple of 4 is cleared with 16-byte
// stores (eight threads per row); otherwise with 4-byte stores, skipping
// environments past B.
__device__ __forceinline__ void m_clear_tile(float* __restrict__ M, int64_t rows, int64_t B, int64_t e0, int W,
                                             int w) {
  const int t = (threadIdx.x & 31) + (w << 5), nt = W << 5;
  if (e0 + kLaneEnvs <= B && (B & 3) == 0 && ((reinterpret_cast<unsigned long long>(M) & 15ull) == 0)) {
    const int part = t & 7;
    const int64_t step = (int64_t)(nt >> 3) * B;
    float4* p = reinterpret_cast<float4*>(M + (int64_t)(t >> 3) * B + e0 + 4 * part);
    for (int64_t r = t >> 3; r < rows; r += nt >> 3, p += step >> 2) *p = make_float4(0.f, 0.f, 0.f, 0.f);
    return;
  }
  const int l = t & 31;
  if (e0 + l >= B) return;
  float* p = M + (int64_t)(t >> 5) * B + e0 + l;
  for (int64_t r = t >> 5; r < rows; r += W, p += (int64_t)W * B) *p = 0.f;
}

template <class TP>
__device__ __forceinline__ void crba_level(const TP& tp, const Col& q, int nv, const LaneState& S,
                                           float* __restrict__ M, int64_t B, int64_t e, bool act) {
  const int W = n_warps(), w = warp_id();
  enum { X_ = 0, IC_ = 12, CT_ = 22 };
  // Structural zeros: the tile clears its whole nv x nv block of M first,
  // and the column phase below overwrites the entries that are not zero.
  // The block barriers of the composite pass order the two sets of stores.
  // Nothing is read back, so DRAM sees each line once; the clear costs L2
  // writes, not a per-entry ancestry test.
  if (tp.depth() > 0) m_clear_tile(M, (int64_t)nv * nv, B, e - (threadIdx.x & 31), W, w);
  FST_UNROLL
  for (int l = tp.depth() - 1; l >= 0; --l) {
    FST_FOR_MY_BODIES(tp, l, k) {
      const int i = tp.level_body(k);
      const BodyI bi = tp.I(i);
      const Xf X = joint_X(tp.C(i), bi, q);
      In10 Ic = in_load(tp.theta(i));
      for (int ch = tp.child_begin(i + 1) - 1; ch >= tp.child_begin(i); --ch) in_add(Ic, S.in10(tp.child(ch), CT_));
      S.putX(i, X_, X);
      S.putin(i, IC_, Ic);
      if (bi.parent >= 0) S.putin(i, CT_, in_to_parent(X, Ic));
    }
    __syncthreads();
  }
  if (!act) return;
  const MOut<false> Me{M + e, nv, B};
  for (int i = w; i < tp.n(); i += W) {
    const BodyI bi = tp.I(i);
    if (bi.type == FST_JOINT_REVOLUTE || bi.type == FST_JOINT_PRISMATIC) {
      const In10 Ic = S.in10(i, IC_);
      SV F = in_mul(Ic, S_of(tp.C(i)));
      Me.one(bi.vi, bi.vi, dot(S_of(tp.C(i)), F));
      // up the support path, parent by parent (parents precede children)
      int kk = i;
      for (int j = bi.parent; j >= 0; j = tp.I(j).parent) {
        F = XT_force(S.X(kk, X_), F);
        kk = j;
        const BodyI bj = tp.I(j);
        if (bj.type == FST_JOINT_REVOLUTE || bj.type == FST_JOINT_PRISMATIC) {
          Me.sym(bi.vi, bj.vi, dot(S_of(tp.C(j)), F));
        } else if (bj.type == FST_JOINT_FREE) {
          const float col[6] = {F.v.x, F.v.y, F.v.z, F.w.x, F.w.y, F.w.z};
#pragma unroll
          for (int r = 0; r < 6; ++r) Me.sym(bj.vi + r, bi.vi, col[r]);
        }
      }
    } else if (bi.type == FST_JOINT_FREE) {
      const In10 I = S.in10(i, IC_);
      const float blk[6][6] = {
          {I.m, 0.f, 0.f, 0.f, I.h.z, -I.h.y},
          {0.f, I.m, 0.f, -I.h.z, 0.f, I.h.x},
          {0.f, 0.f, I.m, I.h.y, -I.h.x, 0.f},
          {0.f, -I.h.z, I.h.y, I.I[0], I.I[1], I.I[3]},
          {I.h.z, 0.f, -I.h.x, I.I[1], I.I[2], I.I[4]},
          {-I.h.y, I.h.x, 0.f, I.I[3], I.I[4], I.I[5]},
      };
#pragma unroll
      for (int r = 0; r < 6; ++r)
#pragma unroll
        for (int cc = 0; cc < 6; ++cc) Me.one(bi.vi + r, bi.vi + cc, blk[r][cc]);
    }
  }
}

// ---- CRBA, lean shared memory ---------------------------------------------------
// Joint transform of body i with its coordinates read straight from global
// memory (rows of B; ec a valid environment index), for kernels that do not
// stage q in shared memory.
__device__ __forceinline__ Xf joint_X_rows(const BodyC& c, const BodyI& bi, const float* __restrict__ q, int64_t B,
                                           int64_t ec) {
  const int nqb = bi.type == FST_JOINT_FREE ? 7 : bi.type == FST_JOINT_FIXED ? 0 : 1;
  float qb[7];
#pragma unroll
  for (int k = 0; k < 7; ++k) qb[k] = k < nqb ? ld_input(q + (int64_t)(bi.qi + k) * B + ec) : 0.f;
  BodyI b0 = bi;
  b0.qi = 0;
  return joint_X(c, b0, Col{qb, 1});
}

// The composite-rigid-body algorithm with less shared memory per tile (so
// that three tiles of a large tree fit on one SM): per body only X and
// F = I^c S stay (kCrbaLeanBodyFloats); a body's composite inertia moved to
// its parent lives in a slot of R (BodyC::slot) until the parent has added it;
// the root keeps its own I^c in its slot for a free base's 6 x 6 block. X_of(c, b)
// gives a joint's transform, from staged rows of q or, where those do not fit,
// from global memory. Same arithmetic, in the same order, as crba_level.
template <bool PACKED = false, bool AHEAD = true, class TP, class XF>
__device__ __forceinline__ void crba_level_lean(const TP& tp, const XF& X_of, int nv,
                                                const LaneState& S, const LaneState& R,
                                                float* __restrict__ M, int64_t B, int64_t e, bool act) {
  const int W = n_warps(), w = warp_id();
  enum { X_ = 0, F_ = 12 };
  if (tp.depth() > 0) m_clear_tile(M, PACKED ? (int64_t)nv * (nv + 1) / 2 : (int64_t)nv * nv, B, e - (threadIdx.x & 31), W, w);
  struct Own {
    int i, type, parent, slot, ch, ch_end;
    Xf X;
    In10 I;
  };
  level_pass<true, AHEAD>(
      tp,
      [&](int i) {
        const BodyI bi = tp.I(i);
        Own o;
        o.i = i;
        o.type = bi.type;
        o.parent = bi.parent;
        o.slot = tp.C(i).slot;
        o.ch = tp.child_begin(i);
        o.ch_end = tp.child_begin(i + 1);
        o.X = X_of(tp.C(i), bi);
        o.I = in_load(tp.theta(i));
        S.putX(i, X_, o.X);
        return o;
      },
      [&](const Own& o) {
        In10 Ic = o.I;
        for (int ch = o.ch_end - 1; ch >= o.ch; --ch) in_add(Ic, R.in10(tp.C(tp.child(ch)).slot, 0));
        if (o.type == FST_JOINT_REVOLUTE || o.type == FST_JOINT_PRISMATIC)
          S.put(o.i, F_, in_mul(Ic, S_of(tp.C(o.i))));
        R.putin(o.slot, 0, o.parent >= 0 ? in_to_parent(o.X, Ic) : Ic);
      });
  if (!act) return;
  const MOut<PACKED> Me{M + e, nv, B};
  // deepest bodies, and so longest walks, first: the warps end together
  for (int k = tp.n() - 1 - w; k >= 0; k -= W) {
    const int i = tp.level_body(k);
    const BodyI bi = tp.I(i);
    if (bi.type == FST_JOINT_REVOLUTE || bi.type == FST_JOINT_PRISMATIC) {
      SV F = S.sv(i, F_);
      Me.one(bi.vi, bi.vi, dot(S_of(tp.C(i)), F));
      int kk = i;
      for (int j = bi.parent; j >= 0; j = tp.I(j).parent) {
        F = XT_force(S.X(kk, X_), F);
        kk = j;
        const BodyI bj = tp.I(j);
        if (bj.type == FST_JOINT_REVOLUTE || bj.type == FST_JOINT_PRISMATIC) {
          Me.sym(bi.vi, bj.vi, dot(S_of(tp.C(j)), F));
        } else if (bj.type == FST_JOINT_FREE) {
          const float col[6] = {F.v.x, F.v.y, F.v.z, F.w.x, F.w.y, F.w.z};
#pragma unroll
          for (int r = 0; r < 6; ++r) Me.sym(bj.vi + r, bi.vi, col[r]);
        }
      }
    } else if (bi.type == FST_JOINT_FREE) {
      const In10 I = R.in10(tp.C(i).slot, 0);  // the root's own slot
      const float blk[6][6] = {
          {I.m, 0.f, 0.f, 0.f, I.h.z, -I.h.y},
          {0.f, I.m, 0.f, -I.h.z, 0.f, I.h.x},
          {0.f, 0.f, I.m, I.h.y, -I.h.x, 0.f},
          {0.f, -I.h.z, I.h.y, I.I[0], I.I[1], I.I[3]},
          {I.h.z, 0.f, -I.h.x, I.I[1], I.I[2], I.I[4]},
          {-I.h.y, I.h.x, 0.f, I.I[3], I.I[4], I.I[5]},
      };
#pragma unroll
      for (int r = 0; r < 6; ++r)
#pragma unroll
        for (int cc = 0; cc < 6; ++cc) Me.one(bi.vi + r, bi.vi + cc, blk[r][cc]);
    }
  }
}

// ---- ABA ------------------------------------------------------------------------
template <class TP>
__device__ __forceinline__ void aba_level(const TP& tp, SV a0, const Col& q, const Col& qd, const Col& tau,
                                          const LaneState& S, float* __restrict__ qdd, int64_t B, int64_t e,
                                          bool act) {
  const int W = n_warps(), w = warp_id();
  enum { X_ = 0, VA_ = 12, C_ = 18, IA_ = 24, PA_ = 45, U_ = 51, ID_ = 57, u_ = 58 };
  // 1. root to leaf: velocities, bias accelerations, rigid inertias
  FST_UNROLL
  for (int l = 0; l < tp.depth(); ++l) {
    FST_FOR_MY_BODIES(tp, l, k) {
      const int i = tp.level_body(k);
      const BodyC& c = tp.C(i);
      const BodyI bi = tp.I(i);
      const Xf X = joint_X(c, bi, q);
      const SV vJ = S_times(c, bi, qd);
      SV vi, ci;
      if (bi.parent < 0) {
        vi = vJ;
        ci = sv_zero();
      } else {
        vi = X_motion(X, S.sv(bi.parent, VA_)) + vJ;
        ci = crm(vi, vJ);
      }
      const In10 I = in_load(tp.theta(i));
      S.putX(i, X_, X);
      S.put(i, VA_, vi);
      S.put(i, C_, ci);
      S.putsym(i, IA_, sym6_from_in(I));
      S.put(i, PA_, crf(vi, in_mul(I, vi)));
    }
    __syncthreads();
  }
  // 2. leaf to root: articulated inertias; each body leaves X^T I^a X and
  //    X^T p^a for its parent in its own IA/PA slots
  FST_UNROLL
  for (int l = tp.depth() - 1; l >= 0; --l) {
    FST_FOR_MY_BODIES(tp, l, k) {
      const int i = tp.level_body(k);
      const BodyI bi = tp.I(i);
      Sym6 IA = S.sym(i, IA_);
      SV pA = S.sv(i, PA_);
      for (int ch = tp.child_begin(i + 1) - 1; ch >= tp.child_begin(i); --ch) {
        sym6_add(IA, S.sym(tp.child(ch), IA_));
        pA = pA + S.sv(tp.child(ch), PA_);
      }
      if (bi.type == FST_JOINT_FREE) {
        S.putsym(i, IA_, IA);
        S.put(i, PA_, pA);
        continue;
      }
      Sym6 Ia = IA;
      SV pa = pA;
      if (bi.type != FST_JOINT_FIXED) {
        const SV Sv = S_of(tp.C(i));
        const SV Ui = sym6_mul(IA, Sv);
        const float iD = 1.0f / dot(Sv, Ui);
        const float ui = tau[bi.vi] - dot(Sv, pA);
        S.put(i, U_, Ui);
        *S.at(i, ID_) = iD;
        *S.at(i, u_) = ui;
        if (bi.parent < 0) continue;
        sym6_rank1_sub(Ia, Ui, iD);
        pa = sv_fma(ui * iD, Ui, pa + sym6_mul(Ia, S.sv(i, C_)));
      } else {
        if (bi.parent < 0) continue;
        pa = pa + sym6_mul(Ia, S.sv(i, C_));
      }
      const Xf X = S.X(i, X_);
      S.putsym(i, IA_, sym6_to_parent(X, Ia));
      S.put(i, PA_, XT_force(X, pa));
    }
    __syncthreads();
  }
  // 3. root to leaf: accelerations
  FST_UNROLL
  for (int l = 0; l < tp.depth(); ++l) {
    FST_FOR_MY_BODIES(tp, l, k) {
      const int i = tp.level_body(k);
      const BodyI bi = tp.I(i);
      const SV ap = bi.parent < 0 ? a0 : S.sv(bi.parent, VA_);
      SV ai = X_motion(S.X(i, X_), ap) + S.sv(i, C_);
      if (bi.type == FST_JOINT_REVOLUTE || bi.type == FST_JOINT_PRISMATIC) {
        const float qi = (*S.at(i, u_) - dot(S.sv(i, U_), ai)) * *S.at(i, ID_);
        if (act) qdd[(int64_t)bi.vi * B + e] = qi;
        ai = sv_fma(qi, S_of(tp.C(i)), ai);
      } else if (bi.type == FST_JOINT_FREE) {
        const SV tf = SV{f3{tau[bi.vi + 3], tau[bi.vi + 4], tau[bi.vi + 5]}, f3{tau[bi.vi], tau[bi.vi + 1], tau[bi.vi + 2]}};
        const SV anew = sym6_solve(S.sym(i, IA_), tf - S.sv(i, PA_));
        const SV x = anew - ai;
        if (act) {
          const float xo[6] = {x.v.x, x.v.y, x.v.z, x.w.x, x.w.y, x.w.z};
#pragma unroll
          for (int r = 0; r < 6; ++r) qdd[(int64_t)(bi.vi + r) * B + e] = xo[r];
        }
        ai = anew;
      }
      S.put(i, VA_, ai);
    }
    __syncthreads();
  }
}

// ---- ABA, lean shared memory ------------------------------------------------------
// The same three passes with less state per tile, so that a large tree's
// tiles fit two per SM: per body only VU (v in pass 1, U from pass 2, a in
// pass 3), c, invD and u stay (kAbaLeanBodyFloats); a body's contribution to
// its parent (X^T I^a X, X^T p^a) lives in a slot of R only until the parent
// has read it (kAbaLeanSlotFloats each; the parent reuses its first child's,
// BodyC::slot, so the humanoid needs 4); the rigid inertia and
// the bias force are formed in pass 2, and the joint transforms recomputed
// in passes 2 and 3 instead of stored. The root's I^A and p^A, which pass 3
// needs for a free base, stay in its slot.
// SPEND: the caller has no further use for the staged rows. The sines of all
// joints are then taken first, by all warps at once and not once a pass on the
// chain of levels, and stay in the rows of q and the state; 1 / D and u move
// to the rows of qd and tau once pass 2 has read them (B = 4096: quadruped
// 11.0 -> 10.3 us, arm7 13.8 -> 12.6; humanoid B = 65536 93.2 -> 91.6).
template <bool SPEND = false, bool AHEAD = false, class TP>
__device__ __forceinline__ void aba_level_lean(const TP& tp, SV a0, const Col& q, const Col& qd, const Col& tau,
                                               const LaneState& S, const LaneState& R,
                                               float* __restrict__ qdd, int64_t B, int64_t e, bool act,
                                               float* qdd_col = nullptr) {
  const int W = n_warps(), w = warp_id();
  enum { VU_ = 0, C_ = 6, OMC_ = 12, ID_ = 12, u_ = 13 };  // per body
  enum { RI_ = 0, RP_ = 21 };                              // per slot
  if (SPEND) {
    for (int i = w; i < tp.n(); i += W) {
      const BodyI bi = tp.I(i);
      if (bi.type != FST_JOINT_REVOLUTE) continue;
      const SinOmc t = sin_omc(q[bi.qi]);
      *q.spent(bi.qi) = t.s;
      *S.at(i, OMC_) = t.omc;
    }
    __syncthreads();
  }
  auto X_of = [&](int i, const BodyI& bi) { return joint_X<SPEND>(tp.C(i), bi, q, S.at(i, OMC_)); };
  // 1. root to leaf: velocities and bias accelerations
  struct Moved {
    int i, parent;
    Xf X;
    SV vJ;
  };
  level_pass<false, AHEAD>(
      tp,
      [&](int i) {
        const BodyI bi = tp.I(i);
        Moved m;
        m.i = i;
        m.parent = bi.parent;
        m.vJ = S_times(tp.C(i), bi, qd);
        if (bi.parent >= 0) m.X = X_of(i, bi);
        return m;
      },
      [&](const Moved& m) {
        SV vi = m.vJ, ci = sv_zero();
        if (m.parent >= 0) {
          vi = X_motion(m.X, S.sv(m.parent, VU_)) + m.vJ;
          ci = crm(vi, m.vJ);
        }
        S.put(m.i, VU_, vi);
        S.put(m.i, C_, ci);
      });
  // 2. leaf to root: articulated inertias
  struct Own {
    int i, slot, ch, ch_end, ch_slot;
    BodyI b;
    In10 I;
    SV p;
    Xf X;
  };
  level_pass<true, AHEAD>(
      tp,
      [&](int i) {
        const BodyI bi = tp.I(i);
        Own o;
        o.i = i;
        o.b = bi;
        o.slot = tp.C(i).slot;
        o.ch = tp.child_begin(i);
        o.ch_end = tp.child_begin(i + 1);
        o.ch_slot = AHEAD && o.ch < o.ch_end ? tp.C(tp.child(o.ch_end - 1)).slot : 0;
        o.I = in_load(tp.theta(i));
        const SV vi = S.sv(i, VU_);
        o.p = crf(vi, in_mul(o.I, vi));
        if (AHEAD && bi.parent >= 0) o.X = X_of(i, bi);
        return o;
      },
      [&](const Own& o) {
        Sym6 IA = sym6_from_in(o.I);
        SV pA = o.p;
        for (int ch = o.ch_end - 1; ch >= o.ch; --ch) {
          const int cs = AHEAD && ch == o.ch_end - 1 ? o.ch_slot : tp.C(tp.child(ch)).slot;
          sym6_add(IA, R.sym(cs, RI_));
          pA = pA + R.sv(cs, RP_);
        }
        if (o.b.type == FST_JOINT_FREE) {
          R.putsym(o.slot, RI_, IA);
          R.put(o.slot, RP_, pA);
          return;
        }
        Sym6 Ia = IA;
        SV pa = pA;
        if (o.b.type != FST_JOINT_FIXED) {
          const SV Sv = S_of(tp.C(o.i));
          const SV Ui = sym6_mul(IA, Sv);
          const float iD = 1.0f / dot(Sv, Ui);
          const float ui = tau[o.b.vi] - dot(Sv, pA);
          S.put(o.i, VU_, Ui);
          *(SPEND ? qd.spent(o.b.vi) : S.at(o.i, ID_)) = iD;
          *(SPEND ? tau.spent(o.b.vi) : S.at(o.i, u_)) = ui;
          if (o.b.parent < 0) return;
          sym6_rank1_sub(Ia, Ui, iD);
          pa = sv_fma(ui * iD, Ui, pa + sym6_mul(Ia, S.sv(o.i, C_)));
        } else {
          if (o.b.parent < 0) return;
          pa = pa + sym6_mul(Ia, S.sv(o.i, C_));
        }
        const Xf X = AHEAD ? o.X : X_of(o.i, o.b);
        R.putsym(o.slot, RI_, sym6_to_parent(X, Ia));
        R.put(o.slot, RP_, XT_force(X, pa));
      });
  // 3. root to leaf: accelerations (each body reads its U before it
  //    overwrites VU with its acceleration)
  struct Joint {
    int i;
    BodyI b;
    Xf X;
    SV c, U;
  };
  level_pass<false, AHEAD>(
      tp,
      [&](int i) {
        Joint m;
        m.i = i;
        m.b = tp.I(i);
        if (AHEAD) {
          m.X = X_of(i, m.b);
          m.c = S.sv(i, C_);
          m.U = S.sv(i, VU_);
        }
        return m;
      },
      [&](const Joint& m) {
        const SV ap = m.b.parent < 0 ? a0 : S.sv(m.b.parent, VU_);
        SV ai = X_motion(AHEAD ? m.X : X_of(m.i, m.b), ap) + (AHEAD ? m.c : S.sv(m.i, C_));
        if (m.b.type == FST_JOINT_REVOLUTE || m.b.type == FST_JOINT_PRISMATIC) {
          const float u = SPEND ? tau[m.b.vi] : *S.at(m.i, u_), iD = SPEND ? qd[m.b.vi] : *S.at(m.i, ID_);
          const float qi = (u - dot(AHEAD ? m.U : S.sv(m.i, VU_), ai)) * iD;
          if (act && qdd) qdd[(int64_t)m.b.vi * B + e] = qi;
          if (qdd_col) qdd_col[m.b.vi << 5] = qi;
          ai = sv_fma(qi, S_of(tp.C(m.i)), ai);
        } else if (m.b.type == FST_JOINT_FREE) {
          const int slot = tp.C(m.i).slot, vi = m.b.vi;
          const SV tf = SV{f3{tau[vi + 3], tau[vi + 4], tau[vi + 5]}, f3{tau[vi], tau[vi + 1], tau[vi + 2]}};
          const SV anew = sym6_solve(R.sym(slot, RI_), tf - R.sv(slot, RP_));
          const SV x = anew - ai;
          const float xo[6] = {x.v.x, x.v.y, x.v.z, x.w.x, x.w.y, x.w.z};
#pragma unroll
          for (int r = 0; r < 6; ++r) {
            if (act && qdd) qdd[(int64_t)(vi + r) * B + e] = xo[r];
            if (qdd_col) qdd_col[(vi + r) << 5] = xo[r];
          }
          ai = anew;
        }
        S.put(m.i, VU_, ai);
      });
}

}  // namespace fst
