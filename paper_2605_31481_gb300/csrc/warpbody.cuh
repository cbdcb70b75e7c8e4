// One warp per body: a block is one tile of 32 environments (one per lane) of
// a tree of at most 16 bodies, and warp w owns body level_body[w] for the
// whole call.
//
// Everything of a body that nobody else reads stays in its warp's registers:
// its joint transform, subspace, inertia, bias terms, articulated inertia.
// Only what passes along the tree goes through shared memory, once: a body's
// rotation, velocity and acceleration for its children, and one already
// shifted contribution for its parent. Inputs are read straight from global
// memory by the warp that needs them (a row of 32 environments is one
// 128-byte line), constants through the L1, and the topology is a kernel
// argument, so a block's first loads leave in its first cycles.
//
// The level kernels of level.cuh share a tile's bodies among a few warps
// instead: their per-body state lives in shared memory (humanoid RNEA 30
// floats a body, ABA 59, the adjoint 51), each phase starts with a chain of
// dependent index loads, and only the bodies of one level have a warp. With a
// warp per body all joint transforms, inertias and forces of the tree are
// formed at once, and a level phase is what really depends on the parent.
//
// The adjoint's quantities are in body-origin frames with root-aligned axes
// (aligned.cuh).
//
// Every warp of a block meets every barrier (phases are loops over the tree's
// levels with a warp-uniform test inside); lanes past B work on the last
// environment and store nothing.
#pragma once

#include "aligned.cuh"

namespace fst {

// What a warp knows about its body.
struct Me {
  int i, type, lev, par, nch, c0, qi, vi, depth;
  __device__ __forceinline__ explicit Me(const WarpTree& t) {
    const WarpTree::Entry x = t.e[threadIdx.x >> 5];
    i = x.body;
    type = x.type;
    lev = x.level;
    par = x.parent;
    nch = x.n_child;
    c0 = x.child0;
    qi = x.qi;
    vi = x.vi;
    depth = t.depth;
  }
  __device__ __forceinline__ bool free_joint() const { return type == FST_JOINT_FREE; }
  __device__ __forceinline__ bool one_dof() const {
    return type == FST_JOINT_REVOLUTE || type == FST_JOINT_PRISMATIC;
  }
  __device__ __forceinline__ int nv() const { return nv_of(type); }
};

// This body's coordinates of a [rows][B] array: up to 7 values in registers.
struct Own {
  float x[7];
};
__device__ __forceinline__ Own own_rows(const float* __restrict__ src, int first, int count, int64_t B, int64_t ec) {
  Own o;
#pragma unroll
  for (int k = 0; k < 7; ++k) o.x[k] = k < count ? ld_input(src + (int64_t)(first + k) * B + ec) : 0.f;
  return o;
}
__device__ __forceinline__ Own own_q(const Me& me, const float* __restrict__ q, int64_t B, int64_t ec) {
  return own_rows(q, me.qi, me.free_joint() ? 7 : me.one_dof() ? 1 : 0, B, ec);
}
__device__ __forceinline__ Own own_v(const Me& me, const float* __restrict__ v, int64_t B, int64_t ec) {
  return own_rows(v, me.vi, me.nv(), B, ec);
}
// S x of a free joint, whose coordinates are [v; w]
__device__ __forceinline__ SV free_motion(const Own& o) {
  return SV{f3{o.x[3], o.x[4], o.x[5]}, f3{o.x[0], o.x[1], o.x[2]}};
}

__device__ __forceinline__ const float* own_theta(const Me& me, const ModelView& mv) {
  return mv.theta ? mv.theta + 10 * me.i : mv.c[me.i].theta;
}
__device__ __forceinline__ In10 own_inertia(const Me& me, const ModelView& mv) {
  const float* th = own_theta(me, mv);
  float t[10];
#pragma unroll
  for (int k = 0; k < 10; ++k) t[k] = ld_input(th + k);
  return in_load(t);
}

__device__ __forceinline__ Xf own_joint(const Me& me, const ModelView& mv, const Own& q) {
  const BodyI b{me.par, me.type, 0, 0};
  return joint_X(mv.c[me.i], b, Col{q.x, 1});
}

// The body's kinematics down the tree: rotation in root axes, offset, and the
// parent's velocity and acceleration at this body's origin.
struct Down {
  float R[9];
  f3 r;
  SV psi;
};

// Composes this body's rotation with its parent's (slot R9 of the parent).
__device__ __forceinline__ void own_rotation(const Me& me, const BodyC& c, const Xf& X, const LaneState& S, Down& d) {
  if (me.free_joint()) {
#pragma unroll
    for (int k = 0; k < 9; ++k) d.R[k] = (k & 3) == 0 ? 1.f : 0.f;
    d.r = f3{0.f, 0.f, 0.f};
  } else if (me.par < 0) {
#pragma unroll
    for (int k = 0; k < 9; ++k) d.R[k] = X.R[k];
    d.r = tvec(X);
  } else {
    float Rp[9], t[3];
    S.get_n(me.par, 0, Rp, 9);
    const float zero[3] = {0.f, 0.f, 0.f};
    compose(Rp, zero, X, d.R, t);
    d.r = f3{t[0], t[1], t[2]};
  }
  d.psi = me.one_dof() ? psi_of(c, d.R) : sv_zero();
}

// ---- the adjoint of inverse dynamics ---------------------------------------------
// Shared floats per body: R 9 | v 6 | a 6 | w 6 going down; going up the same
// space holds the force (6), then A 6 and H 3, already about the parent's origin.
constexpr int kWbVjpFloats = 27;

// The sweep down the tree. v, a: the body's own; vl, al: its parent's at its
// origin.
struct Sweep {
  Down d;
  SV v, a, vl, al, psd;
};

template <bool WITH_W, bool BODY>
__device__ __forceinline__ void sweep_down(const Me& me, const ModelView& mv, const Xf& X, const Own& qd, const Own& qdd,
                                           const Own& tb, const LaneState& S, Sweep& s, SV& wl, SV& wv) {
  const BodyC& c = mv.c[me.i];
  const SV a0 = world_accel(mv);
  s.vl = sv_zero();
  s.al = a0;
  wl = sv_zero();
  wv = sv_zero();
  for (int l = 0; l < me.depth; ++l) {
    if (me.lev == l) {
      if (BODY)
        s.d.psi = me.one_dof() ? S_of(c) : sv_zero();
      else
        own_rotation(me, c, X, S, s.d);
      if (me.free_joint()) {
        s.al = SV{f3{0.f, 0.f, 0.f}, RTmul(X.R, a0.v)};
        s.v = free_motion(qd);
        s.a = free_motion(qdd) + s.al;
        s.psd = sv_zero();
        if (WITH_W) wv = free_motion(tb);
      } else {
        auto to_child = [&](SV m) { return BODY ? X_motion(X, m) : shift_motion(m, s.d.r); };
        if (me.par >= 0) {
          s.vl = to_child(S.sv(me.par, 9));
          s.al = to_child(S.sv(me.par, 15));
          if (WITH_W) wl = to_child(S.sv(me.par, 21));
        } else if (BODY) {
          s.al = X_motion(X, a0);
        }
        s.v = s.vl;
        s.a = s.al;
        wv = wl;
        s.psd = sv_zero();
        if (me.one_dof()) {
          s.psd = crm(s.vl, s.d.psi);
          s.v = sv_fma(qd.x[0], s.d.psi, s.vl);
          s.a = sv_fma(qdd.x[0], s.d.psi, sv_fma(qd.x[0], s.psd, s.al));
          if (WITH_W) wv = sv_fma(tb.x[0], s.d.psi, wl);
        }
      }
      if (me.nch) {
        if (!BODY) S.put_n(me.i, 0, s.d.R, 9);
        S.put(me.i, 9, s.v);
        S.put(me.i, 15, s.a);
        if (WITH_W) S.put(me.i, 21, wv);
      }
    }
    __syncthreads();
  }
}

// f := the subtree's force; each body leaves its own about the parent's origin in slot 0.
__device__ __forceinline__ void force_up(const Me& me, const WarpTree& t, const LaneState& S, f3 r, SV& f) {
  for (int l = me.depth - 1; l >= 0; --l) {
    if (me.lev == l) {
      for (int k = 0; k < me.nch; ++k) f = f + S.sv(t.child[me.c0 + k], 0);
      if (me.par >= 0) S.put(me.i, 0, shift_force(f, r));
    }
    if (l > 0) __syncthreads();
  }
}

// The adjoint; formulas, modes and results as in rnea_vjp_aligned, whose sums
// run in the same order (the two give the same bits). tb: this body's rows of
// the cotangent or of the measured torques. BODY: in body axes, as there.
template <int MODE, bool BODY = false>
__device__ __forceinline__ float vjp_warp(const Me& me, const WarpTree& t, const ModelView& mv,
                                          const float* __restrict__ q, const float* __restrict__ qd,
                                          const float* __restrict__ qdd, Own tb, const LaneState& S,
                                          const VjpAligned& o, int64_t B, int64_t e, bool act) {
  static_assert(!BODY || MODE == VJP_GIVEN, "the loss runs in root axes");
  const int64_t ec = act ? e : B - 1;
  const Own xq = own_q(me, q, B, ec), xd = own_v(me, qd, B, ec), xdd = own_v(me, qdd, B, ec);
  Sweep s;
  SV wl, wv;
  float loss = 0.f;
  const Xf X = own_joint(me, mv, xq);
  sweep_down<MODE == VJP_GIVEN, BODY>(me, mv, X, xd, xdd, tb, S, s, wl, wv);
  const In10 I = BODY ? own_inertia(me, mv) : in_rotate(s.d.R, own_inertia(me, mv));
  const SV hv = in_mul(I, s.v);
  SV f = in_mul(I, s.a) + crf(s.v, hv);
  if (MODE != VJP_GIVEN) {
    force_up(me, t, S, s.d.r, f);
    // the residual, its cotangent, and the cotangent's velocity down the tree
    const float t6[6] = {f.v.x, f.v.y, f.v.z, f.w.x, f.w.y, f.w.z};
    const float t1 = dot(s.d.psi, f);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      if (k >= me.nv()) break;
      const float res = (me.one_dof() ? t1 : t6[k]) - tb.x[k];
      loss = fmaf(res, res, loss);
      tb.x[k] = 2.f * res;
    }
    __syncthreads();  // every parent has read its children's forces
    for (int l = 0; l < me.depth; ++l) {
      if (me.lev == l) {
        if (me.free_joint()) {
          wv = free_motion(tb);
        } else {
          if (me.par >= 0) wl = shift_motion(S.sv(me.par, 21), s.d.r);
          wv = me.one_dof() ? sv_fma(tb.x[0], s.d.psi, wl) : wl;
        }
        if (me.nch) S.put(me.i, 21, wv);
      }
      __syncthreads();
    }
  }
  SV A = in_mul(I, wv);
  f3 H = 2.f * (second_moment_mul(I, cross(s.v.w, wv.w)) + (dot(I.h, s.v.v) * wv.w - dot(s.v.v, wv.w) * I.h) -
                cross(wv.v, hv.v));
  if (o.thbar) {
    float g[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    inertia_contract(wv, s.a, g);
    inertia_contract(crm(wv, s.v), s.v, g);
    if (!BODY) inertia_grad_to_body(s.d.R, g);
#pragma unroll
    for (int c = 0; c < 10; ++c) g[c] = act ? o.sign * g[c] : 0.f;
    warp_sum10_store(g, o.thbar + 10 * me.i);
  }
  if (!o.qbar && !o.qdbar && !o.qddbar) return loss;  // block-uniform
  for (int l = me.depth - 1; l >= 0; --l) {
    if (me.lev == l) {
      for (int k = 0; k < me.nch; ++k) {
        const int c = t.child[me.c0 + k];
        if (MODE == VJP_GIVEN) f = f + S.sv(c, 0);
        A = A + S.sv(c, 6);
        const float* h = S.at(c, 12);
        H = H + f3{h[0], h[32], h[64]};
      }
      if (me.par >= 0) {
        if (MODE == VJP_GIVEN) S.put(me.i, 0, BODY ? XT_force(X, f) : shift_force(f, s.d.r));
        S.put(me.i, 6, BODY ? XT_force(X, A) : shift_force(A, s.d.r));
        const f3 hp = BODY ? Rmul(X.R, H) : H;
        float* h = S.at(me.i, 12);
        h[0] = hp.x;
        h[32] = hp.y;
        h[64] = hp.z;
      }
    }
    if (l > 0) __syncthreads();
  }
  if (!act || me.nv() == 0) return loss;
  if (me.free_joint()) {
    // v = S qd, a = X a0 + S qdd: q enters through gravity only
    const SV y = crf(s.v, A);  // eta . A = -psi . (v_0 x* A)
    const f3 g1 = RTmul(mv.c[me.i].R0, world_accel(mv).v);
    const float G[9] = {g1.x * A.v.x, g1.x * A.v.y, g1.x * A.v.z, g1.y * A.v.x, g1.y * A.v.y,
                        g1.y * A.v.z, g1.z * A.v.x, g1.z * A.v.y, g1.z * A.v.z};
    float gq[4];
    quat_grad(xq.x[3], xq.x[4], xq.x[5], xq.x[6], G, gq);
    const float qo[7] = {0.f, 0.f, 0.f, gq[0], gq[1], gq[2], gq[3]};
    const float vo[6] = {-y.v.x, -y.v.y, -y.v.z, H.x - y.w.x, H.y - y.w.y, H.z - y.w.z};
    const float ao[6] = {A.v.x, A.v.y, A.v.z, A.w.x, A.w.y, A.w.z};
#pragma unroll
    for (int r = 0; r < 7; ++r) store_if(o.qbar, me.qi + r, B, e, o.sign * qo[r], true);
#pragma unroll
    for (int r = 0; r < 6; ++r) {
      store_if(o.qdbar, me.vi + r, B, e, o.sign * vo[r], true);
      store_if(o.qddbar, me.vi + r, B, e, o.sign * ao[r], true);
    }
    return loss;
  }
  const SV psi = s.d.psi;
  const SV psdd = crm(s.al, psi) + crm(s.vl, s.psd);
  store_if(o.qbar, me.qi, B, e, o.sign * (dot(crm(wl, psi), f) + dot(psdd, A) + dot(s.psd.w, H)), true);
  store_if(o.qdbar, me.vi, B, e, o.sign * fmaf(2.f, dot(s.psd, A), dot(psi.w, H)), true);
  store_if(o.qddbar, me.vi, B, e, o.sign * dot(psi, A), true);
  return loss;
}

// ---- M^-1 ---------------------------------------------------------------
// In body frames, unlike the adjoint above: D = S . I^A S of a joint then holds
// the rounding of the rotations below it, not that of the product of all those
// up to the root, which turning inertia and subspace to the root's axes would
// put into every D and so into the result (tau_bar of the ABA adjoint against 64
// bits, relative 2-norm: quadruped11 1.3e-7 and 3.7e-7 in root axes, arm7 2.1e-7
// and 4.6e-7). There is no sweep of rotations down the tree before it, either.
// Shared floats per body: the articulated inertia and bias force about the
// parent's origin (21 | 6) going up, the acceleration 6 going down.
static_assert(kWbVjpFloats == 27, "M^-1 and the adjoint share one layout");

// M^-1 applied to tau: the articulated-body sweep at rest and without gravity.
// The result goes to out (may be null) and is returned for this body.
__device__ __forceinline__ Own minv_warp(const Me& me, const WarpTree& t, const ModelView& mv,
                                         const float* __restrict__ q, const float* __restrict__ tau,
                                         const LaneState& S, float* __restrict__ out, int64_t B, int64_t e, bool act) {
  const int64_t ec = act ? e : B - 1;
  const Own xt = own_v(me, tau, B, ec);
  const Xf X = own_joint(me, mv, own_q(me, q, B, ec));
  Sym6 IA = sym6_from_in(own_inertia(me, mv));
  SV pA = sv_zero(), U = sv_zero();
  float invD = 0.f, u = 0.f;
  for (int l = me.depth - 1; l >= 0; --l) {
    if (me.lev == l) {
      for (int k = me.nch - 1; k >= 0; --k) {  // as in the other forms of ABA
        const int ch = t.child[me.c0 + k];
        sym6_add(IA, S.sym(ch, 0));
        pA = pA + S.sv(ch, 21);
      }
      if (me.one_dof()) {
        const SV s = S_of(mv.c[me.i]);
        U = sym6_mul(IA, s);
        invD = 1.0f / dot(s, U);
        u = xt.x[0] - dot(s, pA);
      }
      if (me.par >= 0) {
        if (me.one_dof()) {
          sym6_rank1_sub(IA, U, invD);
          pA = sv_fma(u * invD, U, pA);
        }
        S.putsym(me.i, 0, sym6_to_parent(X, IA));
        S.put(me.i, 21, XT_force(X, pA));
      }
    }
    __syncthreads();
  }
  Own x{};
  for (int l = 0; l < me.depth; ++l) {
    if (me.lev == l) {
      SV a = me.par < 0 ? sv_zero() : X_motion(X, S.sv(me.par, 0));
      if (me.free_joint()) {
        a = sym6_solve(IA, free_motion(xt) - pA);
        const float xo[6] = {a.v.x, a.v.y, a.v.z, a.w.x, a.w.y, a.w.z};
#pragma unroll
        for (int r = 0; r < 6; ++r) x.x[r] = xo[r];
      } else if (me.one_dof()) {
        x.x[0] = (u - dot(U, a)) * invD;
        a = sv_fma(x.x[0], S_of(mv.c[me.i]), a);
      }
      if (me.nch) S.put(me.i, 0, a);
      if (out && act)
#pragma unroll
        for (int r = 0; r < 6; ++r)
          if (r < me.nv()) out[(int64_t)(me.vi + r) * B + e] = x.x[r];
    }
    if (l + 1 < me.depth) __syncthreads();
  }
  return x;
}

}  // namespace fst
