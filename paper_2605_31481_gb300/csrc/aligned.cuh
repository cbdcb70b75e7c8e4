// Dynamics in body-origin frames whose axes are aligned with the root.
//
// Every spatial quantity of body i is expressed with the axes of its tree's
// root (the world for a fixed base, body 0 for a floating one) and about
// body i's own origin. Moving a vector between a body and its parent is then
// a shift by r_i (the body's origin seen from the parent's), one cross
// product, instead of a rotation and a shift, and the quantities keep the
// magnitudes they have in body coordinates: no moment arm to a far root
// enters, so nothing cancels that does not cancel there.
//
// What that buys is a short chain. The only serial recursions left are the
// rotations and velocities down the tree and plain sums (with a shift) up it;
// joint transforms, inertias, forces and every derivative below are per-body
// work that all warps of a block share between two barriers.
//
// Derivatives, in the manner of Singh, Russell and Wensing (Efficient Analytical
// Derivatives of Rigid-Body Dynamics using Spatial Vector Algebra, IEEE RA-L 7(2),
// 2022). With psi_j the motion subspace of degree of freedom j in this
// form, v, a the velocity and acceleration (gravity included) of j's parent
// at j's origin,
//     psid_j = v x psi_j,   psidd_j = a x psi_j + v x psid_j,
//     eta_j  = 2 psid_j     (a free root: psid = 0, eta_j = v_0 x psi_j),
// and for body k  f_k = I a_k + v_k x* I v_k  and the velocity operator
//     2 B_k x = v_k x* (I x) - I (v_k x x) + x x* (I v_k).
// Displacing q_j moves j's subtree rigidly; the difference to moving the
// whole world is a velocity psid_j and an acceleration psidd_j + psid_j x v_k
// added to the subtree, so the force of the subtree changes by
//     psi_j x* f + I psidd_j + 2 B psid_j        (f, I, B summed over it),
// and adding to qd_j changes it by  I eta_j + 2 B psi_j.  Projected on
// psi_i this gives every entry of d tau / d q and d tau / d qd as dot products
// along the support paths (the analytic form of the derivatives that the
// paper names as the step after autograd, Sec. 3.5), and summed against a
// cotangent it gives the adjoint. Expanding 2 B for a rigid body (mass m,
// first moment h, inertia I_o about the origin, S = tr(I_o)/2 1 - I_o) shows
// that it acts on the angular part only:
//     2 B (w, u) = 2 (P w, p x w),
//     P = -[omega] S + (h . nu) 1 - nu h^T,   p = h x omega - m nu
// with v_k = (omega, nu), so a subtree's B is 12 numbers.
#pragma once

#include "adjoint.cuh"
#include "level.cuh"

namespace fst {

// motion about the parent's origin -> about the child's, and force back; r = child - parent
__device__ __forceinline__ SV shift_motion(SV m, f3 r) { return SV{m.w, m.v + cross(m.w, r)}; }
__device__ __forceinline__ SV shift_force(SV f, f3 r) { return SV{f.w + cross(r, f.v), f.v}; }

// A rigid-body inertia's axes rotated by R (no shift).
__device__ __forceinline__ In10 in_rotate(const float* R, const In10& I) {
  In10 o;
  o.m = I.m;
  o.h = Rmul(R, I.h);
  sym_rot(R, I.I, o.I);
  return o;
}

// The same body about the parent's origin, r = child - parent (parallel axes).
__device__ __forceinline__ In10 in_shift(const In10& I, f3 r) {
  In10 o;
  o.m = I.m;
  o.h = f3{fmaf(I.m, r.x, I.h.x), fmaf(I.m, r.y, I.h.y), fmaf(I.m, r.z, I.h.z)};
  const float d = fmaf(2.0f, dot(I.h, r), I.m * dot(r, r));
  const float hm = 0.5f * I.m;  // h r^T + r h^T + m r r^T = z r^T + r z^T
  const f3 z = f3{fmaf(hm, r.x, I.h.x), fmaf(hm, r.y, I.h.y), fmaf(hm, r.z, I.h.z)};
  o.I[0] = I.I[0] + fmaf(-2.0f * z.x, r.x, d);
  o.I[1] = I.I[1] - fmaf(z.x, r.y, r.x * z.y);
  o.I[2] = I.I[2] + fmaf(-2.0f * z.y, r.y, d);
  o.I[3] = I.I[3] - fmaf(z.x, r.z, r.x * z.z);
  o.I[4] = I.I[4] - fmaf(z.y, r.z, r.y * z.z);
  o.I[5] = I.I[5] + fmaf(-2.0f * z.z, r.z, d);
  return o;
}

// The motion subspace of a 1-DOF joint with its axes rotated
__device__ __forceinline__ SV psi_of(const BodyC& c, const float* R) {
  const SV s = S_of(c);
  return SV{Rmul(R, s.w), Rmul(R, s.v)};
}

__device__ __forceinline__ bool one_dof(const BodyI& b) {
  return b.type == FST_JOINT_REVOLUTE || b.type == FST_JOINT_PRISMATIC;
}

// S x with S = tr(I_o)/2 1 - I_o
__device__ __forceinline__ f3 second_moment_mul(const In10& I, f3 x) {
  const float ht = 0.5f * (I.I[0] + I.I[2] + I.I[5]);
  return ht * x - sym_mul(I.I, x);
}

// The velocity operator of a body or subtree (see above).
struct BOp {
  float P[9];
  f3 p;
};

__device__ __forceinline__ BOp b_of(const In10& I, SV v, SV hv) {
  BOp b;
  const float ht = 0.5f * (I.I[0] + I.I[2] + I.I[5]);
  // columns of -[omega] S: S column c crossed with omega
  const f3 s0 = f3{ht - I.I[0], -I.I[1], -I.I[3]};
  const f3 s1 = f3{-I.I[1], ht - I.I[2], -I.I[4]};
  const f3 s2 = f3{-I.I[3], -I.I[4], ht - I.I[5]};
  const f3 c0 = cross(s0, v.w), c1 = cross(s1, v.w), c2 = cross(s2, v.w);
  const float hn = dot(I.h, v.v);
  b.P[0] = c0.x + fmaf(-v.v.x, I.h.x, hn);
  b.P[1] = fmaf(-v.v.x, I.h.y, c1.x);
  b.P[2] = fmaf(-v.v.x, I.h.z, c2.x);
  b.P[3] = fmaf(-v.v.y, I.h.x, c0.y);
  b.P[4] = c1.y + fmaf(-v.v.y, I.h.y, hn);
  b.P[5] = fmaf(-v.v.y, I.h.z, c2.y);
  b.P[6] = fmaf(-v.v.z, I.h.x, c0.z);
  b.P[7] = fmaf(-v.v.z, I.h.y, c1.z);
  b.P[8] = c2.z + fmaf(-v.v.z, I.h.z, hn);
  b.p = -hv.v;
  return b;
}

// a += the child's operator b moved to the parent's origin
__device__ __forceinline__ void b_add_shifted(BOp& a, const BOp& b, f3 r) {
  const float rp = dot(r, b.p);
  a.P[0] += b.P[0] + fmaf(b.p.x, r.x, -rp);
  a.P[1] += fmaf(b.p.x, r.y, b.P[1]);
  a.P[2] += fmaf(b.p.x, r.z, b.P[2]);
  a.P[3] += fmaf(b.p.y, r.x, b.P[3]);
  a.P[4] += b.P[4] + fmaf(b.p.y, r.y, -rp);
  a.P[5] += fmaf(b.p.y, r.z, b.P[5]);
  a.P[6] += fmaf(b.p.z, r.x, b.P[6]);
  a.P[7] += fmaf(b.p.z, r.y, b.P[7]);
  a.P[8] += b.P[8] + fmaf(b.p.z, r.z, -rp);
  a.p = a.p + b.p;
}

// 2 B (w, .) as a force
__device__ __forceinline__ SV b_mul2(const BOp& b, f3 w) {
  return SV{2.f * Rmul(b.P, w), 2.f * cross(b.p, w)};
}
// The functional x -> psi . 2 B x, which only sees x's angular part
__device__ __forceinline__ f3 b_row2(const BOp& b, SV psi) {
  return 2.f * (RTmul(b.P, psi.w) + cross(psi.v, b.p));
}

// ---- dense derivatives of inverse dynamics ------------------------------------
// Floats of shared state per body and environment: psi 6 | psid 6 | psidd 6 |
// r 3 | then R 9, v 6, a 6 while the kinematics run down the tree, replaced
// in place by the body's (then its subtree's) I 10, f 6, P 9, p 3
// (kDerivState = 49).

// The mass matrix keeps only entries of related degrees of freedom: row c
// holds M_cc, then c's ancestors from the nearest to the root (DofLists), in
// shared memory as [entry][lane].
struct TreeMat {
  float* base;
  const int* off;   // first entry of each row
  const int* dep;   // entries of each row (the diagonal included)
  const int* anc;   // degree of freedom of each entry
  __device__ __forceinline__ float* at(int entry) const { return base + (entry << 5) + (threadIdx.x & 31); }
};

// d tau / d q and d tau / d qd, [nv][nv][B] each (either may be null), and
// with MASS the mass matrix into H, of one tile of 32 environments. The caller
// has staged q, qd and qdd.
template <bool MASS>
__device__ __forceinline__ void rnea_derivs_aligned(const SmemModel& tp, SV a0, const Col& q, const Col& qd,
                                                    const Col& qdd, int nv, const LaneState& S, const TreeMat& H,
                                                    float* __restrict__ dq, float* __restrict__ dqd, int64_t B,
                                                    int64_t e, bool act) {
  const int W = n_warps(), w = warp_id(), n = tp.n();
  enum { PSI = 0, PSD = 6, PSDD = 12, RR = 18, R_ = 21, V_ = 30, A_ = 36, I_ = 21, F_ = 31, P_ = 37, p_ = 46 };
  // structural zeros: entries of unrelated degrees of freedom
  const int64_t e0 = e - (threadIdx.x & 31);
  if (dq) m_clear_tile(dq, (int64_t)nv * nv, B, e0, W, w);
  if (dqd) m_clear_tile(dqd, (int64_t)nv * nv, B, e0, W, w);
  // joint transforms, all bodies at once
  for (int i = w; i < n; i += W) {
    const BodyI bi = tp.I(i);
    S.putX(i, R_, joint_X(tp.C(i), bi, q));  // R 9, t 3 (t in the V slot until the level pass reads it)
  }
  __syncthreads();
  // down the tree: rotations, velocities, accelerations, subspaces
  for (int l = 0; l < tp.depth(); ++l) {
    FST_FOR_MY_BODIES(tp, l, k) {
      const int i = tp.level_body(k);
      const BodyI bi = tp.I(i);
      const Xf X = S.X(i, R_);
      if (bi.type == FST_JOINT_FREE) {  // the root frame is this body's own
        const SV v0 = S_times(tp.C(i), bi, qd);
        const SV g{f3{0.f, 0.f, 0.f}, RTmul(X.R, a0.v)};
        const float Id[9] = {1.f, 0.f, 0.f, 0.f, 1.f, 0.f, 0.f, 0.f, 1.f};
        S.put_n(i, R_, Id, 9);
        S.put(i, V_, v0);
        S.put(i, A_, S_times(tp.C(i), bi, qdd) + g);
        S.put(i, PSI, v0);   // what its columns need later: v_0 and the gravity term
        S.put(i, PSD, g);
        continue;
      }
      float R[9];
      f3 r;
      SV vl = sv_zero(), al = a0;
      if (bi.parent < 0) {
#pragma unroll
        for (int c = 0; c < 9; ++c) R[c] = X.R[c];
        r = tvec(X);
      } else {
        float Rp[9];
        S.get_n(bi.parent, R_, Rp, 9);
        const float zero[3] = {0.f, 0.f, 0.f};
        float rr[3];
        compose(Rp, zero, X, R, rr);
        r = f3{rr[0], rr[1], rr[2]};
        vl = shift_motion(S.sv(bi.parent, V_), r);
        al = shift_motion(S.sv(bi.parent, A_), r);
      }
      const float rv[3] = {r.x, r.y, r.z};
      S.put_n(i, RR, rv, 3);
      S.put_n(i, R_, R, 9);
      if (one_dof(bi)) {
        const SV psi = psi_of(tp.C(i), R);
        const SV psd = crm(vl, psi);
        S.put(i, PSI, psi);
        S.put(i, PSD, psd);
        S.put(i, PSDD, crm(al, psi) + crm(vl, psd));
        al = sv_fma(qdd[bi.vi], psi, sv_fma(qd[bi.vi], psd, al));
        vl = sv_fma(qd[bi.vi], psi, vl);
      }
      S.put(i, V_, vl);
      S.put(i, A_, al);
    }
    __syncthreads();
  }
  // inertias, forces and velocity operators, all bodies at once
  for (int i = w; i < n; i += W) {
    float R[9];
    S.get_n(i, R_, R, 9);
    const SV v = S.sv(i, V_), a = S.sv(i, A_);
    const In10 I = in_rotate(R, in_load(tp.theta(i)));
    const SV hv = in_mul(I, v);
    const BOp b = b_of(I, v, hv);
    S.putin(i, I_, I);
    S.put(i, F_, in_mul(I, a) + crf(v, hv));
    S.put_n(i, P_, b.P, 9);
    const float pv[3] = {b.p.x, b.p.y, b.p.z};
    S.put_n(i, p_, pv, 3);
  }
  __syncthreads();
  // up the tree: sums over subtrees (the deepest level has no children)
  for (int l = tp.depth() - 2; l >= 0; --l) {
    FST_FOR_MY_BODIES(tp, l, k) {
      const int i = tp.level_body(k);
      const int c0 = tp.child_begin(i), c1 = tp.child_begin(i + 1);
      if (c0 == c1) continue;
      In10 I = S.in10(i, I_);
      SV f = S.sv(i, F_);
      BOp b;
      float t3[3];
      S.get_n(i, P_, b.P, 9);
      S.get_n(i, p_, t3, 3);
      b.p = f3{t3[0], t3[1], t3[2]};
      for (int ch = c0; ch < c1; ++ch) {
        const int c = tp.child(ch);
        S.get_n(c, RR, t3, 3);
        const f3 r = f3{t3[0], t3[1], t3[2]};
        in_add(I, in_shift(S.in10(c, I_), r));
        f = f + shift_force(S.sv(c, F_), r);
        BOp bc;
        S.get_n(c, P_, bc.P, 9);
        S.get_n(c, p_, t3, 3);
        bc.p = f3{t3[0], t3[1], t3[2]};
        b_add_shifted(b, bc, r);
      }
      S.putin(i, I_, I);
      S.put(i, F_, f);
      S.put_n(i, P_, b.P, 9);
      const float pv[3] = {b.p.x, b.p.y, b.p.z};
      S.put_n(i, p_, pv, 3);
    }
    __syncthreads();
  }
  // every pair of related degrees of freedom, from the deeper one up its
  // support path (deepest bodies first: they have the longest paths)
  float* const Q = dq && act ? dq + e : nullptr;
  float* const D = dqd && act ? dqd + e : nullptr;
  for (int it = w; it < n; it += W) {
    const int i = tp.level_body(n - 1 - it);
    const BodyI bi = tp.I(i);
    if (nv_of(bi.type) == 0) continue;
    const In10 I = S.in10(i, I_);
    BOp b;
    float t3[3];
    S.get_n(i, P_, b.P, 9);
    S.get_n(i, p_, t3, 3);
    b.p = f3{t3[0], t3[1], t3[2]};
    auto at = [&](int r, int c) { return ((int64_t)r * nv + c) * B; };
    if (bi.type == FST_JOINT_FREE) {  // the root's own 6 x 6 blocks, rows and columns [v; w]
      const SV v0 = S.sv(i, PSI), g = S.sv(i, PSD);
#pragma unroll 1
      for (int j = 0; j < 6; ++j) {
        SV psi = sv_zero();
        if (j < 3)
          (j == 0 ? psi.v.x : j == 1 ? psi.v.y : psi.v.z) = 1.f;
        else
          (j == 3 ? psi.w.x : j == 4 ? psi.w.y : psi.w.z) = 1.f;
        const SV cq = in_mul(I, crm(g, psi));
        const SV cd = in_mul(I, crm(v0, psi)) + b_mul2(b, psi.w);
        const SV cm = in_mul(I, psi);
        const float xq[6] = {cq.v.x, cq.v.y, cq.v.z, cq.w.x, cq.w.y, cq.w.z};
        const float xd[6] = {cd.v.x, cd.v.y, cd.v.z, cd.w.x, cd.w.y, cd.w.z};
        const float xm[6] = {cm.v.x, cm.v.y, cm.v.z, cm.w.x, cm.w.y, cm.w.z};
        if (MASS)  // row vi + j: the diagonal, then columns j - 1 .. 0
#pragma unroll
          for (int r = 0; r < 6; ++r)
            if (r <= j) *H.at(H.off[bi.vi + j] + j - r) = xm[r];
#pragma unroll
        for (int r = 0; r < 6; ++r) {
          const int64_t o = at(bi.vi + r, bi.vi + j);
          if (Q) Q[o] = xq[r];
          if (D) D[o] = xd[r];
        }
      }
      continue;
    }
    const int c = bi.vi;
    const SV psi = S.sv(i, PSI), psd = S.sv(i, PSD);
    SV t = in_mul(I, psi);
    SV uq = in_mul(I, S.sv(i, PSDD)) + b_mul2(b, psd.w);
    SV ud = 2.f * in_mul(I, psd) + b_mul2(b, psi.w);
    const f3 rw = b_row2(b, psi);
    if (Q) Q[at(c, c)] = dot(psi, uq);
    if (D) D[at(c, c)] = dot(psi, ud);
    float* hrow = MASS ? H.at(H.off[c]) : nullptr;  // the row's next entry
    if (MASS) {
      *hrow = dot(psi, t);
      hrow += 32;
    }
    uq = uq + crf(psi, S.sv(i, F_));
    int kk = i;
    for (int j = bi.parent; j >= 0; j = tp.I(j).parent) {
      S.get_n(kk, RR, t3, 3);
      const f3 r = f3{t3[0], t3[1], t3[2]};
      kk = j;
      t = shift_force(t, r);
      uq = shift_force(uq, r);
      ud = shift_force(ud, r);
      const BodyI bj = tp.I(j);
      if (one_dof(bj)) {
        const SV pj = S.sv(j, PSI), pdj = S.sv(j, PSD);
        if (Q) {
          Q[at(bj.vi, c)] = dot(pj, uq);
          Q[at(c, bj.vi)] = dot(t, S.sv(j, PSDD)) + dot(rw, pdj.w);
        }
        if (D) {
          D[at(bj.vi, c)] = dot(pj, ud);
          D[at(c, bj.vi)] = fmaf(2.f, dot(t, pdj), dot(rw, pj.w));
        }
        if (MASS) {
          *hrow = dot(pj, t);
          hrow += 32;
        }
      } else if (bj.type == FST_JOINT_FREE) {
        const SV v0 = S.sv(j, PSI), g = S.sv(j, PSD);
        const f3 z = cross(t.v, g.v);        // t . psidd of the angular directions
        const SV y = crf(v0, t);             // t . eta = -psi . (v0 x* t)
        const float uqr[6] = {uq.v.x, uq.v.y, uq.v.z, uq.w.x, uq.w.y, uq.w.z};
        const float udr[6] = {ud.v.x, ud.v.y, ud.v.z, ud.w.x, ud.w.y, ud.w.z};
        const float tr[6] = {t.v.x, t.v.y, t.v.z, t.w.x, t.w.y, t.w.z};
        const float zq[6] = {0.f, 0.f, 0.f, z.x, z.y, z.z};
        const float yd[6] = {-y.v.x, -y.v.y, -y.v.z, rw.x - y.w.x, rw.y - y.w.y, rw.z - y.w.z};
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          const int64_t up = at(bj.vi + k, c), left = at(c, bj.vi + k);
          if (Q) {
            Q[up] = uqr[k];
            Q[left] = zq[k];
          }
          if (D) {
            D[up] = udr[k];
            D[left] = yd[k];
          }
          if (MASS) hrow[(5 - k) * 32] = tr[k];  // the nearest ancestor is the root's last coordinate
        }
      }
    }
  }
}

// ---- the adjoint of inverse dynamics ------------------------------------------
// For the cotangent tbar of tau let w_k be the velocity that tbar would give
// body k as a joint velocity. Then L = sum_k w_k . f_k, and with f, A = I w and
// H = 2 B^T w (angular only, 3 numbers) summed over j's subtree
//     qbar_j   = (w x psi_j) . f + psidd_j . A + psid_j . H   (w of the parent)
//     qdbar_j  = eta_j . A + psi_j . H
//     qddbar_j = psi_j . A,
// so the reverse sweep is one sum of 15 numbers up the tree. The gradient in
// the inertial parameters is local to a body: the contraction of (w, a) and
// (w x v, v), turned back to body axes.
// Floats of shared state per body and environment (kVjpState = 51):
// psi 6 | R 9 | r 3 | v 6 | a 6 | w 6 | f 6 | A 6 | H 3.

// Where the cotangent comes from.
enum VjpMode {
  VJP_GIVEN = 0,  // staged in tb
  VJP_LOSS,       // tb holds measured torques; the cotangent is 2 (tau - tb), the loss their squared difference
};

struct VjpAligned {
  float* qbar;     // [nq][B] or null
  float* qdbar;    // [nv][B] or null
  float* qddbar;   // [nv][B] or null
  float* thbar;    // this tile's [n][10] partial sums in global memory, or null
  float sign;      // multiplies every cotangent
};

// Sums each of 10 values over the warp: halving the set of values a lane
// still carries at every step takes 16 shuffles instead of 50. The sum of
// value k ends in lanes whose bits 4, 3, 2, 1 spell k.
__device__ __forceinline__ void warp_sum10_store(const float* g, float* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  float v[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) v[k] = k < 10 ? g[k] : 0.f;
#pragma unroll
  for (int half = 8; half >= 1; half >>= 1) {
    const bool hi = lane & (2 * half);
#pragma unroll
    for (int k = 0; k < half; ++k) {
      const float send = hi ? v[k] : v[k + half];
      v[k] = (hi ? v[k + half] : v[k]) + __shfl_xor_sync(0xffffffffu, send, 2 * half);
    }
  }
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
  const int k = lane >> 1;
  if ((lane & 1) == 0 && k < 10) out[k] = v[0];
}

// d/dtheta of y . (I x), accumulated in g in the order of the 10 parameters,
// for vectors in the axes of the caller (theta_contract's formulas).
__device__ __forceinline__ void inertia_contract(SV y, SV x, float* g) {
  g[0] += dot(y.v, x.v);
  const f3 dh = cross(x.v, y.w) - cross(x.w, y.v);
  g[1] += dh.x;
  g[2] += dh.y;
  g[3] += dh.z;
  g[4] = fmaf(y.w.x, x.w.x, g[4]);
  g[5] = fmaf(y.w.x, x.w.y, fmaf(y.w.y, x.w.x, g[5]));
  g[6] = fmaf(y.w.y, x.w.y, g[6]);
  g[7] = fmaf(y.w.x, x.w.z, fmaf(y.w.z, x.w.x, g[7]));
  g[8] = fmaf(y.w.y, x.w.z, fmaf(y.w.z, x.w.y, g[8]));
  g[9] = fmaf(y.w.z, x.w.z, g[9]);
}

// The same gradient for the parameters in axes turned by R (in = R body).
__device__ __forceinline__ void inertia_grad_to_body(const float* R, float* g) {
  const f3 h = RTmul(R, f3{g[1], g[2], g[3]});
  g[1] = h.x;
  g[2] = h.y;
  g[3] = h.z;
  const float G[6] = {g[4], 0.5f * g[5], g[6], 0.5f * g[7], 0.5f * g[8], g[9]};
  const float Rt[9] = {R[0], R[3], R[6], R[1], R[4], R[7], R[2], R[5], R[8]};
  float o[6];
  sym_rot(Rt, G, o);
  g[4] = o[0];
  g[5] = 2.f * o[1];
  g[6] = o[2];
  g[7] = 2.f * o[3];
  g[8] = 2.f * o[4];
  g[9] = o[5];
}

// One tile of 32 environments. The caller has staged q, qd, qdd and
// tb ([nv] rows of 32; VJP_LOSS writes the cotangent there). Returns this thread's share of the loss (VJP_LOSS).
// BODY: the same in body axes, the joint transforms staying as they are: motions
// and forces are rotated and shifted from body to body, and inertias, subspaces
// and the parameter gradient not at all. The adjoint of ABA takes it: its errors
// against 64 bits are those of M^-1 and of the accelerations carried through this
// sweep, and where all three round the same transforms they partly cancel
// (q_bar, relative 2-norm, in body axes and in root axes after a body-frame M^-1:
// humanoid29 8.0e-7 and 1.36e-6, quadruped11 2.7e-7 and 4.7e-7). By itself the sweep
// is the more exact one in root axes.
template <int MODE, bool BODY = false>
__device__ __forceinline__ float rnea_vjp_aligned(const SmemModel& tp, SV a0, const Col& q, const Col& qd,
                                                  const Col& qdd, float* tbcol, const LaneState& S,
                                                  const VjpAligned& o, int64_t B, int64_t e, bool act) {
  const int W = n_warps(), w = warp_id(), n = tp.n();
  enum { PSI = 0, R_ = 6, RR = 15, V_ = 18, A_ = 24, W_ = 30, F_ = 36, AS_ = 42, H_ = 48 };
  static_assert(!BODY || MODE == VJP_GIVEN, "the loss runs in root axes");
  const Col tb{tbcol, kLaneEnvs};
  float loss = 0.f;
  for (int i = w; i < n; i += W) S.putX(i, R_, joint_X(tp.C(i), tp.I(i), q));  // R 9 | r 3
  __syncthreads();
  // down the tree: rotations, velocities, accelerations (and w when tb is known)
  for (int l = 0; l < tp.depth(); ++l) {
    FST_FOR_MY_BODIES(tp, l, k) {
      const int i = tp.level_body(k);
      const BodyI bi = tp.I(i);
      const Xf X = S.X(i, R_);
      if (bi.type == FST_JOINT_FREE) {  // the root frame is this body's own
        const float Id[9] = {1.f, 0.f, 0.f, 0.f, 1.f, 0.f, 0.f, 0.f, 1.f};
        if (!BODY) S.put_n(i, R_, Id, 9);
        S.put(i, V_, S_times(tp.C(i), bi, qd));
        S.put(i, A_, S_times(tp.C(i), bi, qdd) + SV{f3{0.f, 0.f, 0.f}, RTmul(X.R, a0.v)});
        if (MODE == VJP_GIVEN) S.put(i, W_, S_times(tp.C(i), bi, tb));
        continue;
      }
      SV vl = sv_zero(), al = a0, wl = sv_zero();
      float R[9];
      if (BODY) {
        if (bi.parent >= 0) {
          vl = X_motion(X, S.sv(bi.parent, V_));
          al = X_motion(X, S.sv(bi.parent, A_));
          wl = X_motion(X, S.sv(bi.parent, W_));
        } else {
          al = X_motion(X, a0);
        }
      } else if (bi.parent < 0) {
#pragma unroll
        for (int c = 0; c < 9; ++c) R[c] = X.R[c];
      } else {
        float Rp[9], rr[3];
        S.get_n(bi.parent, R_, Rp, 9);
        const float zero[3] = {0.f, 0.f, 0.f};
        compose(Rp, zero, X, R, rr);
        const f3 r = f3{rr[0], rr[1], rr[2]};
        S.put_n(i, RR, rr, 3);
        S.put_n(i, R_, R, 9);
        vl = shift_motion(S.sv(bi.parent, V_), r);
        al = shift_motion(S.sv(bi.parent, A_), r);
        if (MODE == VJP_GIVEN) wl = shift_motion(S.sv(bi.parent, W_), r);
      }
      if (one_dof(bi)) {
        const SV psi = BODY ? S_of(tp.C(i)) : psi_of(tp.C(i), R);
        if (!BODY) S.put(i, PSI, psi);
        const SV psd = crm(vl, psi);
        al = sv_fma(qdd[bi.vi], psi, sv_fma(qd[bi.vi], psd, al));
        vl = sv_fma(qd[bi.vi], psi, vl);
        if (MODE == VJP_GIVEN) wl = sv_fma(tb[bi.vi], psi, wl);
      }
      S.put(i, V_, vl);
      S.put(i, A_, al);
      if (MODE == VJP_GIVEN) S.put(i, W_, wl);
    }
    __syncthreads();
  }
  // the cotangent's velocity, force functionals and parameter gradient of a body
  auto local_adjoint = [&](int i, const float* R, const In10& I, SV v, SV a, SV hv) {
    const SV wv = S.sv(i, W_);
    S.put(i, AS_, in_mul(I, wv));
    const f3 H = 2.f * (second_moment_mul(I, cross(v.w, wv.w)) +
                        (dot(I.h, v.v) * wv.w - dot(v.v, wv.w) * I.h) - cross(wv.v, hv.v));
    const float Hn[3] = {H.x, H.y, H.z};
    S.put_n(i, H_, Hn, 3);
    if (o.thbar) {
      float g[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
      inertia_contract(wv, a, g);
      inertia_contract(crm(wv, v), v, g);
      if (!BODY) inertia_grad_to_body(R, g);
#pragma unroll
      for (int c = 0; c < 10; ++c) g[c] = act ? o.sign * g[c] : 0.f;
      warp_sum10_store(g, o.thbar + 10 * i);
    }
  };
  for (int i = w; i < n; i += W) {
    float R[9];
    if (!BODY) S.get_n(i, R_, R, 9);
    const SV v = S.sv(i, V_), a = S.sv(i, A_);
    const In10 I = BODY ? in_load(tp.theta(i)) : in_rotate(R, in_load(tp.theta(i)));
    const SV hv = in_mul(I, v);
    S.put(i, F_, in_mul(I, a) + crf(v, hv));
    if (MODE == VJP_GIVEN) local_adjoint(i, R, I, v, a, hv);
  }
  __syncthreads();
  if (MODE != VJP_GIVEN) {
    // forces up the tree, tau and the cotangent, then its velocity down the tree
    for (int l = tp.depth() - 1; l >= 0; --l) {
      FST_FOR_MY_BODIES(tp, l, k) {
        const int i = tp.level_body(k);
        const BodyI bi = tp.I(i);
        SV f = S.sv(i, F_);
        for (int ch = tp.child_begin(i); ch < tp.child_begin(i + 1); ++ch) {
          const int c = tp.child(ch);
          float t3[3];
          S.get_n(c, RR, t3, 3);
          f = f + shift_force(S.sv(c, F_), f3{t3[0], t3[1], t3[2]});
        }
        S.put(i, F_, f);
        const int ni = nv_of(bi.type);
        float tau[6];
        if (ni == 1) {
          tau[0] = dot(S.sv(i, PSI), f);
        } else {
          tau[0] = f.v.x, tau[1] = f.v.y, tau[2] = f.v.z;
          tau[3] = f.w.x, tau[4] = f.w.y, tau[5] = f.w.z;
        }
#pragma unroll
        for (int r = 0; r < 6; ++r) {
          if (r >= ni) break;
          float* tr = tbcol + (bi.vi + r) * kLaneEnvs;
          const float res = tau[r] - *tr;
          loss = fmaf(res, res, loss);
          *tr = 2.f * res;
        }
      }
      __syncthreads();
    }
    for (int l = 0; l < tp.depth(); ++l) {
      FST_FOR_MY_BODIES(tp, l, k) {
        const int i = tp.level_body(k);
        const BodyI bi = tp.I(i);
        SV wl = sv_zero();
        if (bi.type == FST_JOINT_FREE) {
          wl = S_times(tp.C(i), bi, tb);
        } else {
          if (bi.parent >= 0) {
            float t3[3];
            S.get_n(i, RR, t3, 3);
            wl = shift_motion(S.sv(bi.parent, W_), f3{t3[0], t3[1], t3[2]});
          }
          if (one_dof(bi)) wl = sv_fma(tb[bi.vi], S.sv(i, PSI), wl);
        }
        S.put(i, W_, wl);
      }
      __syncthreads();
    }
    for (int i = w; i < n; i += W) {
      float R[9];
      S.get_n(i, R_, R, 9);
      const SV v = S.sv(i, V_);
      const In10 I = in_rotate(R, in_load(tp.theta(i)));
      local_adjoint(i, R, I, v, S.sv(i, A_), in_mul(I, v));
    }
    __syncthreads();
  }
  if (!o.qbar && !o.qdbar && !o.qddbar) return loss;  // block-uniform: only the parameters were asked for
  // up the tree: A and H (and f where it has not been summed yet)
  for (int l = tp.depth() - 2; l >= 0; --l) {
    FST_FOR_MY_BODIES(tp, l, k) {
      const int i = tp.level_body(k);
      const int c0 = tp.child_begin(i), c1 = tp.child_begin(i + 1);
      if (c0 == c1) continue;
      SV f = S.sv(i, F_), A = S.sv(i, AS_);
      float H[3], t3[3];
      S.get_n(i, H_, H, 3);
      for (int ch = c0; ch < c1; ++ch) {
        const int c = tp.child(ch);
        if (BODY) {
          const Xf X = S.X(c, R_);
          A = A + XT_force(X, S.sv(c, AS_));
          f = f + XT_force(X, S.sv(c, F_));
          S.get_n(c, H_, t3, 3);
          const f3 h = Rmul(X.R, f3{t3[0], t3[1], t3[2]});
          H[0] += h.x;
          H[1] += h.y;
          H[2] += h.z;
          continue;
        }
        S.get_n(c, RR, t3, 3);
        const f3 r = f3{t3[0], t3[1], t3[2]};
        A = A + shift_force(S.sv(c, AS_), r);
        if (MODE == VJP_GIVEN) f = f + shift_force(S.sv(c, F_), r);
        S.get_n(c, H_, t3, 3);
        H[0] += t3[0];
        H[1] += t3[1];
        H[2] += t3[2];
      }
      S.put(i, AS_, A);
      S.put_n(i, H_, H, 3);
      if (MODE == VJP_GIVEN) S.put(i, F_, f);
    }
    __syncthreads();
  }
  if (!act) return loss;
  for (int i = w; i < n; i += W) {
    const BodyI bi = tp.I(i);
    if (nv_of(bi.type) == 0) continue;
    const SV A = S.sv(i, AS_);
    float t3[3];
    S.get_n(i, H_, t3, 3);
    const f3 H = f3{t3[0], t3[1], t3[2]};
    if (bi.type == FST_JOINT_FREE) {
      // v = S qd, a = X a0 + S qdd: q enters through gravity only
      const SV y = crf(S.sv(i, V_), A);  // eta . A = -psi . (v_0 x* A)
      const f3 g1 = RTmul(tp.C(i).R0, a0.v);
      const float G[9] = {g1.x * A.v.x, g1.x * A.v.y, g1.x * A.v.z, g1.y * A.v.x, g1.y * A.v.y,
                          g1.y * A.v.z, g1.z * A.v.x, g1.z * A.v.y, g1.z * A.v.z};
      float gq[4];
      quat_grad(q[bi.qi + 3], q[bi.qi + 4], q[bi.qi + 5], q[bi.qi + 6], G, gq);
      const float qo[7] = {0.f, 0.f, 0.f, gq[0], gq[1], gq[2], gq[3]};
      const float vo[6] = {-y.v.x, -y.v.y, -y.v.z, H.x - y.w.x, H.y - y.w.y, H.z - y.w.z};
      const float ao[6] = {A.v.x, A.v.y, A.v.z, A.w.x, A.w.y, A.w.z};
#pragma unroll
      for (int r = 0; r < 7; ++r) store_if(o.qbar, bi.qi + r, B, e, o.sign * qo[r], true);
#pragma unroll
      for (int r = 0; r < 6; ++r) {
        store_if(o.qdbar, bi.vi + r, B, e, o.sign * vo[r], true);
        store_if(o.qddbar, bi.vi + r, B, e, o.sign * ao[r], true);
      }
      continue;
    }
    SV vl = sv_zero(), al = a0, wl = sv_zero();
    if (BODY) {
      const Xf X = S.X(i, R_);
      if (bi.parent >= 0) {
        vl = X_motion(X, S.sv(bi.parent, V_));
        al = X_motion(X, S.sv(bi.parent, A_));
        wl = X_motion(X, S.sv(bi.parent, W_));
      } else {
        al = X_motion(X, a0);
      }
    } else if (bi.parent >= 0) {
      S.get_n(i, RR, t3, 3);
      const f3 r = f3{t3[0], t3[1], t3[2]};
      vl = shift_motion(S.sv(bi.parent, V_), r);
      al = shift_motion(S.sv(bi.parent, A_), r);
      wl = shift_motion(S.sv(bi.parent, W_), r);
    }
    const SV psi = BODY ? S_of(tp.C(i)) : S.sv(i, PSI);
    const SV psd = crm(vl, psi);
    const SV psdd = crm(al, psi) + crm(vl, psd);
    store_if(o.qbar, bi.qi, B, e,
             o.sign * (dot(crm(wl, psi), S.sv(i, F_)) + dot(psdd, A) + dot(psd.w, H)), true);
    store_if(o.qdbar, bi.vi, B, e, o.sign * fmaf(2.f, dot(psd, A), dot(psi.w, H)), true);
    store_if(o.qddbar, bi.vi, B, e, o.sign * dot(psi, A), true);
  }
  return loss;
}

// Barrier of one tile's warps in a (32, T, W) block: a named one for each
// tile, so that its tiles drift apart and one's arithmetic fills the other's
// waits.
__device__ __forceinline__ void tile_barrier() {
  asm volatile("barrier.sync %0, %1;" ::"r"((int)threadIdx.y + 1), "r"((int)(blockDim.x * blockDim.z)) : "memory");
}

// The same adjoint (VJP_GIVEN, the same arithmetic and bits) with 36 floats a
// body, so that two tiles of the humanoid share an SM: nothing is staged (a
// body's coordinates wait in the slots that its velocities will take), the
// inertia and the functionals are formed on the way up instead of stored
// between two sweeps, and a body's contribution to its parent takes the place
// of its own v, a and w, which only its children needed.
// psi 6 | v 6, a 6, w 6, then the force, A and H for the parent | R 9 | r 3.
__device__ __forceinline__ void rnea_vjp_lean(const SmemModel& tp, SV a0, const float* __restrict__ q,
                                              const float* __restrict__ qd, const float* __restrict__ qdd,
                                              const float* __restrict__ tbar, const LaneState& S, const VjpAligned& o,
                                              int64_t B, int64_t e, bool act) {
  const int W = n_warps(), w = warp_id(), n = tp.n();
  enum { PSI = 0, V_ = 6, A_ = 12, W_ = 18, R_ = 24, RR = 33 };
  const int64_t ec = act ? e : B - 1;
  for (int i = w; i < n; i += W) {
    const BodyI bi = tp.I(i);
    const int nqb = bi.type == FST_JOINT_FREE ? 7 : bi.type == FST_JOINT_FIXED ? 0 : 1, nvb = nv_of(bi.type);
    float qb[7];
#pragma unroll
    for (int k = 0; k < 7; ++k) qb[k] = k < nqb ? ld_input(q + (int64_t)(bi.qi + k) * B + ec) : 0.f;
    float x[3][6];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const int64_t at = (int64_t)(bi.vi + k) * B + ec;
      x[0][k] = k < nvb ? ld_input(qd + at) : 0.f;
      x[1][k] = k < nvb ? ld_input(qdd + at) : 0.f;
      x[2][k] = k < nvb ? ld_input(tbar + at) : 0.f;
    }
    BodyI b0 = bi;
    b0.qi = 0;
    S.putX(i, R_, joint_X(tp.C(i), b0, Col{qb, 1}));
    if (bi.type == FST_JOINT_FREE) {
#pragma unroll
      for (int c = 0; c < 3; ++c)
        S.put(i, V_ + 6 * c, SV{f3{x[c][3], x[c][4], x[c][5]}, f3{x[c][0], x[c][1], x[c][2]}});
    } else {
#pragma unroll
      for (int c = 0; c < 3; ++c) *S.at(i, V_ + 6 * c) = x[c][0];
    }
  }
  tile_barrier();
  auto barrier = [] { tile_barrier(); };
  struct Joint {
    int i;
    BodyI b;
    Xf X;
  };
  level_pass<false, true>(
      tp,
      [&](int i) { return Joint{i, tp.I(i), S.X(i, R_)}; },
      [&](const Joint& j) {
        const int i = j.i;
        const BodyI& bi = j.b;
        if (bi.type == FST_JOINT_FREE) {  // the root frame is this body's own; v and w are in place
          const float Id[9] = {1.f, 0.f, 0.f, 0.f, 1.f, 0.f, 0.f, 0.f, 1.f};
          S.put_n(i, R_, Id, 9);
          S.put(i, A_, S.sv(i, A_) + SV{f3{0.f, 0.f, 0.f}, RTmul(j.X.R, a0.v)});
          return;
        }
        SV vl = sv_zero(), al = a0, wl = sv_zero();
        float R[9];
        if (bi.parent < 0) {
#pragma unroll
          for (int c = 0; c < 9; ++c) R[c] = j.X.R[c];
        } else {
          float Rp[9], rr[3];
          S.get_n(bi.parent, R_, Rp, 9);
          const float zero[3] = {0.f, 0.f, 0.f};
          compose(Rp, zero, j.X, R, rr);
          const f3 r = f3{rr[0], rr[1], rr[2]};
          S.put_n(i, RR, rr, 3);
          S.put_n(i, R_, R, 9);
          vl = shift_motion(S.sv(bi.parent, V_), r);
          al = shift_motion(S.sv(bi.parent, A_), r);
          wl = shift_motion(S.sv(bi.parent, W_), r);
        }
        if (one_dof(bi)) {
          const SV psi = psi_of(tp.C(i), R);
          S.put(i, PSI, psi);
          const float xd = *S.at(i, V_);
          const SV psd = crm(vl, psi);
          al = sv_fma(*S.at(i, A_), psi, sv_fma(xd, psd, al));
          vl = sv_fma(xd, psi, vl);
          wl = sv_fma(*S.at(i, W_), psi, wl);
        }
        S.put(i, V_, vl);
        S.put(i, A_, al);
        S.put(i, W_, wl);
      },
      barrier);
  auto contract = [&](int i, const float* R, SV v, SV acc, SV wv) {
    float g[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    inertia_contract(wv, acc, g);
    inertia_contract(crm(wv, v), v, g);
    inertia_grad_to_body(R, g);
#pragma unroll
    for (int c = 0; c < 10; ++c) g[c] = act ? o.sign * g[c] : 0.f;
    warp_sum10_store(g, o.thbar + 10 * i);
  };
  if (!o.qbar && !o.qdbar && !o.qddbar) {  // uniform over the launch
    for (int i = w; o.thbar && i < n; i += W) {
      float R[9];
      S.get_n(i, R_, R, 9);
      contract(i, R, S.sv(i, V_), S.sv(i, A_), S.sv(i, W_));
    }
    return;
  }
  // A body's own force and functionals, its part of theta's gradient and what
  // its outputs take from its parent's velocities are formed before its level:
  // only the sums over the children and the outputs wait for it.
  struct Own {
    int i, ch, ch_end;
    BodyI b;
    SV f, A, psi, psd, psdd, cwp;
    f3 H, r;
  };
  level_pass<true, true>(
      tp,
      [&](int i) {
        Own s;
        s.i = i;
        s.b = tp.I(i);
        s.ch = tp.child_begin(i);
        s.ch_end = tp.child_begin(i + 1);
        const SV v = S.sv(i, V_), wv = S.sv(i, W_);
        float R[9];
        S.get_n(i, R_, R, 9);
        const In10 I = in_rotate(R, in_load(tp.theta(i)));
        const SV hv = in_mul(I, v), acc = S.sv(i, A_);
        if (o.thbar) contract(i, R, v, acc, wv);
        s.f = in_mul(I, acc) + crf(v, hv);
        s.A = in_mul(I, wv);
        s.H = 2.f * (second_moment_mul(I, cross(v.w, wv.w)) + (dot(I.h, v.v) * wv.w - dot(v.v, wv.w) * I.h) -
                     cross(wv.v, hv.v));
        const float* t = S.at(i, RR);
        s.r = f3{t[0], t[32], t[64]};
        if (one_dof(s.b)) {
          SV vl = sv_zero(), al = a0, wl = sv_zero();
          if (s.b.parent >= 0) {
            vl = shift_motion(S.sv(s.b.parent, V_), s.r);
            al = shift_motion(S.sv(s.b.parent, A_), s.r);
            wl = shift_motion(S.sv(s.b.parent, W_), s.r);
          }
          s.psi = S.sv(i, PSI);
          s.psd = crm(vl, s.psi);
          s.psdd = crm(al, s.psi) + crm(vl, s.psd);
          s.cwp = crm(wl, s.psi);
        }
        return s;
      },
      [&](const Own& s) {
        const int i = s.i;
        const BodyI& bi = s.b;
        SV f = s.f, A = s.A;
        f3 H = s.H;
        for (int ch = s.ch; ch < s.ch_end; ++ch) {
          const int c = tp.child(ch);
          const float* h = S.at(c, W_);
          A = A + S.sv(c, A_);
          f = f + S.sv(c, V_);
          H = H + f3{h[0], h[32], h[64]};
        }
        if (act && bi.type == FST_JOINT_FREE) {
          const SV y = crf(S.sv(i, V_), A);
          const f3 g1 = RTmul(tp.C(i).R0, a0.v);
          const float G[9] = {g1.x * A.v.x, g1.x * A.v.y, g1.x * A.v.z, g1.y * A.v.x, g1.y * A.v.y,
                              g1.y * A.v.z, g1.z * A.v.x, g1.z * A.v.y, g1.z * A.v.z};
          const float* qq = q + (int64_t)(bi.qi + 3) * B + e;
          float gq[4];
          quat_grad(ld_input(qq), ld_input(qq + B), ld_input(qq + 2 * B), ld_input(qq + 3 * B), G, gq);
          const float qo[7] = {0.f, 0.f, 0.f, gq[0], gq[1], gq[2], gq[3]};
          const float vo[6] = {-y.v.x, -y.v.y, -y.v.z, H.x - y.w.x, H.y - y.w.y, H.z - y.w.z};
          const float ao[6] = {A.v.x, A.v.y, A.v.z, A.w.x, A.w.y, A.w.z};
#pragma unroll
          for (int c = 0; c < 7; ++c) store_if(o.qbar, bi.qi + c, B, e, o.sign * qo[c], true);
#pragma unroll
          for (int c = 0; c < 6; ++c) {
            store_if(o.qdbar, bi.vi + c, B, e, o.sign * vo[c], true);
            store_if(o.qddbar, bi.vi + c, B, e, o.sign * ao[c], true);
          }
        } else if (act && one_dof(bi)) {
          store_if(o.qbar, bi.qi, B, e, o.sign * (dot(s.cwp, f) + dot(s.psdd, A) + dot(s.psd.w, H)), true);
          store_if(o.qdbar, bi.vi, B, e, o.sign * fmaf(2.f, dot(s.psd, A), dot(s.psi.w, H)), true);
          store_if(o.qddbar, bi.vi, B, e, o.sign * dot(s.psi, A), true);
        }
        if (bi.parent >= 0) {
          S.put(i, V_, shift_force(f, s.r));
          S.put(i, A_, shift_force(A, s.r));
          float* h = S.at(i, W_);
          h[0] = H.x;
          h[32] = H.y;
          h[64] = H.z;
        }
      },
      barrier);
}

// ---- the adjoint of forward kinematics -----------------------------------------
// Moving joint i turns and shifts its whole subtree as one rigid body, so of
// the poses' cotangents (Rbar_k, pbar_k) only the total force F = sum pbar_k
// and moment T = sum (R_k's columns x Rbar_k's columns) + moments of the pbar_k
// act on it: qbar_i = S_w . T + S_v . F, with T about body i's origin. Summing
// six numbers up the tree replaces twelve and two matrix products per body. A
// free root's quaternion sees the moment alone: qbar = 2 (0, T) (x) q.
// Floats of shared state per body and environment: world pose 12 | T 3, F 3.
__device__ __forceinline__ void fk_vjp_tile(const SmemModel& tp, const Col& q, const float* __restrict__ pbar,
                                            const LaneState& S, float* __restrict__ qbar, int64_t B, int64_t e,
                                            bool act) {
  const int W = n_warps(), w = warp_id(), n = tp.n();
  enum { P_ = 0, T_ = 12 };
  // the cotangents' local part needs the world rotation: run the poses first
  for (int l = 0; l < tp.depth(); ++l) {
    FST_FOR_MY_BODIES(tp, l, k) {
      const int i = tp.level_body(k);
      const BodyI bi = tp.I(i);
      const Xf X = joint_X(tp.C(i), bi, q);
      Xf P = X;
      if (bi.parent >= 0) {
        const Xf Pp = S.X(bi.parent, P_);
        compose(Pp.R, Pp.t, X, P.R, P.t);
      }
      S.putX(i, P_, P);
    }
    __syncthreads();
  }
  for (int i = w; i < n; i += W) {
    float g[12];
    const float* src = pbar + (int64_t)i * 12 * B + e;
#pragma unroll
    for (int k = 0; k < 12; ++k) g[k] = act ? ld_input(src + (int64_t)k * B) : 0.f;
    float R[9];
    S.get_n(i, P_, R, 9);
    SV f{f3{0.f, 0.f, 0.f}, f3{g[9], g[10], g[11]}};
#pragma unroll
    for (int c = 0; c < 3; ++c) f.w = f.w + cross(f3{R[c], R[3 + c], R[6 + c]}, f3{g[c], g[3 + c], g[6 + c]});
    S.put(i, T_, f);
  }
  __syncthreads();
  for (int l = tp.depth() - 1; l >= 0; --l) {
    FST_FOR_MY_BODIES(tp, l, k) {
      const int i = tp.level_body(k);
      const BodyI bi = tp.I(i);
      const BodyC& c = tp.C(i);
      const Xf P = S.X(i, P_);
      SV f = S.sv(i, T_);
      for (int ch = tp.child_begin(i); ch < tp.child_begin(i + 1); ++ch) {
        const float* t = S.at(tp.child(ch), P_ + 9);
        f = f + shift_force(S.sv(tp.child(ch), T_), f3{t[0] - P.t[0], t[32] - P.t[1], t[64] - P.t[2]});
      }
      S.put(i, T_, f);
      if (!act) continue;
      if (one_dof(bi)) {
        const SV psi = psi_of(c, P.R);
        qbar[(int64_t)bi.qi * B + e] = dot(psi, f);
      } else if (bi.type == FST_JOINT_FREE) {
        const f3 F = RTmul(c.R0, f.v), T = RTmul(c.R0, f.w);
        f3 v = f3{q[bi.qi + 3], q[bi.qi + 4], q[bi.qi + 5]};
        float s = q[bi.qi + 6];
        const float inv = rsqrtf(fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, s * s))));
        v = inv * v;
        s *= inv;
        const f3 gv = 2.f * inv * (s * T + cross(T, v));
        const float out[7] = {F.x, F.y, F.z, gv.x, gv.y, gv.z, -2.f * inv * dot(T, v)};
#pragma unroll
        for (int r = 0; r < 7; ++r) qbar[(int64_t)(bi.qi + r) * B + e] = out[r];
      }
    }
    __syncthreads();
  }
}

// ---- forward-dynamics derivatives: the tree-sparse factorisation ----------------
// M = L^T D L with L unit lower triangular and as sparse as the tree: an
// elimination from the leaves to the roots fills no entry of unrelated degrees
// of freedom (Featherstone, Rigid Body Dynamics Algorithms, Sec. 6.5). Rows of
// one depth are independent; a row's updates all come from one warp (row mod
// W), so the block needs one barrier per depth. On return H holds L below the
// diagonal and 1 / D on it.
__device__ __forceinline__ void axpy_rows(float x, const float* src, float* dst, int n) {
  // dst += x src, four rows at a time: src and dst never overlap, which the
  // compiler cannot know, so the loads are issued ahead of the stores by hand
  int b = 0;
  for (; b + 4 <= n; b += 4, src += 128, dst += 128) {
    const float s0 = src[0], s1 = src[32], s2 = src[64], s3 = src[96];
    const float d0 = dst[0], d1 = dst[32], d2 = dst[64], d3 = dst[96];
    dst[0] = fmaf(x, s0, d0);
    dst[32] = fmaf(x, s1, d1);
    dst[64] = fmaf(x, s2, d2);
    dst[96] = fmaf(x, s3, d3);
  }
  for (; b < n; ++b, src += 32, dst += 32) *dst = fmaf(x, *src, *dst);
}

__device__ __forceinline__ void tree_factor(const TreeMat& H, const int* order, const int* level, int dof_depth) {
  const int W = n_warps(), w = warp_id();
  for (int l = dof_depth - 1; l >= 0; --l) {
    for (int s = level[l]; s < level[l + 1]; ++s) {
      const int k = order[s], o = H.off[k], d = H.dep[k];
      const float inv = 1.0f / fmaxf(*H.at(o), 1e-30f);
      for (int a = 1; a < d; ++a) {
        const int i = H.anc[o + a];
        if (i % W != w) continue;
        const float x = *H.at(o + a) * inv;
        axpy_rows(-x, H.at(o + a), H.at(H.off[i]), d - a);
      }
    }
    __syncthreads();
    // scale the finished rows (every warp has read them)
    for (int s = level[l] + w; s < level[l + 1]; s += W) {
      const int k = order[s], o = H.off[k], d = H.dep[k];
      const float inv = 1.0f / fmaxf(*H.at(o), 1e-30f);
      *H.at(o) = inv;
      for (int a = 1; a < d; ++a) *H.at(o + a) *= inv;
    }
  }
  __syncthreads();
}

// x := M^-1 x for NC columns held as [nv][32] in shared memory, one after the
// other `ld` floats apart (this lane's element of row i at x[i * 32]).
// Children have larger indices than their ancestors.
template <int NC>
__device__ __forceinline__ void tree_solve(const TreeMat& H, int nv, float* x, int ld) {
  for (int i = nv - 1; i >= 0; --i) {  // L^T y = x, from the leaves
    const int o = H.off[i], d = H.dep[i];
    float xi[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) xi[c] = x[c * ld + (i << 5)];
    int a = 1;
    for (; a + 4 <= d; a += 4) {  // distinct ancestors: all loads ahead of the stores
      int j[4];
      float l[4], t[4][NC];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        j[u] = H.anc[o + a + u] << 5;
        l[u] = *H.at(o + a + u);
#pragma unroll
        for (int c = 0; c < NC; ++c) t[u][c] = x[c * ld + j[u]];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int c = 0; c < NC; ++c) x[c * ld + j[u]] = fmaf(-l[u], xi[c], t[u][c]);
    }
    for (; a < d; ++a) {
      const int j = H.anc[o + a] << 5;
      const float l = *H.at(o + a);
#pragma unroll
      for (int c = 0; c < NC; ++c) x[c * ld + j] = fmaf(-l, xi[c], x[c * ld + j]);
    }
  }
  for (int i = 0; i < nv; ++i) {  // D, then L x = y, from the roots
    const int o = H.off[i], d = H.dep[i];
    const float inv = *H.at(o);
    float s[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) s[c] = x[c * ld + (i << 5)] * inv;
#pragma unroll 4
    for (int a = 1; a < d; ++a) {
      const int j = H.anc[o + a] << 5;
      const float l = *H.at(o + a);
#pragma unroll
      for (int c = 0; c < NC; ++c) s[c] = fmaf(-l, x[c * ld + j], s[c]);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) x[c * ld + (i << 5)] = s[c];
  }
}

}  // namespace fst
