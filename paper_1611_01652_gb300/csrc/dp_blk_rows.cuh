// The reverse pass' stages of the compiled topologies (quadruped, arms): the same blocks and items as
// in dp_blk_bwd.cuh, with one accumulator per row and body side, and every sum formed row by row in
// slot order with one rounding each.
//
// Why rows and not items: the controller's reverse carries its deltas as two bfloat16 planes (16
// significant bits). A last-bit difference in an output adjoint falls the other way in the low plane
// now and then, 2^-17 of a delta, and a hundred steps of back-propagation through an ill-conditioned
// robot amplify that to 1e-5 and more of the initial state's adjoint. Item by item (as dp_blk_bwd.cuh
// sums robots without a compiled topology) the gradients are as exact, but not those that the
// sequential walk over the rows gives: of 36 batches of 1500 recurrent quadrupeds over 100 steps, 16
// were more than 2e-5 of the adjoint's norm away, up to 4.6e-4. Here every sum is that of the sequential
// walk, so schedules, warps and layouts do not show in it; state, weight, mass and inertia gradients of
// 138 batches (recurrent, feed-forward and wide quadrupeds, arms) have its bits.
// What it costs, us with rollout, against the sums by items: quadruped 100 steps 27487 -> 28748, 1000
// steps warm 165907 -> 176146, recurrent 19462 -> 20427, wide 17182 -> 17600, arms 227721 -> 235395.
// Bound: issue and latency of the blocks' chains, as in dp_blk_bwd.cuh.
//
// Products with a coordinate axis' zeros are left out (exact zeros); where a sum's order of rounding
// matters it is written out.
#pragma once
#include "dp_blk_fwd.cuh"

// Accumulators behind a joint's record (from JR_N on): per linear row k, from JX_LIN + 7 k, the two
// components of the parent's and the child's angular adjoint that are not along axis k (cyclic order),
// the effective mass' adjoint (the parent's share with bias and impulse; the child's apart, added
// afterwards) and the bias'; per angular row from JX_ANG + 9 k, and for limit and servo row, both
// angular adjoints in full, then the same three (the servo row also its bound's).
enum { JX_LIN = 0, JX_ANG = 21, JX_LIM = 39, JX_MOT = 48, JX_N = 58 };
enum { LX_A = 0, LX_B = 2, LX_ME = 4, LX_MEB = 5, LX_BI = 6 };
enum { AX_A = 0, AX_B = 3, AX_ME = 6, AX_MEB = 7, AX_BI = 8, AX_BND = 9 };
// Contact (from CR_N on): row m from 4 m: two components, effective mass, bias (normal row) or bound.
enum { CX_A = 0, CX_ME = 2, CX_BI = 3, CX_N = 12 };
// Packages over the records; lever arms and angular directions stay where they are (fields 0 to 11, 0
// to 2). Joint: per linear row rab, rbb and two components each of Kb angA, Kb angB; per angular row
// the adjoint of t, that of ub and Kb t; Kb u of limit and servo row; anchors, tau, child axis; masses.
enum { XP_LIN = 12, XP_ANG = 42, XP_LIM = 60, XP_MOT = 63, XP_ANCA = 66, XP_ANCB = 69, XP_TAU = 72, XP_AXB = 78, XP_KB = 81, XP_N = 84 };
enum { XC_KA = 3, XC_N = 9, XC_T1 = 12, XC_T2 = 14, XC_V = 16, XC_OFF = 17, XC_KB = 20, XC_SIZE = 23 };
enum { XH_W = 0, XH_WA = 3, XH_WB = 6, XH_UB = 9, XH_REFA = 12, XH_REFB = 15, XH_AXA = 18, XH_SIZE = 21 };
static_assert(RX_REC_J >= JR_N + JX_N && RX_REC_J >= XP_N && RX_REC_J >= XH_SIZE && RX_REC_C >= CR_N + CX_N && RX_REC_C >= XC_SIZE, "a package must fit in its record");

// dotx and symx (dp_blk.cuh) of r x e_K with a vector and a matrix.
template <int K>
__device__ __forceinline__ float dotx_axis(float3 r, float3 w) {
  if (K == 0) return fmaf(-r.y, w.z, __fmul_rn(r.z, w.y));
  if (K == 1) return fmaf(r.x, w.z, __fmul_rn(-r.z, w.x));
  return fmaf(r.y, w.x, __fmul_rn(-r.x, w.y));
}
template <int K>
__device__ __forceinline__ float3 symx_axis(const float (&s)[6], float3 r) {
  if (K == 0)  // (0, r.z, -r.y)
    return f3(fmaf(s[2], -r.y, __fmul_rn(s[1], r.z)), fmaf(s[4], -r.y, __fmul_rn(s[3], r.z)), fmaf(s[5], -r.y, __fmul_rn(s[4], r.z)));
  if (K == 1)  // (-r.z, 0, r.x)
    return f3(fmaf(s[2], r.x, __fmul_rn(s[0], -r.z)), fmaf(s[4], r.x, __fmul_rn(s[1], -r.z)), fmaf(s[5], r.x, __fmul_rn(s[2], -r.z)));
  return f3(fmaf(s[0], r.y, __fmul_rn(s[1], -r.x)), fmaf(s[1], r.y, __fmul_rn(s[3], -r.x)), fmaf(s[4], -r.x, __fmul_rn(s[2], r.y)));
}
// q += g (x) a, row-major 3 x 3; in the second form a = r x e_K.
__device__ __forceinline__ void outer9(float (&q)[9], float3 g, float3 a) {
  q[0] = fmaf(g.x, a.x, q[0]); q[1] = fmaf(g.x, a.y, q[1]); q[2] = fmaf(g.x, a.z, q[2]);
  q[3] = fmaf(g.y, a.x, q[3]); q[4] = fmaf(g.y, a.y, q[4]); q[5] = fmaf(g.y, a.z, q[5]);
  q[6] = fmaf(g.z, a.x, q[6]); q[7] = fmaf(g.z, a.y, q[7]); q[8] = fmaf(g.z, a.z, q[8]);
}
template <int K>
__device__ __forceinline__ void outer9_axis(float (&q)[9], float3 g, float3 r) {
  constexpr int i = (K + 1) % 3, j = (K + 2) % 3;  // r x e_K = r_j e_i - r_i e_j
  const float ai = j == 0 ? r.x : (j == 1 ? r.y : r.z), aj = -(i == 0 ? r.x : (i == 1 ? r.y : r.z));
  q[i] = fmaf(g.x, ai, q[i]); q[j] = fmaf(g.x, aj, q[j]);
  q[3 + i] = fmaf(g.y, ai, q[3 + i]); q[3 + j] = fmaf(g.y, aj, q[3 + j]);
  q[6 + i] = fmaf(g.z, ai, q[6 + i]); q[6 + j] = fmaf(g.z, aj, q[6 + j]);
}
// q += (k a) (x) a with a = sg r x e_K: ki, kj the two components of k a.
template <int K>
__device__ __forceinline__ void outer4_axis(float (&q)[9], float ki, float kj, float3 r, float sg) {
  constexpr int i = (K + 1) % 3, j = (K + 2) % 3;
  const float ai = sg * (j == 0 ? r.x : (j == 1 ? r.y : r.z)), aj = -sg * (i == 0 ? r.x : (i == 1 ? r.y : r.z));
  q[3 * i + i] = fmaf(ki, ai, q[3 * i + i]); q[3 * i + j] = fmaf(ki, aj, q[3 * i + j]);
  q[3 * j + i] = fmaf(kj, ai, q[3 * j + i]); q[3 * j + j] = fmaf(kj, aj, q[3 * j + j]);
}
// Component c of a vector, c known at compile time.
template <int C>
__device__ __forceinline__ float comp(float3 v) { return C == 0 ? v.x : (C == 1 ? v.y : v.z); }
template <int K>
__device__ __forceinline__ float comp_i(float3 v) { return comp<(K + 1) % 3>(v); }
template <int K>
__device__ __forceinline__ float comp_j(float3 v) { return comp<(K + 2) % 3>(v); }

// One body of a block: velocities, their adjoints, inverse mass and inertia, and the running sums of
// the adjoints of those (q: of the inverse inertia).
struct RowBody {
  float3 v, w, vb, wb;
  float im, imb, ii[6], q[9];
};
__device__ __forceinline__ void rx_init(const DevTopo& T, const SL& S, int b, RowBody& B) {
  B.v = B.w = B.vb = B.wb = f3(0.f, 0.f, 0.f);
  B.im = B.imb = 0.f;
#pragma unroll
  for (int k = 0; k < 6; ++k) B.ii[k] = 0.f;
#pragma unroll
  for (int k = 0; k < 9; ++k) B.q[k] = 0.f;
  if (b < 0) return;
  B.im = S[T.sm_invm + b];
  load6(S, T.sm_iinv + 6 * b, B.ii);
}
__device__ __forceinline__ void rx_load(const DevTopo& T, const SL& S, const SL& VW, int b, RowBody& B) {
  if (b < 0) return;
  B.v = VW.v3(6 * b);
  B.w = VW.v3(6 * b + 3);
  B.vb = S.v3(T.sm_vb + 6 * b);
  B.wb = S.v3(T.sm_vb + 6 * b + 3);
  B.imb = S[T.sm_invmb + b];
#pragma unroll
  for (int k = 0; k < 9; ++k) B.q[k] = S[T.sm_iinvb + 9 * b + k];
}
__device__ __forceinline__ void rx_store(const DevTopo& T, const SL& S, const SL& VW, int b, const RowBody& B, bool lin) {
  if (b < 0) return;
  if (lin) {
    VW.s3(6 * b, B.v);
    S.s3(T.sm_vb + 6 * b, B.vb);
    S[T.sm_invmb + b] = B.imb;
  }
  VW.s3(6 * b + 3, B.w);
  S.s3(T.sm_vb + 6 * b + 3, B.wb);
#pragma unroll
  for (int k = 0; k < 9; ++k) S[T.sm_iinvb + 9 * b + k] = B.q[k];
}

// One linear row of a joint (world: its parent is the world, a body of zeros). lam: the impulse's
// adjoint; acc: what the row adds to its accumulators (components and bias); me_a, me_b: the sums of
// the effective mass' adjoint.
template <int K>
__device__ __forceinline__ void rx_lin(const DevTopo& T, bool world, float la, float lb, float me, float bi, float3 ra,
                                       float3 rb, RowBody& A, RowBody& B, float& lam, float& me_a, float& me_b,
                                       float (&acc)[5]) {
  const float dl = la - lb;
  const float3 IA = symx_axis<K>(A.ii, ra), IB = -symx_axis<K>(B.ii, rb);
  const float da = fmaf(A.im, axis_of<K>(A.vb), dotx(IA, A.wb));
  const float dbar = __fadd_rn(da, fmaf(-B.im, axis_of<K>(B.vb), dotx(IB, B.wb)));
  const float pbar = __fadd_rn(lam, dbar), jvb = __fmul_rn(-me, pbar);
  lam = fmaf(pbar, fmaf(-me, T.gamma, 1.f), -dbar);
  // velocities before the row
  axis_of<K>(A.v) = fmaf(-dl, A.im, axis_of<K>(A.v));
  A.w = axpy3(-dl, IA, A.w);
  axis_of<K>(B.v) = fmaf(dl, B.im, axis_of<K>(B.v));
  B.w = axpy3(-dl, IB, B.w);
  const float3 ga = f3(__fmul_rn(dl, A.wb.x), __fmul_rn(dl, A.wb.y), __fmul_rn(dl, A.wb.z));
  const float3 gb = f3(__fmul_rn(dl, B.wb.x), __fmul_rn(dl, B.wb.y), __fmul_rn(dl, B.wb.z));
  const float3 ua = symx(A.ii, ga), ub = symx(B.ii, gb);
  acc[0] = fmaf(jvb, comp_i<K>(A.w), comp_i<K>(ua));
  acc[1] = fmaf(jvb, comp_j<K>(A.w), comp_j<K>(ua));
  acc[2] = fmaf(jvb, comp_i<K>(B.w), comp_i<K>(ub));
  acc[3] = fmaf(jvb, comp_j<K>(B.w), comp_j<K>(ub));
  acc[4] = jvb;
  outer9_axis<K>(A.q, ga, ra);
  outer9_axis<K>(B.q, -gb, rb);
  A.imb = fmaf(dl, axis_of<K>(A.vb), A.imb);
  B.imb = fmaf(-dl, axis_of<K>(B.vb), B.imb);
  const float jva = __fadd_rn(axis_of<K>(A.v), dotx_axis<K>(ra, A.w));
  const float jvc = __fsub_rn(-dotx_axis<K>(rb, B.w), axis_of<K>(B.v));
  me_a = fmaf(-pbar, fmaf(T.gamma, lb, __fadd_rn(world ? jvc : jva, bi)), me_a);
  if (!world) me_b = fmaf(-pbar, jvc, me_b);
  axis_of<K>(A.vb) = __fadd_rn(axis_of<K>(A.vb), jvb);
  axis_of<K>(B.vb) = __fsub_rn(axis_of<K>(B.vb), jvb);
  A.wb = axpy3(jvb, cross_axis<K>(ra), A.wb);
  B.wb = axpy3(jvb, -cross_axis<K>(rb), B.wb);
}
// A row without a linear part, J_wa = -d, J_wb = d (angular, limit and servo rows). br: the clamp branch
// (0 inside); lbar: the clamped impulse's adjoint; ca, cb: what it adds to the two angular adjoints.
__device__ __forceinline__ float rx_ang(const DevTopo& T, bool world, float la, float lb, float me, float bi, int br, float3 d,
                                        RowBody& A, RowBody& B, float& lam, float& me_a, float& me_b, float& lbar, float3& ca,
                                        float3& cb) {
  const float dl = la - lb;
  const float3 IA = symx(A.ii, -d), IB = symx(B.ii, d);
  const float dbar = __fadd_rn(dotx(IA, A.wb), dotx(IB, B.wb));
  lbar = __fadd_rn(lam, dbar);
  const float pbar = br == 0 ? lbar : 0.f, jvb = __fmul_rn(-me, pbar);
  lam = fmaf(pbar, fmaf(-me, T.gamma, 1.f), -dbar);
  A.w = axpy3(-dl, IA, A.w);
  B.w = axpy3(-dl, IB, B.w);
  const float3 ga = f3(__fmul_rn(dl, A.wb.x), __fmul_rn(dl, A.wb.y), __fmul_rn(dl, A.wb.z));
  const float3 gb = f3(__fmul_rn(dl, B.wb.x), __fmul_rn(dl, B.wb.y), __fmul_rn(dl, B.wb.z));
  ca = axpy3(jvb, A.w, symx(A.ii, ga));
  cb = axpy3(jvb, B.w, symx(B.ii, gb));
  outer9(A.q, ga, -d);
  outer9(B.q, gb, d);
  const float jva = dotx(-d, A.w), jvc = dotx(d, B.w);
  me_a = fmaf(-pbar, fmaf(T.gamma, lb, __fadd_rn(world ? jvc : jva, bi)), me_a);
  if (!world) me_b = fmaf(-pbar, jvc, me_b);
  A.wb = axpy3(jvb, -d, A.wb);
  B.wb = axpy3(jvb, d, B.wb);
  return jvb;
}

// Blocks, last row first (see rev_joint and its neighbours in dp_blk_bwd.cuh for what is loaded when). A
// joint's five rows and a contact's three are one block each (plan_blocks sees to it).
template <class TP, class RD>
__device__ __forceinline__ void rx_joint(const DevTopo& T, const SL& S, const TP& tp, const BlkOp& op, const SL& R, RowBody& A,
                                         RowBody& B, const RD& ready) {
  const int s0 = op.slot();
  const bool world = op.a() < 0;
  const SL Q = R.at(JR_N);
  const float3 ra = R.v3(JF_RA), rb = R.v3(JF_RB);
  float la[5], lb[5], lam[5], me[5], bi[5], mea[5], meb[5], acc[3][5], bia[2];
  float3 t[2], ca[2], cb[2];
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const int f = k < 3 ? JX_LIN + 7 * k + LX_ME : JX_ANG + 9 * (k - 3) + AX_ME;
    la[k] = tp.la[s0 + k];
    lb[k] = tp.lb[s0 + k];
    lam[k] = S[T.sm_lam + s0 + k];
    me[k] = R[JF_ME + k];
    bi[k] = R[JF_BI + k];
    mea[k] = Q[f];
    meb[k] = Q[f + 1];
    if (k >= 3) t[k - 3] = R.v3(JF_T + 3 * (k - 3));
  }
  ready();
  float unused;
#pragma unroll
  for (int k = 4; k >= 3; --k)
    bia[k - 3] = rx_ang(T, world, la[k], lb[k], me[k], bi[k], 0, -t[k - 3], A, B, lam[k], mea[k], meb[k], unused, ca[k - 3], cb[k - 3]);
  rx_lin<2>(T, world, la[2], lb[2], me[2], bi[2], ra, rb, A, B, lam[2], mea[2], meb[2], acc[2]);
  rx_lin<1>(T, world, la[1], lb[1], me[1], bi[1], ra, rb, A, B, lam[1], mea[1], meb[1], acc[1]);
  rx_lin<0>(T, world, la[0], lb[0], me[0], bi[0], ra, rb, A, B, lam[0], mea[0], meb[0], acc[0]);
  // (every row's accumulators are its own block's: the loads here wait for nothing)
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const SL q = Q.at(JX_LIN + 7 * k);
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[k][c] += q[c];
    acc[k][4] += q[LX_BI];
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const SL q = Q.at(JX_ANG + 9 * k);
    ca[k] = q.v3(AX_A) + ca[k];
    cb[k] = q.v3(AX_B) + cb[k];
    bia[k] += q[AX_BI];
  }
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const SL q = Q.at(k < 3 ? JX_LIN + 7 * k : JX_ANG + 9 * (k - 3));
    S[T.sm_lam + s0 + k] = lam[k];
    if (k < 3) {
#pragma unroll
      for (int c = 0; c < 4; ++c) q[c] = acc[k][c];
      q[LX_ME] = mea[k];
      q[LX_MEB] = meb[k];
      q[LX_BI] = acc[k][4];
    } else {
      q.s3(AX_A, ca[k - 3]);
      q.s3(AX_B, cb[k - 3]);
      q[AX_ME] = mea[k];
      q[AX_MEB] = meb[k];
      q[AX_BI] = bia[k - 3];
    }
  }
}
template <class TP, class RD>
__device__ __forceinline__ void rx_hinge(const DevTopo& T, const SL& S, const TP& tp, const BlkOp& op, const SL& R, RowBody& A,
                                         RowBody& B, const RD& ready) {
  const bool lim = op.type() == BT_LIMIT;
  const int s = op.slot(), m = lim ? 5 : 6;
  const SL Q = R.at(JR_N + (lim ? JX_LIM : JX_MOT));
  const float sg = lim ? R[JF_LS] : 1.f;
  const int br = tp.br[s * 32];
  const float me = R[JF_ME + m], bi = R[JF_BI + m], la = tp.la[s], lb = tp.lb[s];
  const float3 d = sg * S.v3(T.sm_ua + 3 * op.idx());
  const float3 a0 = Q.v3(AX_A), b0 = Q.v3(AX_B);
  const float bi0 = Q[AX_BI], bnd0 = lim ? 0.f : Q[AX_BND];
  float lam = S[T.sm_lam + s], mea = Q[AX_ME], meb = Q[AX_MEB], lbar;
  float3 ca, cb;
  ready();
  const float jvb = rx_ang(T, op.a() < 0, la, lb, me, bi, br, d, A, B, lam, mea, meb, lbar, ca, cb);
  S[T.sm_lam + s] = lam;
  Q.s3(AX_A, a0 + ca);
  Q.s3(AX_B, b0 + cb);
  Q[AX_ME] = mea;
  Q[AX_MEB] = meb;
  Q[AX_BI] = bi0 + jvb;
  if (!lim) Q[AX_BND] = bnd0 + (br == 2 ? 1.f : (br == 1 ? -1.f : 0.f)) * lbar;
}
template <class TP, class RD>
__device__ __forceinline__ void rx_contact(const DevTopo& T, const SL& S, const TP& tp, const BlkOp& op, const SL& R, RowBody& A,
                                           const RD& ready) {
  const int s0 = op.slot();
  const SL Q = R.at(CR_N);
  float la[3], lb[3], lam[3], me[3], mea[3], acc[3][3];
  int br[3];
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    la[m] = tp.la[s0 + m];
    lb[m] = tp.lb[s0 + m];
    br[m] = tp.br[(s0 + m) * 32];
    lam[m] = S[T.sm_lam + s0 + m];
    me[m] = R[CF_ME + m];
    mea[m] = Q[4 * m + CX_ME];
  }
  const float3 ra = R.v3(CF_RA);
  const float mu = R[CF_MU], bias0 = R[CF_BI];
  ready();
  const float lnrm = la[0];  // the normal impulse a friction row saw (the normal row comes first)
  auto row = [&](auto MI, auto AI, float bias) {
    constexpr int m = decltype(MI)::value, K = decltype(AI)::value;
    const float dl = la[m] - lb[m];
    const float3 IA = symx_axis<K>(A.ii, ra);
    const float dbar = fmaf(A.im, axis_of<K>(A.vb), dotx(IA, A.wb));
    const float lbar = __fadd_rn(lam[m], dbar);
    const float pbar = br[m] == 0 ? lbar : 0.f, jvb = __fmul_rn(-me[m], pbar);
    acc[m][2] = jvb;
    if (m > 0) {
      const float sg = br[m] == 2 ? 1.f : (br[m] == 1 ? -1.f : 0.f);
      acc[m][2] = sg * lnrm * lbar;
      lam[0] = fmaf(sg * mu, lbar, lam[0]);
    }
    lam[m] = fmaf(pbar, fmaf(-me[m], T.gamma, 1.f), -dbar);
    axis_of<K>(A.v) = fmaf(-dl, A.im, axis_of<K>(A.v));
    A.w = axpy3(-dl, IA, A.w);
    const float3 g = f3(__fmul_rn(dl, A.wb.x), __fmul_rn(dl, A.wb.y), __fmul_rn(dl, A.wb.z));
    const float3 u = symx(A.ii, g);
    acc[m][0] = fmaf(jvb, comp_i<K>(A.w), comp_i<K>(u));
    acc[m][1] = fmaf(jvb, comp_j<K>(A.w), comp_j<K>(u));
    outer9_axis<K>(A.q, g, ra);
    A.imb = fmaf(dl, axis_of<K>(A.vb), A.imb);
    const float jv = __fadd_rn(axis_of<K>(A.v), dotx_axis<K>(ra, A.w));
    mea[m] = fmaf(-pbar, fmaf(T.gamma, lb[m], __fadd_rn(jv, bias)), mea[m]);
    axis_of<K>(A.vb) = __fadd_rn(axis_of<K>(A.vb), jvb);
    A.wb = axpy3(jvb, cross_axis<K>(ra), A.wb);
  };
  using I0 = std::integral_constant<int, 0>;
  using I1 = std::integral_constant<int, 1>;
  using I2 = std::integral_constant<int, 2>;
  row(I2{}, I1{}, 0.f);
  row(I1{}, I0{}, 0.f);
  row(I0{}, I2{}, bias0);
#pragma unroll
  for (int m = 0; m < 3; ++m)
#pragma unroll
    for (int c = 0; c < 3; ++c) acc[m][c] += Q[4 * m + (c < 2 ? c : CX_BI)];
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    S[T.sm_lam + s0 + m] = lam[m];
    Q[4 * m + CX_A] = acc[m][0];
    Q[4 * m + CX_A + 1] = acc[m][1];
    Q[4 * m + CX_ME] = mea[m];
    Q[4 * m + CX_BI] = acc[m][2];
  }
}

// ------------------------------------------------------------------------------ items
// Joint j after the sweeps: the start's application (impulses lam0, also left in the place of the
// impulse adjoints for the bodies' sums) and the effective masses, row by row; parameter gradients;
// the package over the record. The hinge axis', angle's and servo target's adjoints go to the joint's.
template <class CTX>
__device__ __forceinline__ void rx_joint_item(const DevTopo& T, const CTX& C, const TapeStep& tp, bool ws, int j) {
  const SL& S = C.S;
  const float bh = T.beta / T.dt;
  const int a = T.ja[j], b = T.jb[j], s0 = T.jslot[j], fl = T.jflags[j];
  const SL R = joint_rec(T, S, j);
  const SL Q = R.at(JR_N);
  RowBody A, B;
  rx_init(T, S, a, A);
  rx_init(T, S, b, B);
  if (a >= 0) { A.vb = C.VB.v3(6 * a); A.wb = C.VB.v3(6 * a + 3); }
  B.vb = C.VB.v3(6 * b);
  B.wb = C.VB.v3(6 * b + 3);
  const float3 ra = R.v3(JF_RA), rb = R.v3(JF_RB);
  float me[7], bib[7], M[7], l0[7], acc[3][4];
  float3 ca[4], cb[4];
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    const bool has = k < 5 || (k == 5 ? (fl & 1) != 0 : (fl & 2) != 0);
    const int f = k < 3 ? JX_LIN + 7 * k + LX_ME : (k < 5 ? JX_ANG + 9 * (k - 3) : (k == 5 ? JX_LIM : JX_MOT)) + AX_ME;
    me[k] = has ? R[JF_ME + k] : 0.f;
    M[k] = Q[f] + Q[f + 1];
    bib[k] = Q[f + 2];
    l0[k] = 0.f;
    if (ws && has && k != 5) l0[k] = tp.lam0[(k < 5 ? s0 + k : T.jmot[j]) * 32];
    if (k < 3) {
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[k][c] = Q[JX_LIN + 7 * k + c];
    } else {
      const SL q = Q.at(k < 5 ? JX_ANG + 9 * (k - 3) : (k == 5 ? JX_LIM : JX_MOT));
      ca[k - 3] = q.v3(AX_A);
      cb[k - 3] = q.v3(AX_B);
    }
  }
  const float bndb = Q[JX_MOT + AX_BND], ls = fl & 1 ? R[JF_LS] : 1.f;
  const float3 t[2] = {R.v3(JF_T), R.v3(JF_T + 3)};
  const M3 Ra = body_R(C.X, a), Rb = loadR(C.X, 18 * b);
  float3 rab[3], rbb[3];
  float ka[3][2], kb[3][2], kl[3];
  auto lin = [&](auto KI) {
    constexpr int K = decltype(KI)::value;
    if (l0[K] != 0.f) {
      const float l = l0[K];
      const float3 ga = f3(__fmul_rn(l, A.wb.x), __fmul_rn(l, A.wb.y), __fmul_rn(l, A.wb.z));
      const float3 gb = f3(__fmul_rn(l, B.wb.x), __fmul_rn(l, B.wb.y), __fmul_rn(l, B.wb.z));
      const float3 ua = symx(A.ii, ga), ub = symx(B.ii, gb);
      acc[K][0] += comp_i<K>(ua); acc[K][1] += comp_j<K>(ua);
      acc[K][2] += comp_i<K>(ub); acc[K][3] += comp_j<K>(ub);
    }
    const float Kb = __fmul_rn(__fmul_rn(-me[K], me[K]), M[K]), C0 = __fmul_rn(bh, bib[K]);
    const float3 IA = symx_axis<K>(A.ii, ra), IB = -symx_axis<K>(B.ii, rb);
    const float a0 = fmaf(2.f * Kb, comp_i<K>(IA), acc[K][0]), a1 = fmaf(2.f * Kb, comp_j<K>(IA), acc[K][1]);
    const float b0 = fmaf(2.f * Kb, comp_i<K>(IB), acc[K][2]), b1 = fmaf(2.f * Kb, comp_j<K>(IB), acc[K][3]);
    if (me[K] == 0.f) {  // (an infinite mass matrix entry: a constant row)
      rab[K] = rbb[K] = f3(0.f, 0.f, 0.f);
      ka[K][0] = ka[K][1] = kb[K][0] = kb[K][1] = kl[K] = 0.f;
      return;
    }
    // ra's adjoint e x (angA's) + the position error's, rb's -(e x (angB's)) less it
    rab[K] = K == 0 ? f3(C0, -a1, a0) : (K == 1 ? f3(a0, C0, -a1) : f3(-a1, a0, C0));
    rbb[K] = K == 0 ? f3(-C0, b1, -b0) : (K == 1 ? f3(-b0, -C0, b1) : f3(b1, -b0, -C0));
    ka[K][0] = __fmul_rn(Kb, comp_j<K>(ra)); ka[K][1] = __fmul_rn(Kb, -comp_i<K>(ra));
    kb[K][0] = __fmul_rn(Kb, -comp_j<K>(rb)); kb[K][1] = __fmul_rn(Kb, comp_i<K>(rb));
    kl[K] = Kb;
  };
  lin(std::integral_constant<int, 0>{});
  lin(std::integral_constant<int, 1>{});
  lin(std::integral_constant<int, 2>{});
  const float3 anca = C.P.v3(T.o_anchor + 6 * j), ancb = C.P.v3(T.o_anchor + 6 * j + 3);
  C.G.red3(T.o_anchor + 6 * j, mtv(Ra, rab[0] + rab[1] + rab[2]));  // (identity for the world)
  C.G.red3(T.o_anchor + 6 * j + 3, mtv(Rb, rbb[0] + rbb[1] + rbb[2]));
  float3 tau[2];
  onb3(C.P.v3(T.o_axis + 6 * j), tau[0], tau[1]);
  const float3 axb = C.P.v3(T.o_axis + 6 * j + 3);
  const float3 ub = mv(Rb, axb), ua = S.v3(T.sm_ua + 3 * j);
  const float3 cr = cross3(ub, ua);
  float3 uab = f3(0.f, 0.f, 0.f), tb[2], ubb[2], kt[4];
  float thb = 0.f, wstb = 0.f;
#pragma unroll
  for (int k = 0; k < 4; ++k) {  // angular rows, limit, servo
    const bool lim = k == 2;
    kt[k] = f3(0.f, 0.f, 0.f);
    if (me[3 + k] == 0.f) {  // (a row that is not there, or an inactive lane's limit: a constant)
      if (k < 2) tb[k] = ubb[k] = f3(0.f, 0.f, 0.f);
      continue;
    }
    const float l = l0[3 + k];
    if (l != 0.f) {
      const float3 ga = f3(__fmul_rn(l, A.wb.x), __fmul_rn(l, A.wb.y), __fmul_rn(l, A.wb.z));
      const float3 gb = f3(__fmul_rn(l, B.wb.x), __fmul_rn(l, B.wb.y), __fmul_rn(l, B.wb.z));
      ca[k] = ca[k] + symx(A.ii, ga);
      cb[k] = cb[k] + symx(B.ii, gb);
    }
    // the child's direction: -t, the limit's sign times u, u
    const float3 d = k < 2 ? -t[k & 1] : (lim ? ls : 1.f) * ua;
    const float Kb = __fmul_rn(__fmul_rn(-me[3 + k], me[3 + k]), M[3 + k]);
    const float3 ab = axpy3(2.f * Kb, symx(A.ii, -d), ca[k]), bb = axpy3(2.f * Kb, symx(B.ii, d), cb[k]);
    kt[k] = f3(__fmul_rn(Kb, d.x), __fmul_rn(Kb, d.y), __fmul_rn(Kb, d.z));
    const float g = __fmul_rn(bh, bib[3 + k]);
    if (k < 2) {
      tb[k] = axpy3(g, cr, ab - bb);
      const float3 crb = f3(__fmul_rn(g, t[k & 1].x), __fmul_rn(g, t[k & 1].y), __fmul_rn(g, t[k & 1].z));
      uab = uab + cross3(crb, ub);  // c = ub x ua
      ubb[k] = cross3(ua, crb);
    } else if (lim) {
      const bool low = ls > 0.f;
      uab = uab + (low ? bb - ab : ab - bb);
      thb = low ? g : -g;
      C.G.red(T.o_limit + 2 * j + (low ? 0 : 1), low ? -g : g);
    } else {
      uab = uab + (bb - ab);
      wstb = -bib[6];
      C.G.red(T.o_motor + 3 * j + 1, T.dt * bndb);
    }
  }
  S[T.sm_thb + j] = thb;
  S[T.sm_thdb + j] = 0.f;
  S[T.sm_wstb + j] = wstb;
  S.s3(T.sm_uab + 3 * j, uab);
#pragma unroll
  for (int k = 0; k < 5; ++k) S[T.sm_lam + s0 + k] = l0[k];
  if (fl & 2) S[T.sm_lam + T.jmot[j]] = l0[6];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const SL q = R.at(XP_LIN + 10 * k);
    q.s3(0, rab[k]);
    q.s3(3, rbb[k]);
    q[6] = ka[k][0]; q[7] = ka[k][1]; q[8] = kb[k][0]; q[9] = kb[k][1];
    R[XP_KB + k] = kl[k];
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const SL q = R.at(XP_ANG + 9 * k);
    q.s3(0, tb[k]);
    q.s3(3, ubb[k]);
    q.s3(6, -kt[k]);  // Kb t
    R.s3(XP_TAU + 3 * k, tau[k]);
  }
  R.s3(XP_LIM, ls * kt[2]);  // Kb u
  R.s3(XP_MOT, kt[3]);
  R.s3(XP_ANCA, anca);
  R.s3(XP_ANCB, ancb);
  R.s3(XP_AXB, axb);
}

// Ground contact q after the sweeps (rows of an inactive lane are constants: an empty package).
template <class CTX>
__device__ __forceinline__ void rx_contact_item(const DevTopo& T, const CTX& C, const TapeStep& tp, bool ws, int q) {
  const SL& S = C.S;
  const float bh = T.beta / T.dt;
  const int a = T.sbody[q], s0 = T.cslot + 3 * q;
  const SL R = contact_rec(T, S, q);
  const SL Q = R.at(CR_N);
  float ka[3][2] = {}, kl[3] = {}, v[3][2] = {}, l0[3] = {}, db = 0.f, vnb = 0.f;
  float3 off = f3(0.f, 0.f, 0.f);
  if (ws)
#pragma unroll
    for (int m = 0; m < 3; ++m) l0[m] = tp.lam0[(s0 + m) * 32];
  if (R[CF_ME] != 0.f) {
    float ii[6];
    load6(S, T.sm_iinv + 6 * a, ii);
    const float3 ra = R.v3(CF_RA), wb = C.VB.v3(6 * a + 3);
    auto row = [&](auto MI, auto AI) {
      constexpr int m = decltype(MI)::value, K = decltype(AI)::value;
      float c0 = Q[4 * m + CX_A], c1 = Q[4 * m + CX_A + 1];
      if (l0[m] != 0.f) {
        const float l = l0[m];
        const float3 u = symx(ii, f3(__fmul_rn(l, wb.x), __fmul_rn(l, wb.y), __fmul_rn(l, wb.z)));
        c0 += comp_i<K>(u);
        c1 += comp_j<K>(u);
      }
      const float me = R[CF_ME + m], Kb = __fmul_rn(__fmul_rn(-me, me), Q[4 * m + CX_ME]);
      const float3 IA = symx_axis<K>(ii, ra);
      v[m][0] = fmaf(2.f * Kb, comp_i<K>(IA), c0);
      v[m][1] = fmaf(2.f * Kb, comp_j<K>(IA), c1);
      ka[m][0] = __fmul_rn(Kb, comp_j<K>(ra));
      ka[m][1] = __fmul_rn(Kb, -comp_i<K>(ra));
      kl[m] = Kb;
    };
    using I0 = std::integral_constant<int, 0>;
    using I1 = std::integral_constant<int, 1>;
    using I2 = std::integral_constant<int, 2>;
    row(I0{}, I2{});
    row(I1{}, I0{});
    row(I2{}, I1{});
    const M3 Ra = loadR(C.X, 18 * a);
    off = C.P.v3(T.o_sph_off + 3 * q);
    const float rad = C.P[T.o_sph_rad + q];
    const float d = (C.X[18 * a + 2] + mv(Ra, off).z) - rad - T.ground_z;
    const float biasb = Q[CX_BI];
    const float3 vm = f3(tp.vminus[(6 * a) * 32], tp.vminus[(6 * a + 1) * 32], tp.vminus[(6 * a + 2) * 32]);
    const float3 wm = f3(tp.vminus[(6 * a + 3) * 32], tp.vminus[(6 * a + 4) * 32], tp.vminus[(6 * a + 5) * 32]);
    const float vn = __fadd_rn(vm.z, dotx_axis<2>(ra, wm));
    if (d + T.slop < 0.f) db = __fmul_rn(bh, biasb);
    if (vn < 0.f) {
      C.G.red(T.o_sph_e + q, vn * biasb);
      vnb = __fmul_rn(C.P[T.o_sph_e + q], biasb);
      v[0][0] = fmaf(vnb, wm.x, v[0][0]);
      v[0][1] = fmaf(vnb, wm.y, v[0][1]);
    }
    C.G.red(T.o_sph_mu + q, Q[4 + CX_BI] + Q[8 + CX_BI]);
    // the offset's adjoint, e x (angA's) of the three rows (along z, x and y), and the depth's
    const float3 cb = f3(-v[0][1] + v[2][0], v[0][0] - v[1][1], db + (v[1][0] - v[2][1]));
    C.G.red3(T.o_sph_off + 3 * q, mtv(Ra, cb));
    C.G.red(T.o_sph_rad + q, -cb.z);
  }
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    S[T.sm_lam + s0 + m] = l0[m];
    R[XC_KA + 2 * m] = ka[m][0];
    R[XC_KA + 2 * m + 1] = ka[m][1];
    R[XC_KB + m] = kl[m];
  }
  R.s3(XC_N, f3(-v[0][1], v[0][0], db));
  R[XC_T1] = -v[1][1];      // y
  R[XC_T1 + 1] = v[1][0];   // z
  R[XC_T2] = v[2][0];       // x
  R[XC_T2 + 1] = -v[2][1];  // z
  R[XC_V] = vnb;
  R.s3(XC_OFF, off);
}

// Body b: the rows that touch it in slot order into the adjoints of its pose, of its inverse inertia
// and mass and (restitution) of the solver's input velocities; the start's application first.
template <class CTX>
__device__ __forceinline__ void rx_body(const DevTopo& T, const CTX& C, bool ws, int b) {
  const SL& S = C.S;
  const uint8_t* first = blk_bytes(T) + T.blk_inc0;
  const uint8_t* inc = blk_bytes(T) + T.blk_inc;
  const int k0 = first[b], k1 = first[b + 1];
  float q[9], gR[9], imb = S[T.sm_invmb + b];
  float3 vb = C.VB.v3(6 * b), wb = C.VB.v3(6 * b + 3), pb = C.XB.v3(18 * b);
#pragma unroll
  for (int k = 0; k < 9; ++k) { q[k] = S[T.sm_iinvb + 9 * b + k]; gR[k] = C.XB[18 * b + 3 + k]; }
  using I0 = std::integral_constant<int, 0>;
  using I1 = std::integral_constant<int, 1>;
  using I2 = std::integral_constant<int, 2>;
  auto scaled = [&](float l) { return f3(__fmul_rn(l, wb.x), __fmul_rn(l, wb.y), __fmul_rn(l, wb.z)); };
  if (ws) {
    for (int k = k0; k < k1 && inc[k] < 0x40; ++k) {
      const int j = inc[k] & 31, s0 = T.jslot[j];
      const bool sb = inc[k] & 0x20;
      const SL R = joint_rec(T, S, j);
      const float sg = sb ? -1.f : 1.f;
      const float3 r = R.v3(sb ? JF_RB : JF_RA);
      const float3 l = sg * S.v3(T.sm_lam + s0);
      outer9_axis<0>(q, scaled(l.x), r);
      outer9_axis<1>(q, scaled(l.y), r);
      outer9_axis<2>(q, scaled(l.z), r);
      imb = fmaf(l.z, vb.z, fmaf(l.y, vb.y, fmaf(l.x, vb.x, imb)));
#pragma unroll
      for (int m = 0; m < 2; ++m) outer9(q, scaled(sg * S[T.sm_lam + s0 + 3 + m]), R.v3(JF_T + 3 * m));
    }
    for (int k = k0; k < k1 && inc[k] < 0x40; ++k) {  // servo rows (limit rows start cold)
      const int j = inc[k] & 31;
      if (T.jmot[j] < 0) continue;
      outer9(q, scaled((inc[k] & 0x20 ? 1.f : -1.f) * S[T.sm_lam + T.jmot[j]]), S.v3(T.sm_ua + 3 * j));
    }
    for (int k = k0; k < k1; ++k) {
      if (inc[k] < 0x40) continue;
      const int c = inc[k] & 31, s0 = T.cslot + 3 * c;
      const float3 r = contact_rec(T, S, c).v3(CF_RA);
      const float3 l = S.v3(T.sm_lam + s0);  // along z, x and y
      outer9_axis<2>(q, scaled(l.x), r);
      outer9_axis<0>(q, scaled(l.y), r);
      outer9_axis<1>(q, scaled(l.z), r);
      imb = fmaf(l.z, vb.y, fmaf(l.y, vb.x, fmaf(l.x, vb.z, imb)));
    }
  }
  for (int k = k0; k < k1 && inc[k] < 0x40; ++k) {
    const int j = inc[k] & 31;
    const bool sb = inc[k] & 0x20;
    const SL R = joint_rec(T, S, j);
    const float3 r = R.v3(sb ? JF_RB : JF_RA), anc = R.v3(sb ? XP_ANCB : XP_ANCA);
    const float sg = sb ? -1.f : 1.f;
    auto lin = [&](auto KI) {
      constexpr int K = decltype(KI)::value;
      const SL p = R.at(XP_LIN + 10 * K);
      const float3 g = p.v3(sb ? 3 : 0);
      const float ki = p[sb ? 8 : 6], kj = p[sb ? 9 : 7];
      outer4_axis<K>(q, ki, kj, r, sg);
      imb += R[XP_KB + K];
      axis_of<K>(pb) += comp<K>(g);
      outer9(gR, g, anc);
    };
    lin(I0{});
    lin(I1{});
    lin(I2{});
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      const SL p = R.at(XP_ANG + 9 * m);
      outer9(q, p.v3(6), R.v3(JF_T + 3 * m));
      outer9(gR, p.v3(sb ? 3 : 0), R.v3(sb ? XP_AXB : XP_TAU + 3 * m));
    }
  }
  for (int f = XP_LIM; f <= XP_MOT; f += 3)
    for (int k = k0; k < k1 && inc[k] < 0x40; ++k) {
      const int j = inc[k] & 31;
      outer9(q, joint_rec(T, S, j).v3(f), S.v3(T.sm_ua + 3 * j));
    }
  for (int k = k0; k < k1; ++k) {
    if (inc[k] < 0x40) continue;
    const SL R = contact_rec(T, S, inc[k] & 31);
    const float3 r = R.v3(CF_RA), off = R.v3(XC_OFF), n = R.v3(XC_N);
    const float vnb = R[XC_V];
    outer4_axis<2>(q, R[XC_KA], R[XC_KA + 1], r, 1.f);
    vb.z += vnb;
    wb.x = fmaf(vnb, r.y, wb.x);
    wb.y = fmaf(vnb, -r.x, wb.y);
    pb.z += n.z;
    outer9(gR, n, off);
    outer4_axis<0>(q, R[XC_KA + 2], R[XC_KA + 3], r, 1.f);
    outer9(gR, f3(0.f, R[XC_T1], R[XC_T1 + 1]), off);
    outer4_axis<1>(q, R[XC_KA + 4], R[XC_KA + 5], r, 1.f);
    outer9(gR, f3(R[XC_T2], 0.f, R[XC_T2 + 1]), off);
    imb = ((imb + R[XC_KB]) + R[XC_KB + 1]) + R[XC_KB + 2];
  }
  C.VB.s3(6 * b, vb);
  C.VB.s3(6 * b + 3, wb);
  C.XB.s3(18 * b, pb);
#pragma unroll
  for (int k = 0; k < 9; ++k) { S[T.sm_iinvb + 9 * b + k] = q[k]; C.XB[18 * b + 3 + k] = gR[k]; }
  S[T.sm_invmb + b] = imb;
}

// Hinge kinematics of joint j reversed: what it adds to its bodies' R and w; the package over the record.
template <class CTX>
__device__ __forceinline__ void rx_hinge_item(const DevTopo& T, const CTX& C, int j) {
  const SL& S = C.S;
  const int a = T.ja[j], b = T.jb[j];
  float3 uab = S.v3(T.sm_uab + 3 * j);
  const M3 Ra = body_R(C.X, a), Rb = loadR(C.X, 18 * b);
  const float3 axa = C.P.v3(T.o_axis + 6 * j);
  const float3 ua = S.v3(T.sm_ua + 3 * j);
  const float3 refa = C.P.v3(T.o_ref + 6 * j), refb = C.P.v3(T.o_ref + 6 * j + 3);
  const float3 wa = mv(Ra, refa), wb = mv(Rb, refb);
  const float3 c = cross3(wa, wb);
  const float y = dot3(c, ua), x = dot3(wa, wb);
  const float thb = S[T.sm_thb + j], thdb = S[T.sm_thdb + j];
  const float den = x * x + y * y;
  const float yb = thb * x / den, xb = -thb * y / den;
  const float3 cb = yb * ua;
  uab += yb * c;
  const float3 wab = cross3(wb, cb) + xb * wb;
  const float3 wbb = cross3(cb, wa) + xb * wa;
  uab += thdb * (C.X.v3(18 * b + 15) - body_w(C.X, a));
  const SL R = joint_rec(T, S, j);
  R.s3(XH_W, f3(__fmul_rn(thdb, ua.x), __fmul_rn(thdb, ua.y), __fmul_rn(thdb, ua.z)));
  R.s3(XH_WA, wab);
  R.s3(XH_WB, wbb);
  R.s3(XH_UB, uab);
  R.s3(XH_REFA, refa);
  R.s3(XH_REFB, refb);
  R.s3(XH_AXA, axa);
}
template <class CTX>
__device__ __forceinline__ void rx_hinge_body(const DevTopo& T, const CTX& C, int b) {
  const uint8_t* first = blk_bytes(T) + T.blk_inc0;
  const uint8_t* inc = blk_bytes(T) + T.blk_inc;
  float3 w = C.XB.v3(18 * b + 15);
  float gR[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) gR[q] = C.XB[18 * b + 3 + q];
  const int k1 = first[b + 1];
  for (int k = first[b]; k < k1 && inc[k] < 0x40; ++k) {
    const SL R = joint_rec(T, C.S, inc[k] & 31);
    const bool sb = inc[k] & 0x20;
    const float3 c = R.v3(XH_W);
    w = sb ? w + c : w - c;
    outer9(gR, R.v3(sb ? XH_WB : XH_WA), R.v3(sb ? XH_REFB : XH_REFA));
    if (!sb) outer9(gR, R.v3(XH_UB), R.v3(XH_AXA));
  }
  C.XB.s3(18 * b + 15, w);
#pragma unroll
  for (int q = 0; q < 9; ++q) C.XB[18 * b + 3 + q] = gR[q];
}
