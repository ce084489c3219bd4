// The reverse-mode kernels on blocks, one CTA per group of 32 instances (items, blocks and records of
// dp_blk.cuh). A reverse step
//   - reverses the loss term and the integrator (bodies),
//   - re-forms the step's records from x_t (items), bit for bit those of the rollout,
//   - runs the sweeps backwards over the same blocks, levels and streams (last level first): a warp
//     holds a block's two bodies - velocities replayed by undoing each row's impulse, and their
//     adjoints - in registers, and adds the row-side adjoints to the item's accumulators, which lie
//     behind its record: of the linear rows only the adjoints of the two lever arms, of the angular
//     rows those of the two directions, of limit and servo row that of the axis,
//   - pushes every item's adjoints to its bodies: the item's warp writes one package per side over
//     its record, and the bodies' warps add the packages of their items in slot order,
//   - reverses the external impulses (bodies), the controller (tensor-core layers split over the
//     warps) and the hinge kinematics (items, packages again).
// A body belongs to one block at a time (levels), one warp outside the sweeps, so every sum has one
// writer and a fixed order.
// The compiled topologies (kernels with SEQ) form the same adjoints row by row: their blocks, items and
// packages are in dp_blk_rows.cuh, those here are every other robot's.
#pragma once
#include "dp_blk_rows.cuh"

// Accumulators behind a record's first fields (joints: JA_* from JR_N on, contacts from CR_N, pairs
// from PR_N), and the packages that overwrite the records.
enum { JA_RA = 0, JA_RB = 3, JA_T = 6, JA_U = 12, JA_ME = 15, JA_BI = 22, JA_BND = 29, JA_N = 30 };
enum { CA_RA = 0, CA_ME = 3, CA_BI = 6, CA_MU = 7, CA_N = 8 };
enum { PA_LIN = 0, PA_ANGA = 9, PA_ANGB = 18, PA_ME = 27, PA_BI = 30, PA_MU = 31, PA_N = 32 };
enum { JP_P = 0, JP_RA = 3, JP_RB = 12, JP_SA = 21, JP_SB = 27, JP_IA = 33, JP_IB = 34, JP_N = 35 };
enum { CP_Z = 0, CP_R = 1, CP_S = 10, CP_I = 16, CP_V = 17, CP_W = 18, CP_N = 21 };
enum { PP_P = 0, PP_RA = 3, PP_RB = 12, PP_SA = 21, PP_SB = 27, PP_IA = 33, PP_IB = 34, PP_V = 35, PP_WA = 38, PP_WB = 41, PP_GK = 44, PP_GL = 50, PP_N = 56 };
// A pair's share of its two spheres' parameter gradients (at PP_GK and PP_GL): offset, radius, friction,
// restitution.
enum { PG_OFF = 0, PG_RAD = 3, PG_MU = 4, PG_E = 5 };
enum { HP_W = 0, HP_RA = 3, HP_RB = 12, HP_N = 21 };

// One body of a block: velocities, their adjoints, inverse mass and inertia, and the block's sums
// of the adjoints of those (the inertia's as q_xx, q_xy + q_yx, q_xz + q_zx, q_yy, q_yz + q_zy,
// q_zz of the adjoint matrix q: only its symmetric part is used).
struct RevBody {
  float3 v, w, vb, wb;
  float im, imb, ii[6], sb[6];
};
__device__ __forceinline__ void rev_init(const DevTopo& T, const SL& S, int b, RevBody& B) {
  B.imb = 0.f;
#pragma unroll
  for (int q = 0; q < 6; ++q) B.sb[q] = B.ii[q] = 0.f;
  B.v = B.w = B.vb = B.wb = f3(0.f, 0.f, 0.f);
  B.im = 0.f;
  if (b < 0) return;
  B.im = S[T.sm_invm + b];
  load6(S, T.sm_iinv + 6 * b, B.ii);
}
__device__ __forceinline__ void rev_load(const DevTopo& T, const SL& S, const SL& VW, int b, RevBody& B) {
  if (b < 0) return;
  B.v = VW.v3(6 * b);
  B.w = VW.v3(6 * b + 3);
  B.vb = S.v3(T.sm_vb + 6 * b);
  B.wb = S.v3(T.sm_vb + 6 * b + 3);
}
__device__ __forceinline__ void rev_store(const DevTopo& T, const SL& S, const SL& VW, int b, const RevBody& B, bool lin) {
  if (b < 0) return;
  float ib[6];
  load6(S, T.sm_iinvb + 6 * b, ib);
  const float imb = S[T.sm_invmb + b];
  if (lin) {
    VW.s3(6 * b, B.v);
    S.s3(T.sm_vb + 6 * b, B.vb);
    S[T.sm_invmb + b] = imb + B.imb;
  }
  VW.s3(6 * b + 3, B.w);
  S.s3(T.sm_vb + 6 * b + 3, B.wb);
#pragma unroll
  for (int q = 0; q < 6; ++q) S[T.sm_iinvb + 6 * b + q] = ib[q] + B.sb[q];
}

// Products with r x e_K and with e_K x v (two non-zero components each).
template <int K>
__device__ __forceinline__ float dot_axis(float3 r, float3 w) {
  if (K == 0) return r.z * w.y - r.y * w.z;
  if (K == 1) return r.x * w.z - r.z * w.x;
  return r.y * w.x - r.x * w.y;
}
template <int K>
__device__ __forceinline__ void add_axis(float3& w, float s, float3 r) {
  if (K == 0) { w.y = fmaf(s, r.z, w.y); w.z = fmaf(-s, r.y, w.z); }
  if (K == 1) { w.x = fmaf(-s, r.z, w.x); w.z = fmaf(s, r.x, w.z); }
  if (K == 2) { w.x = fmaf(s, r.y, w.x); w.y = fmaf(-s, r.x, w.y); }
}
template <int K>
__device__ __forceinline__ void add_e_cross(float3& a, float s, float3 v) {
  if (K == 0) { a.y = fmaf(-s, v.z, a.y); a.z = fmaf(s, v.y, a.z); }
  if (K == 1) { a.x = fmaf(s, v.z, a.x); a.z = fmaf(-s, v.x, a.z); }
  if (K == 2) { a.x = fmaf(-s, v.y, a.x); a.y = fmaf(s, v.x, a.y); }
}
template <int K>
__device__ __forceinline__ float3 symv_axis(const float (&s)[6], float3 r) {
  if (K == 0) return f3(s[1] * r.z - s[2] * r.y, s[3] * r.z - s[4] * r.y, s[4] * r.z - s[5] * r.y);
  if (K == 1) return f3(s[2] * r.x - s[0] * r.z, s[4] * r.x - s[1] * r.z, s[5] * r.x - s[2] * r.z);
  return f3(s[0] * r.y - s[1] * r.x, s[1] * r.y - s[3] * r.x, s[2] * r.y - s[4] * r.x);
}
__device__ __forceinline__ void sym_outer(float (&q)[6], float3 g, float3 a) {
  q[0] = fmaf(g.x, a.x, q[0]);
  q[1] = fmaf(g.x, a.y, fmaf(g.y, a.x, q[1]));
  q[2] = fmaf(g.x, a.z, fmaf(g.z, a.x, q[2]));
  q[3] = fmaf(g.y, a.y, q[3]);
  q[4] = fmaf(g.y, a.z, fmaf(g.z, a.y, q[4]));
  q[5] = fmaf(g.z, a.z, q[5]);
}
template <int K>
__device__ __forceinline__ void sym_outer_axis(float (&q)[6], float3 g, float3 r) {
  if (K == 0) {
    q[1] = fmaf(g.x, r.z, q[1]); q[2] = fmaf(-g.x, r.y, q[2]); q[3] = fmaf(g.y, r.z, q[3]);
    q[4] = fmaf(-g.y, r.y, fmaf(g.z, r.z, q[4])); q[5] = fmaf(-g.z, r.y, q[5]);
  }
  if (K == 1) {
    q[0] = fmaf(-g.x, r.z, q[0]); q[1] = fmaf(-g.y, r.z, q[1]); q[2] = fmaf(g.x, r.x, fmaf(-g.z, r.z, q[2]));
    q[4] = fmaf(g.y, r.x, q[4]); q[5] = fmaf(g.z, r.x, q[5]);
  }
  if (K == 2) {
    q[0] = fmaf(g.x, r.y, q[0]); q[1] = fmaf(-g.x, r.x, fmaf(g.y, r.y, q[1])); q[2] = fmaf(g.z, r.y, q[2]);
    q[3] = fmaf(-g.y, r.x, q[3]); q[4] = fmaf(-g.z, r.x, q[4]);
  }
}

// One sweep's tape lines on chip: the impulses it left (la) and found (lb), its clamp branches, and
// the velocities after it, which become the working copy.
struct RevTape {
  SL la, lb, vw;
  const uint8_t* br;  // slot s at br[32 s]
};
// Where sweep `it`'s impulses (a ring of three sweeps), velocities and branches (two) lie. ROWS (compiled
// topologies): the buffers that the first sweep does not need lie over x_t (sm_rlam2, sm_vw2, sm_rbr2):
// nothing is written to them before the records are formed.
template <bool ROWS>
__device__ __forceinline__ int rev_lam_at(const DevTopo& T, int it) {
  if (!ROWS) return T.sm_rlam + (it + 3) % 3 * T.nslots;
  const int k = (T.iters - 1 - it) % 3;
  return k == 2 ? T.sm_rlam2 : T.sm_rlam + k * T.nslots;
}
template <bool ROWS>
__device__ __forceinline__ int rev_vw_at(const DevTopo& T, int it) {
  if (!ROWS) return T.sm_vw + (it & 1) * 6 * T.nb;
  return (T.iters - 1 - it) & 1 ? T.sm_vw2 : T.sm_vw;
}
template <bool ROWS>
__device__ __forceinline__ int rev_br_at(const DevTopo& T, int it) {
  if (!ROWS) return T.sm_rbr + (it & 1) * ((T.nslots + 3) / 4);
  return (T.iters - 1 - it) & 1 ? T.sm_rbr2 : T.sm_rbr;
}
template <bool ROWS>
__device__ __forceinline__ RevTape rev_tape(const DevTopo& T, const SL& S, int it) {
  return RevTape{S.at(rev_lam_at<ROWS>(T, it)), S.at(rev_lam_at<ROWS>(T, it - 1)), S.at(rev_vw_at<ROWS>(T, it)),
                 reinterpret_cast<const uint8_t*>(g_smem + rev_br_at<ROWS>(T, it) * 32) + (threadIdx.x & 31)};
}
// n bytes of the tape record (a multiple of 16, like both addresses) into unit `unit`, asynchronously.
__device__ __forceinline__ void rev_copy(int unit, const uint8_t* src, int n) {
  const unsigned dst = (unsigned)__cvta_generic_to_shared(g_smem + unit * 32);
  for (int o = threadIdx.x * 16; o < n; o += blockDim.x * 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + o), "l"(src + o) : "memory");
}
// Impulses after sweep `it` (-1: before the first one) into the ring of three sweeps.
template <bool ROWS>
__device__ __forceinline__ void rev_stage_lam(const DevTopo& T, const TapeStep& tp, int it) {
  const int unit = rev_lam_at<ROWS>(T, it), n = T.nslots * 128;
  if (it >= 0) rev_copy(unit, tp.rec + T.rec_lam + (size_t)it * n, n);
  else if (T.ws) rev_copy(unit, tp.rec + T.rec_lam0, n);
  else
    for (int f = threadIdx.x; f < T.nslots * 32; f += blockDim.x) g_smem[unit * 32 + f] = 0.f;
}
// Velocities after sweep `it` and its clamp branches (two buffers each).
template <bool ROWS>
__device__ __forceinline__ void rev_stage_sweep(const DevTopo& T, const TapeStep& tp, int it) {
  const int nv = 6 * T.nb * 128, nb = T.nslots * 32;
  rev_copy(rev_vw_at<ROWS>(T, it), tp.rec + T.rec_viter + (size_t)it * nv, nv);
  rev_copy(rev_br_at<ROWS>(T, it), tp.rec + T.rec_br + (size_t)it * nb, nb);
}
// The last sweep's lines, asked for at the start of a step.
template <bool ROWS>
__device__ __forceinline__ void rev_stage_first(const DevTopo& T, const TapeStep& tp) {
  rev_stage_lam<ROWS>(T, tp, T.iters - 1);
  rev_stage_lam<ROWS>(T, tp, T.iters - 2);
  rev_stage_sweep<ROWS>(T, tp, T.iters - 1);
}
// Waits for sweep `it`'s lines and asks for those of the sweep before it (every warp calls). Read from
// L2 where they are used, at the head of every block's chain, they cost more than the rows.
template <bool ROWS>
__device__ __forceinline__ void rev_begin_sweep(const DevTopo& T, const TapeStep& tp, int it) {
  asm volatile("cp.async.wait_all;" ::: "memory");
  cta_sync();
  if (it > 0) {
    rev_stage_lam<ROWS>(T, tp, it - 2);
    rev_stage_sweep<ROWS>(T, tp, it - 1);
  }
}

// Rows, last first. As in the rollout, a block loads everything it reads before its first row (what
// only it changes ahead of ready()) and stores after its last one; adjoints of the record are summed in
// registers.
// One linear row of a joint: lam is its impulse's adjoint, meb the sum of the effective mass' adjoint
// (over the step: each row's share is added by one fused multiply-add);
// returns the adjoint of J v.
template <int K>
__device__ __forceinline__ float rev_lin(const DevTopo& T, float la, float lb, float me, float bi, float3 ra, float3 rb,
                                         RevBody& A, RevBody& B, float3& rab, float3& rbb, float& lam, float& meb) {
  const float dl = la - lb;
  const float3 IA = symv_axis<K>(A.ii, ra), IBn = symv_axis<K>(B.ii, rb);  // the child's is -IBn
  // velocities before the row, then the adjoint of the row's change
  const float ca = dl * A.im, cb = dl * B.im;
  axis_of<K>(A.v) -= ca;
  A.w = axpy3(-dl, IA, A.w);
  axis_of<K>(B.v) += cb;
  B.w = axpy3(dl, IBn, B.w);
  const float dbar = (A.im * axis_of<K>(A.vb) + dot3(IA, A.wb)) - (B.im * axis_of<K>(B.vb) + dot3(IBn, B.wb));
  const float pbar = lam + dbar, jvb = -me * pbar;
  lam = fmaf(-me * T.gamma, pbar, lam);  // pbar (1 - me gamma) - dbar, without the cancellation
  // adjoints of M^-1 J^T (before the update of the velocity adjoints)
  const float3 ga = dl * A.wb, gb = dl * B.wb;
  add_e_cross<K>(rab, 1.f, axpy3(jvb, A.w, symv(A.ii, ga)));
  add_e_cross<K>(rbb, -1.f, axpy3(jvb, B.w, symv(B.ii, gb)));
  sym_outer_axis<K>(A.sb, ga, ra);
  sym_outer_axis<K>(B.sb, -gb, rb);
  A.imb = fmaf(dl, axis_of<K>(A.vb), A.imb);
  B.imb = fmaf(-dl, axis_of<K>(B.vb), B.imb);
  const float Jv = (axis_of<K>(A.v) + dot_axis<K>(ra, A.w)) - (axis_of<K>(B.v) + dot_axis<K>(rb, B.w));
  meb += -pbar * (Jv + bi + T.gamma * lb);
  axis_of<K>(A.vb) += jvb;
  add_axis<K>(A.wb, jvb, ra);
  axis_of<K>(B.vb) -= jvb;
  add_axis<K>(B.wb, -jvb, rb);
  return jvb;
}
// A row without a linear part along the child's direction d (J_wb = d, J_wa = -d): angular, limit and
// servo rows. db: adjoint of d. branch: 0 inside, 1 lower bound, 2 upper bound; lbar: the clamped
// impulse's adjoint.
__device__ __forceinline__ float rev_ang(const DevTopo& T, float la, float lb, float me, float bi, int br, float3 d,
                                         RevBody& A, RevBody& B, float3& db, float& lam, float& meb, float& lbar) {
  const float dl = la - lb;
  const float3 IA = symv(A.ii, d), IB = symv(B.ii, d);  // the parent's is -IA
  A.w = axpy3(dl, IA, A.w);
  B.w = axpy3(-dl, IB, B.w);
  const float dbar = dot3(IB, B.wb) - dot3(IA, A.wb);
  lbar = lam + dbar;
  const float pbar = br == 0 ? lbar : 0.f, jvb = -me * pbar;
  lam = br == 0 ? fmaf(-me * T.gamma, pbar, lam) : -dbar;
  const float3 ga = dl * A.wb, gb = dl * B.wb;
  db = (axpy3(jvb, B.w, symv(B.ii, gb))) - (axpy3(jvb, A.w, symv(A.ii, ga)));
  sym_outer(A.sb, -ga, d);
  sym_outer(B.sb, gb, d);
  const float Jv = dot3(d, B.w - A.w);
  meb += -pbar * (Jv + bi + T.gamma * lb);
  A.wb = axpy3(-jvb, d, A.wb);
  B.wb = axpy3(jvb, d, B.wb);
  return jvb;
}

template <bool FULL, class RD>
__device__ __forceinline__ void rev_joint(const DevTopo& T, const SL& S, const RevTape& tp, const BlkOp& op, const SL& R,
                                          RevBody& A, RevBody& B, const RD& ready) {
  const int mask = FULL ? 31 : op.mask(), s0 = op.slot();
  const SL Q = R.at(JR_N);
  const float3 ra = R.v3(JF_RA), rb = R.v3(JF_RB);
  float la[5], lb[5], lam[5], me[5], bi[5], meb[5], bib[5];
  float3 t[2], tb[2];
#pragma unroll
  for (int k = 0; k < 5; ++k)
    if (mask >> k & 1) {
      la[k] = tp.la[s0 + k];
      lb[k] = tp.lb[s0 + k];
      lam[k] = S[T.sm_lam + s0 + k];
      me[k] = R[JF_ME + k];
      bi[k] = R[JF_BI + k];
      meb[k] = Q[JA_ME + k];
      if (k >= 3) t[k - 3] = R.v3(JF_T + 3 * (k - 3));
    }
  ready();
  float unused;
#pragma unroll
  for (int k = 4; k >= 3; --k)
    if (mask >> k & 1)
      bib[k] = rev_ang(T, la[k], lb[k], me[k], bi[k], 0, -t[k - 3], A, B, tb[k - 3], lam[k], meb[k], unused);
  float3 rab = f3(0.f, 0.f, 0.f), rbb = rab;
  if (mask & 4) bib[2] = rev_lin<2>(T, la[2], lb[2], me[2], bi[2], ra, rb, A, B, rab, rbb, lam[2], meb[2]);
  if (mask & 2) bib[1] = rev_lin<1>(T, la[1], lb[1], me[1], bi[1], ra, rb, A, B, rab, rbb, lam[1], meb[1]);
  if (mask & 1) bib[0] = rev_lin<0>(T, la[0], lb[0], me[0], bi[0], ra, rb, A, B, rab, rbb, lam[0], meb[0]);
#pragma unroll
  for (int k = 0; k < 5; ++k)
    if (mask >> k & 1) {
      bib[k] += Q[JA_BI + k];
      if (k >= 3) tb[k - 3] = Q.v3(JA_T + 3 * (k - 3)) - tb[k - 3];
    }
  rab = Q.v3(JA_RA) + rab;
  rbb = Q.v3(JA_RB) + rbb;
#pragma unroll
  for (int k = 0; k < 5; ++k)
    if (mask >> k & 1) {
      S[T.sm_lam + s0 + k] = lam[k];
      Q[JA_ME + k] = meb[k];
      Q[JA_BI + k] = bib[k];
      if (k >= 3) Q.s3(JA_T + 3 * (k - 3), tb[k - 3]);
    }
  Q.s3(JA_RA, rab);
  Q.s3(JA_RB, rbb);
}
template <class RD>
__device__ __forceinline__ void rev_hinge(const DevTopo& T, const SL& S, const RevTape& tp, const BlkOp& op, const SL& R, int j,
                                          RevBody& A, RevBody& B, const RD& ready) {
  const bool lim = op.type() == BT_LIMIT;
  const int s = op.slot(), m = lim ? 5 : 6;
  const SL Q = R.at(JR_N);
  const float sg = lim ? R[JF_LS] : 1.f;
  const int br = tp.br[s * 32];
  const float me = R[JF_ME + m], bi = R[JF_BI + m], la = tp.la[s], lb = tp.lb[s];
  const float bib0 = Q[JA_BI + m], bnd0 = Q[JA_BND];
  const float3 ua = S.v3(T.sm_ua + 3 * j);
  float lam = S[T.sm_lam + s], meb = Q[JA_ME + m], lbar;
  ready();
  const float3 u0 = Q.v3(JA_U);  // (the joint's limit and servo row share it)
  float3 ub;
  const float bib = rev_ang(T, la, lb, me, bi, br, sg * ua, A, B, ub, lam, meb, lbar);
  S[T.sm_lam + s] = lam;
  Q[JA_ME + m] = meb;
  Q[JA_BI + m] = bib0 + bib;
  Q.s3(JA_U, u0 + sg * ub);
  if (!lim) Q[JA_BND] = bnd0 + (br == 2 ? 1.f : (br == 1 ? -1.f : 0.f)) * lbar;
}
template <class RD>
__device__ __forceinline__ void rev_contact(const DevTopo& T, const SL& S, const RevTape& tp, const BlkOp& op, const SL& R,
                                            RevBody& A, const RD& ready) {
  const int mask = op.mask(), s0 = op.slot();
  const SL Q = R.at(CR_N);
  float la[3], lb[3], lam[3], me[3], meb[3];
  int br[3];
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    la[m] = tp.la[s0 + m];
    lb[m] = tp.lb[s0 + m];
    br[m] = tp.br[(s0 + m) * 32];
    lam[m] = S[T.sm_lam + s0 + m];
    me[m] = R[CF_ME + m];
    meb[m] = Q[CA_ME + m];
  }
  const float3 ra = R.v3(CF_RA);
  const float mu = R[CF_MU], bias0 = R[CF_BI];
  float3 rab = f3(0.f, 0.f, 0.f);
  ready();
  if (mask != 7)  // another block of this contact changes their adjoints and sums too
    for (int m = 0; m < 3; ++m) {
      lam[m] = S[T.sm_lam + s0 + m];
      meb[m] = Q[CA_ME + m];
    }
  // the normal impulse a friction row saw: the sweep's own (the normal row comes first)
  const float lnrm = la[0];
  float mub = 0.f, bib = 0.f;
  auto row = [&](auto MI, auto AI, float bias) {
    constexpr int m = decltype(MI)::value, ax = decltype(AI)::value;
    const float dl = la[m] - lb[m];
    const float3 IA = symv_axis<ax>(A.ii, ra);
    const float ca = dl * A.im;
    axis_of<ax>(A.v) -= ca;
    A.w = axpy3(-dl, IA, A.w);
    const float dbar = A.im * axis_of<ax>(A.vb) + dot3(IA, A.wb);
    const float lbar = lam[m] + dbar;
    const float pbar = br[m] == 0 ? lbar : 0.f, jvb = -me[m] * pbar;
    if (m > 0) {
      const float sg = br[m] == 2 ? 1.f : (br[m] == 1 ? -1.f : 0.f);
      mub += sg * lnrm * lbar;
      lam[0] += sg * mu * lbar;
    }
    lam[m] = br[m] == 0 ? fmaf(-me[m] * T.gamma, pbar, lam[m]) : -dbar;
    const float3 ga = dl * A.wb;
    add_e_cross<ax>(rab, 1.f, axpy3(jvb, A.w, symv(A.ii, ga)));
    sym_outer_axis<ax>(A.sb, ga, ra);
    A.imb = fmaf(dl, axis_of<ax>(A.vb), A.imb);
    const float Jv = axis_of<ax>(A.v) + dot_axis<ax>(ra, A.w);
    meb[m] += -pbar * (Jv + bias + T.gamma * lb[m]);
    if (m == 0) bib = jvb;
    axis_of<ax>(A.vb) += jvb;
    add_axis<ax>(A.wb, jvb, ra);
  };
  using I0 = std::integral_constant<int, 0>;
  using I1 = std::integral_constant<int, 1>;
  using I2 = std::integral_constant<int, 2>;
  if (mask & 4) row(I2{}, I1{}, 0.f);
  if (mask & 2) row(I1{}, I0{}, 0.f);
  if (mask & 1) row(I0{}, I2{}, bias0);
  bib += Q[CA_BI];
  mub += Q[CA_MU];
  rab = Q.v3(CA_RA) + rab;
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    S[T.sm_lam + s0 + m] = lam[m];  // (the normal's also from a block of friction rows alone)
    Q[CA_ME + m] = meb[m];
  }
  Q[CA_BI] = bib;
  Q[CA_MU] = mub;
  Q.s3(CA_RA, rab);
}
template <class RD>
__device__ __forceinline__ void rev_pair(const DevTopo& T, const SL& S, const RevTape& tp, const BlkOp& op, const SL& R,
                                         RevBody& A, RevBody& B, const RD& ready) {
  ready();
  const int mask = op.mask(), s0 = op.slot();
  const float mu = R[PF_MU], lnrm = tp.la[s0];
#pragma unroll 1
  for (int m = 2; m >= 0; --m) {
    if (!(mask >> m & 1)) continue;
    const int s = s0 + m, br = tp.br[s * 32];
    const float3 lin = R.v3(PF_LIN + 3 * m), angA = R.v3(PF_ANGA + 3 * m), angB = R.v3(PF_ANGB + 3 * m);
    const float lb = tp.lb[s], dl = tp.la[s] - lb, me = R[PF_ME + m];
    const float3 IA = symv(A.ii, angA), IB = symv(B.ii, angB);
    A.v = axpy3(-dl * A.im, lin, A.v);
    A.w = axpy3(-dl, IA, A.w);
    B.v = axpy3(dl * B.im, lin, B.v);
    B.w = axpy3(-dl, IB, B.w);
    const float dva = dot3(lin, A.vb), dvb = dot3(lin, B.vb);
    const float dbar = (A.im * dva + dot3(IA, A.wb)) + (dot3(IB, B.wb) - B.im * dvb);
    const float lbar = S[T.sm_lam + s] + dbar;
    const float pbar = br == 0 ? lbar : 0.f, jvb = -me * pbar;
    if (m > 0) {
      const float sg = br == 2 ? 1.f : (br == 1 ? -1.f : 0.f);
      R[PR_N + PA_MU] += sg * lnrm * lbar;
      S[T.sm_lam + s0] += sg * mu * lbar;
    }
    S[T.sm_lam + s] = fmaf(pbar, fmaf(-me, T.gamma, 1.f), -dbar);
    const float3 ga = dl * A.wb, gb = dl * B.wb;
    R.a3(PR_N + PA_LIN + 3 * m, dl * (A.im * A.vb - B.im * B.vb) + jvb * (A.v - B.v));
    R.a3(PR_N + PA_ANGA + 3 * m, axpy3(jvb, A.w, symv(A.ii, ga)));
    R.a3(PR_N + PA_ANGB + 3 * m, axpy3(jvb, B.w, symv(B.ii, gb)));
    sym_outer(A.sb, ga, angA);
    sym_outer(B.sb, gb, angB);
    A.imb += dl * dva;
    B.imb -= dl * dvb;
    const float Jv = dot3(lin, A.v - B.v) + dot3(angA, A.w) + dot3(angB, B.w);
    R[PR_N + PA_ME + m] += -pbar * (Jv + (m == 0 ? R[PF_BI] : 0.f) + T.gamma * lb);
    if (m == 0) R[PR_N + PA_BI] += jvb;
    A.vb = axpy3(jvb, lin, A.vb);
    A.wb = axpy3(jvb, angA, A.wb);
    B.vb = axpy3(-jvb, lin, B.vb);
    B.wb = axpy3(jvb, angB, B.wb);
  }
}

// The sweeps backwards (every warp calls; ends after a CTA barrier). On entry VB holds the adjoint
// of the solver's output velocities, on exit that of its input velocities. ROWS: the sums row by row
// (compiled topologies, dp_blk_rows.cuh); else the robot may be of one block, whose warp keeps the bodies'
// adjoints in registers over the sweeps.
template <bool ROWS>
__device__ __forceinline__ void blk_sweeps_rev(const DevTopo& T, const SL& S, const TapeStep& tp, int warp) {
  const uint8_t* st0 = blk_bytes(T) + T.blk_stream + warp * T.blk_stream_len;
  using Body = std::conditional_t<ROWS, RowBody, RevBody>;
  auto rows = [&](const BlkOp& op, const RevTape& rt, Body& A, Body& B, const auto& ready) {
    const int type = op.type(), idx = op.idx();
    if constexpr (ROWS) {  // (a compiled topology has no sphere pairs)
      if (type == BT_GROUND) rx_contact(T, S, rt, op, contact_rec(T, S, idx), A, ready);
      else if (type == BT_JOINT) {
        rx_joint(T, S, rt, op, joint_rec(T, S, idx), A, B, ready);
      } else rx_hinge(T, S, rt, op, joint_rec(T, S, idx), A, B, ready);
    } else if (type == BT_GROUND) rev_contact(T, S, rt, op, contact_rec(T, S, idx), A, ready);
    else if (type == BT_JOINT) {
      if (op.mask() == 31) rev_joint<true>(T, S, rt, op, joint_rec(T, S, idx), A, B, ready);
      else rev_joint<false>(T, S, rt, op, joint_rec(T, S, idx), A, B, ready);
    } else if (type == BT_PAIR) rev_pair(T, S, rt, op, pair_rec(T, S, idx), A, B, ready);
    else rev_hinge(T, S, rt, op, joint_rec(T, S, idx), idx, A, B, ready);
  };
  if constexpr (!ROWS) if (T.blk_single) {
    const bool on = warp == 0 && st0[0] != 0;
    const BlkOp op = blk_op(T, 0);
    const int a = op.a(), b = op.b();
    RevBody A, B;
    SL vw = S.at(T.sm_vw);
    rev_init(T, S, a, A);
    rev_init(T, S, b, B);
    rev_load(T, S, vw, a, A);
    rev_load(T, S, vw, b, B);
    for (int it = T.iters - 1; it >= 0; --it) {
      rev_begin_sweep<ROWS>(T, tp, it);
      const RevTape rt = rev_tape<ROWS>(T, S, it);
      if (!on) continue;
      vw = rt.vw;
      if (a >= 0) { A.v = vw.v3(6 * a); A.w = vw.v3(6 * a + 3); }
      if (b >= 0) { B.v = vw.v3(6 * b); B.w = vw.v3(6 * b + 3); }
      rows(op, rt, A, B, [] {});
    }
    if (on) { rev_store(T, S, vw, a, A, true); rev_store(T, S, vw, b, B, true); }
    cta_sync();
    return;
  }
  for (int it = T.iters - 1; it >= 0; --it) {
    rev_begin_sweep<ROWS>(T, tp, it);
    const RevTape rt = rev_tape<ROWS>(T, S, it);
    const uint8_t* st = st0;
    int e = *st++;
    bool pend = false;  // a level's barrier to meet before the next velocities are read
    BlkOp nop = blk_op(T, e & 63);
    while (e) {
      const int nxt = *st++;
      const BlkOp op = nop;
      nop = blk_op(T, nxt & 63);  // the next entry's block while this one runs
      if (e & BS_OP) {
        const int a = op.a(), b = op.b(), type = op.type();
        const bool lin = type <= BT_JOINT || type >= BT_GROUND;
        Body A, B;
        if constexpr (ROWS) {
          rx_init(T, S, a, A);
          rx_init(T, S, b, B);
          rows(op, rt, A, B, [&] {
            if (pend) cta_sync();
            rx_load(T, S, rt.vw, a, A);
            rx_load(T, S, rt.vw, b, B);
          });
          rx_store(T, S, rt.vw, a, A, lin);
          rx_store(T, S, rt.vw, b, B, lin);
        } else {
          rev_init(T, S, a, A);
          rev_init(T, S, b, B);
          rows(op, rt, A, B, [&] {
            if (pend) cta_sync();
            rev_load(T, S, rt.vw, a, A);
            rev_load(T, S, rt.vw, b, B);
          });
          rev_store(T, S, rt.vw, a, A, lin);
          rev_store(T, S, rt.vw, b, B, lin);
        }
      } else if (pend) {
        cta_sync();
      }
      pend = e & BS_BAR;  // (the last one is met with the next sweep's)
      e = nxt;
    }
  }
  cta_sync();
}

// ------------------------------------------------------------------------------ items
struct RevCtx {
  SL S, X, XB, VB;
  GC P;
  GL G;
  int i;
  float dl;
};

// Joint j after the sweeps: the start's application (impulses lam0, NULL without a warm start),
// the effective masses, and everything pushed to the bodies' poses; the package over the record.
__device__ __forceinline__ void joint_reverse(const DevTopo& T, const RevCtx& C, const TapeStep& tp, bool ws, int j) {
  const SL& S = C.S;
  const float bh = T.beta / T.dt;
  const int a = T.ja[j], b = T.jb[j], s0 = T.jslot[j];
  const SL R = joint_rec(T, S, j);
  const SL Q = R.at(JR_N);
  RevBody A, B;
  A.imb = B.imb = 0.f;
#pragma unroll
  for (int q = 0; q < 6; ++q) A.sb[q] = B.sb[q] = A.ii[q] = 0.f;
  A.vb = A.wb = f3(0.f, 0.f, 0.f);
  if (a >= 0) { load6(S, T.sm_iinv + 6 * a, A.ii); A.vb = C.VB.v3(6 * a); A.wb = C.VB.v3(6 * a + 3); }
  load6(S, T.sm_iinv + 6 * b, B.ii);
  B.vb = C.VB.v3(6 * b);
  B.wb = C.VB.v3(6 * b + 3);
  const float3 uAw = symv(A.ii, A.wb), uBw = symv(B.ii, B.wb);  // I^-1 w_bar
  const float3 ra = R.v3(JF_RA), rb = R.v3(JF_RB);
  float3 rab = Q.v3(JA_RA), rbb = Q.v3(JA_RB);
  float3 Cb = f3(0.f, 0.f, 0.f);
  auto lin = [&](auto KI) {
    constexpr int k = decltype(KI)::value;
    const float me = R[JF_ME + k], Kb = -me * me * Q[JA_ME + k];
    if (ws) {
      const float l = tp.lam0[(s0 + k) * 32];
      add_e_cross<k>(rab, l, uAw);
      add_e_cross<k>(rbb, -l, uBw);
      sym_outer_axis<k>(A.sb, l * A.wb, ra);
      sym_outer_axis<k>(B.sb, -l * B.wb, rb);
      A.imb = fmaf(l, axis_of<k>(A.vb), A.imb);
      B.imb = fmaf(-l, axis_of<k>(B.vb), B.imb);
    }
    // K = im_a + ang_a . I_a^-1 ang_a + ...
    const float3 aa = cross_axis<k>(ra), ab = cross_axis<k>(rb);
    add_e_cross<k>(rab, 2.f * Kb, symv_axis<k>(A.ii, ra));
    add_e_cross<k>(rbb, 2.f * Kb, symv_axis<k>(B.ii, rb));
    sym_outer_axis<k>(A.sb, Kb * aa, ra);
    sym_outer_axis<k>(B.sb, Kb * ab, rb);
    A.imb += Kb;
    B.imb += Kb;
    axis_of<k>(Cb) = bh * Q[JA_BI + k];
  };
  lin(std::integral_constant<int, 0>{});
  lin(std::integral_constant<int, 1>{});
  lin(std::integral_constant<int, 2>{});
  const M3 Ra = body_R(C.X, a), Rb = loadR(C.X, 18 * b);
  rab = a >= 0 ? rab + Cb : Cb;  // a world anchor moves only the position error
  rbb = rbb - Cb;
  const float3 anca = C.P.v3(T.o_anchor + 6 * j), ancb = C.P.v3(T.o_anchor + 6 * j + 3);
  C.G.red3(T.o_anchor + 6 * j, mtv(Ra, rab));  // (identity for the world)
  C.G.red3(T.o_anchor + 6 * j + 3, mtv(Rb, rbb));
  float ga[9], gb[9];
  {
    const float r[3] = {rab.x, rab.y, rab.z}, c[3] = {anca.x, anca.y, anca.z};
    const float s[3] = {rbb.x, rbb.y, rbb.z}, d[3] = {ancb.x, ancb.y, ancb.z};
#pragma unroll
    for (int q = 0; q < 9; ++q) { ga[q] = r[q / 3] * c[q % 3]; gb[q] = s[q / 3] * d[q % 3]; }
  }
  if (T.jtype[j] == 1) {
    float3 tau[2];
    onb3(C.P.v3(T.o_axis + 6 * j), tau[0], tau[1]);
    const float3 axb = C.P.v3(T.o_axis + 6 * j + 3);
    const float3 ub = mv(Rb, axb), ua = S.v3(T.sm_ua + 3 * j);
    const float3 cr = cross3(ub, ua);
    float3 uab = f3(0.f, 0.f, 0.f), ubb = uab;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const float me = R[JF_ME + 3 + k], Kb = -me * me * Q[JA_ME + 3 + k], bib = bh * Q[JA_BI + 3 + k];
      const float3 t = R.v3(JF_T + 3 * k);
      float3 tb = Q.v3(JA_T + 3 * k);
      if (ws) {
        const float l = tp.lam0[(s0 + 3 + k) * 32];
        tb = tb + l * (uAw - uBw);
        sym_outer(A.sb, l * A.wb, t);
        sym_outer(B.sb, -l * B.wb, t);
      }
      tb = tb + (2.f * Kb) * (symv(A.ii, t) + symv(B.ii, t));
      sym_outer(A.sb, Kb * t, t);
      sym_outer(B.sb, Kb * t, t);
      tb = tb + bib * cr;
      const float3 crb = bib * t;
      uab += cross3(crb, ub);  // c = ub x ua
      ubb += cross3(ua, crb);
      const float v[3] = {tb.x, tb.y, tb.z}, c[3] = {tau[k].x, tau[k].y, tau[k].z};
#pragma unroll
      for (int q = 0; q < 9; ++q) ga[q] = fmaf(v[q / 3], c[q % 3], ga[q]);
    }
    {
      const float v[3] = {ubb.x, ubb.y, ubb.z}, c[3] = {axb.x, axb.y, axb.z};
#pragma unroll
      for (int q = 0; q < 9; ++q) gb[q] = fmaf(v[q / 3], c[q % 3], gb[q]);
    }
    const int fl = T.jflags[j];
    float thb = 0.f, wstb = 0.f;
    if (fl) {
      uab += Q.v3(JA_U);
      const float3 IA = symv(A.ii, ua), IB = symv(B.ii, ua);
      float Kb = 0.f;
      if (fl & 1) {
        const float me = R[JF_ME + 5];
        if (me != 0.f) {  // (an inactive lane's accumulators hold nothing of use)
          Kb += -me * me * Q[JA_ME + 5];
          const float g = bh * Q[JA_BI + 5];
          const bool low = R[JF_LS] > 0.f;
          thb = low ? g : -g;
          C.G.red(T.o_limit + 2 * j + (low ? 0 : 1), low ? -g : g);
        }
      }
      if (fl & 2) {
        const float me = R[JF_ME + 6];
        Kb += -me * me * Q[JA_ME + 6];
        wstb = -Q[JA_BI + 6];
        C.G.red(T.o_motor + 3 * j + 1, T.dt * Q[JA_BND]);
        if (ws) {
          const float l = tp.lam0[T.jmot[j] * 32];
          uab += l * (uBw - uAw);
          sym_outer(A.sb, -l * A.wb, ua);
          sym_outer(B.sb, l * B.wb, ua);
        }
      }
      uab += (2.f * Kb) * (IA + IB);
      sym_outer(A.sb, Kb * ua, ua);
      sym_outer(B.sb, Kb * ua, ua);
    }
    S[T.sm_thb + j] = thb;
    S[T.sm_thdb + j] = 0.f;
    S[T.sm_wstb + j] = wstb;
    S.s3(T.sm_uab + 3 * j, uab);
  } else {
    S[T.sm_thb + j] = S[T.sm_thdb + j] = S[T.sm_wstb + j] = 0.f;
    S.s3(T.sm_uab + 3 * j, f3(0.f, 0.f, 0.f));
  }
  R.s3(JP_P, Cb);
#pragma unroll
  for (int q = 0; q < 9; ++q) { R[JP_RA + q] = ga[q]; R[JP_RB + q] = gb[q]; }
#pragma unroll
  for (int q = 0; q < 6; ++q) { R[JP_SA + q] = A.sb[q]; R[JP_SB + q] = B.sb[q]; }
  R[JP_IA] = A.imb;
  R[JP_IB] = B.imb;
}

// Ground contact q after the sweeps (rows of an inactive lane are constants: an empty package).
__device__ __forceinline__ void contact_reverse(const DevTopo& T, const RevCtx& C, const TapeStep& tp, bool ws, int q) {
  const SL& S = C.S;
  const float bh = T.beta / T.dt;
  const int a = T.sbody[q], s0 = T.cslot + 3 * q;
  const SL R = contact_rec(T, S, q);
  const SL Q = R.at(CR_N);
  float sb[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, imb = 0.f, db = 0.f, vnb = 0.f;
  float g[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  float3 wadd = f3(0.f, 0.f, 0.f);
  if (R[CF_ME] != 0.f) {
    float ii[6];
    load6(S, T.sm_iinv + 6 * a, ii);
    const float3 ra = R.v3(CF_RA), vb = C.VB.v3(6 * a), wb = C.VB.v3(6 * a + 3);
    const float3 uw = symv(ii, wb);
    float3 rab = Q.v3(CA_RA);
    auto row = [&](auto MI, auto AI) {
      constexpr int m = decltype(MI)::value, ax = decltype(AI)::value;
      const float me = R[CF_ME + m], Kb = -me * me * Q[CA_ME + m];
      if (ws) {
        const float l = tp.lam0[(s0 + m) * 32];
        add_e_cross<ax>(rab, l, uw);
        sym_outer_axis<ax>(sb, l * wb, ra);
        float3 vv = vb;
        imb = fmaf(l, axis_of<ax>(vv), imb);
      }
      add_e_cross<ax>(rab, 2.f * Kb, symv_axis<ax>(ii, ra));
      sym_outer_axis<ax>(sb, Kb * cross_axis<ax>(ra), ra);
      imb += Kb;
    };
    using I0 = std::integral_constant<int, 0>;
    using I1 = std::integral_constant<int, 1>;
    using I2 = std::integral_constant<int, 2>;
    row(I0{}, I2{});
    row(I1{}, I0{});
    row(I2{}, I1{});
    const M3 Ra = loadR(C.X, 18 * a);
    const float3 off = C.P.v3(T.o_sph_off + 3 * q);
    const float rad = C.P[T.o_sph_rad + q];
    const float d = (C.X[18 * a + 2] + mv(Ra, off).z) - rad - T.ground_z;
    const float biasb = Q[CA_BI];
    const float3 vm = f3(tp.vminus[(6 * a) * 32], tp.vminus[(6 * a + 1) * 32], tp.vminus[(6 * a + 2) * 32]);
    const float3 wm = f3(tp.vminus[(6 * a + 3) * 32], tp.vminus[(6 * a + 4) * 32], tp.vminus[(6 * a + 5) * 32]);
    const float3 an = cross_axis<2>(ra);
    const float vn = vm.z + dot3(an, wm);
    if (d + T.slop < 0.f) db = bh * biasb;
    if (vn < 0.f) {
      C.G.red(T.o_sph_e + q, vn * biasb);
      vnb = C.P[T.o_sph_e + q] * biasb;
      wadd = vnb * an;
      add_e_cross<2>(rab, vnb, wm);
    }
    C.G.red(T.o_sph_mu + q, Q[CA_MU]);
    const float3 cb = rab + f3(0.f, 0.f, db);
    C.G.red3(T.o_sph_off + 3 * q, mtv(Ra, cb));
    C.G.red(T.o_sph_rad + q, -rab.z - db);
    const float v[3] = {cb.x, cb.y, cb.z}, c[3] = {off.x, off.y, off.z};
#pragma unroll
    for (int k = 0; k < 9; ++k) g[k] = v[k / 3] * c[k % 3];
  }
  R[CP_Z] = db;
#pragma unroll
  for (int k = 0; k < 9; ++k) R[CP_R + k] = g[k];
#pragma unroll
  for (int k = 0; k < 6; ++k) R[CP_S + k] = sb[k];
  R[CP_I] = imb;
  R[CP_V] = vnb;
  R.s3(CP_W, wadd);
}

// Sphere pair p after the sweeps.
static __device__ __noinline__ void pair_reverse(const DevTopo& T, const RevCtx& C, const TapeStep tp, bool ws, int p) {
  const SL& S = C.S;
  const float bh = T.beta / T.dt;
  const int k = T.pk[p], l = T.pl[p], a = T.sbody[k], b = T.sbody[l], s0 = T.cslot + 3 * (T.ns + p);
  const SL R = pair_rec(T, S, p);
  const SL Q = R.at(PR_N);
  float sa[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, sb[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, ima_b = 0.f, imb_b = 0.f;
  const float3 z3 = f3(0.f, 0.f, 0.f);
  float3 dlb = z3, ckb = z3, clb = z3, vadd = z3, wadda = z3, waddb = z3, goffk = z3, goffl = z3;
  float rkb = 0.f, rlb = 0.f, muk_b = 0.f, mul_b = 0.f, ek_b = 0.f, el_b = 0.f;
  const float3 offk = C.P.v3(T.o_sph_off + 3 * k), offl = C.P.v3(T.o_sph_off + 3 * l);
  if (R[PF_ME] != 0.f) {
    float ia[6], ib[6];
    load6(S, T.sm_iinv + 6 * a, ia);
    load6(S, T.sm_iinv + 6 * b, ib);
    const float ima = S[T.sm_invm + a], imb = S[T.sm_invm + b];
    const float3 va = C.VB.v3(6 * a), wa = C.VB.v3(6 * a + 3), vb = C.VB.v3(6 * b), wb = C.VB.v3(6 * b + 3);
    const M3 Ra = loadR(C.X, 18 * a), Rb = loadR(C.X, 18 * b);
    const float3 ck = mv(Ra, offk), cl = mv(Rb, offl);
    const float3 dv = (C.X.v3(18 * a) + ck) - (C.X.v3(18 * b) + cl);
    const float dist = sqrtf(dot3(dv, dv));
    const bool deg = !(dist > 1e-9f);
    const float3 n = R.v3(PF_LIN);
    const float rk = C.P[T.o_sph_rad + k], rl = C.P[T.o_sph_rad + l];
    const float3 ra = ck - rk * n, rb = cl + rl * n;
    float3 nb = z3;
    float distb = 0.f;
    for (int m = 0; m < 3; ++m) {
      const float me = R[PF_ME + m], Kb = -me * me * Q[PA_ME + m];
      const float3 lin = R.v3(PF_LIN + 3 * m), angA = R.v3(PF_ANGA + 3 * m), angB = R.v3(PF_ANGB + 3 * m);
      float3 linb = Q.v3(PA_LIN + 3 * m), angAb = Q.v3(PA_ANGA + 3 * m), angBb = Q.v3(PA_ANGB + 3 * m);
      if (ws) {
        const float l0 = tp.lam0[(s0 + m) * 32];
        const float3 ga = l0 * wa, gb = l0 * wb;
        linb += l0 * (ima * va - imb * vb);
        angAb += symv(ia, ga);
        angBb += symv(ib, gb);
        sym_outer(sa, ga, angA);
        sym_outer(sb, gb, angB);
        ima_b += l0 * dot3(lin, va);
        imb_b -= l0 * dot3(lin, vb);
      }
      const float ll = dot3(lin, lin);
      linb += (2.f * Kb * (ima + imb)) * lin;
      angAb += (2.f * Kb) * symv(ia, angA);
      angBb += (2.f * Kb) * symv(ib, angB);
      sym_outer(sa, Kb * angA, angA);
      sym_outer(sb, Kb * angB, angB);
      ima_b += Kb * ll;
      imb_b += Kb * ll;
      if (m == 0) {
        const float3 vma = f3(tp.vminus[(6 * a) * 32], tp.vminus[(6 * a + 1) * 32], tp.vminus[(6 * a + 2) * 32]);
        const float3 wma = f3(tp.vminus[(6 * a + 3) * 32], tp.vminus[(6 * a + 4) * 32], tp.vminus[(6 * a + 5) * 32]);
        const float3 vmb = f3(tp.vminus[(6 * b) * 32], tp.vminus[(6 * b + 1) * 32], tp.vminus[(6 * b + 2) * 32]);
        const float3 wmb = f3(tp.vminus[(6 * b + 3) * 32], tp.vminus[(6 * b + 4) * 32], tp.vminus[(6 * b + 5) * 32]);
        const float biasb = Q[PA_BI];
        const float vn = dot3(n, vma - vmb) + dot3(angA, wma) + dot3(angB, wmb);
        if (dist - rk - rl + T.slop < 0.f) distb += bh * biasb;
        if (vn < 0.f) {
          const float ek = C.P[T.o_sph_e + k], el = C.P[T.o_sph_e + l];
          (ek >= el ? ek_b : el_b) = vn * biasb;
          const float vnb = (ek >= el ? ek : el) * biasb;
          nb += vnb * (vma - vmb);
          vadd = vnb * n;
          wadda = vnb * angA;
          waddb = vnb * angB;
          angAb += vnb * wma;
          angBb += vnb * wmb;
        }
        nb += linb + cross3(angAb, ra) - cross3(angBb, rb);  // angA = ra x n, angB = -(rb x n)
      } else {
        const float3 tb = linb + cross3(angAb, ra) - cross3(angBb, rb);
        if (!deg) nb += onb3_vjp(n, m == 1 ? tb : z3, m == 2 ? tb : z3);
        const float muk = C.P[T.o_sph_mu + k], mul = C.P[T.o_sph_mu + l], mu = sqrtf(muk * mul);
        if (m == 1 && mu > 0.f) {
          const float mub = Q[PA_MU];
          muk_b = mub * mul / (2.f * mu);
          mul_b = mub * muk / (2.f * mu);
        }
      }
      const float3 rab = cross3(lin, angAb), rbb = -cross3(lin, angBb);
      rkb -= dot3(rab, n); nb -= rk * rab;  // ra = ck - rk n, rb = cl + rl n
      rlb += dot3(rbb, n); nb += rl * rbb;
      ckb += rab;
      clb += rbb;
    }
    rkb -= distb; rlb -= distb;  // d = dist - rk - rl
    dlb = deg ? z3 : distb * n + (1.f / dist) * (nb - dot3(n, nb) * n);
    ckb += dlb;
    clb -= dlb;
    goffk = mtv(Ra, ckb);
    goffl = mtv(Rb, clb);
  }
  R.s3(PP_P, dlb);
  const float v[3] = {ckb.x, ckb.y, ckb.z}, c[3] = {offk.x, offk.y, offk.z};
  const float w[3] = {clb.x, clb.y, clb.z}, e[3] = {offl.x, offl.y, offl.z};
  for (int q = 0; q < 9; ++q) { R[PP_RA + q] = v[q / 3] * c[q % 3]; R[PP_RB + q] = w[q / 3] * e[q % 3]; }
  for (int q = 0; q < 6; ++q) { R[PP_SA + q] = sa[q]; R[PP_SB + q] = sb[q]; }
  R[PP_IA] = ima_b;
  R[PP_IB] = imb_b;
  R.s3(PP_V, vadd);
  R.s3(PP_WA, wadda);
  R.s3(PP_WB, waddb);
  R.s3(PP_GK + PG_OFF, goffk);
  R[PP_GK + PG_RAD] = rkb; R[PP_GK + PG_MU] = muk_b; R[PP_GK + PG_E] = ek_b;
  R.s3(PP_GL + PG_OFF, goffl);
  R[PP_GL + PG_RAD] = rlb; R[PP_GL + PG_MU] = mul_b; R[PP_GL + PG_E] = el_b;
}

// The pairs' shares of sphere q's parameter gradients, in pair order (the sphere's contact has added its
// own, before the barrier). Several pairs and the ground contact of a sphere belong to different warps:
// added where they are formed, their order, and the sums' last bits, would change from run to run.
__device__ __forceinline__ void sphere_reverse(const DevTopo& T, const RevCtx& C, int q) {
  for (int p = 0; p < T.np; ++p) {
    if (!blk_live(T)[T.nj + T.ns + p] || (T.pk[p] != q && T.pl[p] != q)) continue;
    const SL R = pair_rec(T, C.S, p).at(T.pk[p] == q ? PP_GK : PP_GL);
    C.G.red3(T.o_sph_off + 3 * q, R.v3(PG_OFF));
    C.G.red(T.o_sph_rad + q, R[PG_RAD]);
    C.G.red(T.o_sph_mu + q, R[PG_MU]);
    C.G.red(T.o_sph_e + q, R[PG_E]);
  }
}

// Body b: the packages of its items (slot order) into the pose adjoint and the adjoints of the
// solver's input velocities and of its inverse mass and inertia, then the reverse of the external
// impulses (see external_reverse).
__device__ __forceinline__ void body_reverse(const DevTopo& T, const RevCtx& C, int b) {
  const SL& S = C.S;
  const uint8_t* first = blk_bytes(T) + T.blk_inc0;
  const uint8_t* inc = blk_bytes(T) + T.blk_inc;
  float sb[6], imb = S[T.sm_invmb + b];
  load6(S, T.sm_iinvb + 6 * b, sb);
  float3 vb = C.VB.v3(6 * b), wmb = C.VB.v3(6 * b + 3), pb = C.XB.v3(18 * b);
  float gR[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) gR[q] = C.XB[18 * b + 3 + q];
  const int k1 = first[b + 1];
  for (int k = first[b]; k < k1; ++k) {
    const int e = inc[k], idx = e & 31;
    const bool side = e & 0x20;
    if (e < 0x40) {
      const SL R = joint_rec(T, S, idx);
      const float3 c = R.v3(JP_P);
      pb = side ? pb - c : pb + c;
#pragma unroll
      for (int q = 0; q < 9; ++q) gR[q] += R[(side ? JP_RB : JP_RA) + q];
#pragma unroll
      for (int q = 0; q < 6; ++q) sb[q] += R[(side ? JP_SB : JP_SA) + q];
      imb += R[side ? JP_IB : JP_IA];
    } else if (e < 0x80) {
      const SL R = contact_rec(T, S, idx);
      pb.z += R[CP_Z];
#pragma unroll
      for (int q = 0; q < 9; ++q) gR[q] += R[CP_R + q];
#pragma unroll
      for (int q = 0; q < 6; ++q) sb[q] += R[CP_S + q];
      imb += R[CP_I];
      vb.z += R[CP_V];
      wmb += R.v3(CP_W);
    } else {
      const SL R = pair_rec(T, S, idx);
      const float3 c = R.v3(PP_P), v = R.v3(PP_V);
      pb = side ? pb - c : pb + c;
      vb = side ? vb - v : vb + v;
      wmb += R.v3(side ? PP_WB : PP_WA);
#pragma unroll
      for (int q = 0; q < 9; ++q) gR[q] += R[(side ? PP_RB : PP_RA) + q];
#pragma unroll
      for (int q = 0; q < 6; ++q) sb[q] += R[(side ? PP_SB : PP_SA) + q];
      imb += R[side ? PP_IB : PP_IA];
    }
  }
  const float h = T.dt;
  const M3 R = loadR(C.X, 18 * b);
  const float3 I = C.P.v3(T.o_inertia + 3 * b);
  const float3 Ii = f3(1.f / I.x, 1.f / I.y, 1.f / I.z);
  const float m = C.P[T.o_mass + b];
  float iw[6], ii[6];
  rot_diag6(R, I, iw);
  rot_diag6(R, Ii, ii);
  const float3 w = C.X.v3(18 * b + 15);
  const float3 z = symv(iw, w);
  const float3 gy = -cross3(w, z);
  // w- = w + h Iinv gy: adjoint of Iinv (symmetric part, as in RevBody) and of w
  sym_outer(sb, h * wmb, gy);
  const float3 gyb = h * symv(ii, wmb);
  float3 wb = wmb - cross3(z, gyb);
  const float3 zb = cross3(w, gyb);
  wb += symv(iw, zb);
  float sw[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};  // adjoint of Iw = zb w^T
  sym_outer(sw, zb, w);
  // R diag(d) R^T reverse: Rbar += (G + G^T) R diag(d), dbar_k = (R^T G R)_kk
  float Ib[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float di = c == 0 ? Ii.x : (c == 1 ? Ii.y : Ii.z), dw = c == 0 ? I.x : (c == 1 ? I.y : I.z);
    const float r0 = R.m[c], r1 = R.m[3 + c], r2 = R.m[6 + c];
    const float s0 = 2.f * sb[0] * r0 + sb[1] * r1 + sb[2] * r2, s1 = sb[1] * r0 + 2.f * sb[3] * r1 + sb[4] * r2,
                s2 = sb[2] * r0 + sb[4] * r1 + 2.f * sb[5] * r2;
    const float t0 = 2.f * sw[0] * r0 + sw[1] * r1 + sw[2] * r2, t1 = sw[1] * r0 + 2.f * sw[3] * r1 + sw[4] * r2,
                t2 = sw[2] * r0 + sw[4] * r1 + 2.f * sw[5] * r2;
    gR[c] += s0 * di + t0 * dw;
    gR[3 + c] += s1 * di + t1 * dw;
    gR[6 + c] += s2 * di + t2 * dw;
    Ib[c] = 0.5f * (t0 * r0 + t1 * r1 + t2 * r2) - 0.5f * (s0 * r0 + s1 * r1 + s2 * r2) * di * di;
  }
  C.XB.s3(18 * b, pb);
#pragma unroll
  for (int q = 0; q < 9; ++q) C.XB[18 * b + 3 + q] = gR[q];
  C.XB.a3(18 * b + 12, vb);
  C.XB.a3(18 * b + 15, wb);
  C.G.red3(T.o_inertia + 3 * b, f3(Ib[0], Ib[1], Ib[2]));
  C.G.red(T.o_mass + b, -(imb / (m * m)));
}

// Hinge kinematics of joint j reversed: axis, angle and rate adjoints to its bodies' R and w; the
// package over the record.
__device__ __forceinline__ void hinge_reverse_item(const DevTopo& T, const RevCtx& C, int j) {
  const SL& S = C.S;
  const int a = T.ja[j], b = T.jb[j];
  float3 uab = S.v3(T.sm_uab + 3 * j), wj = f3(0.f, 0.f, 0.f);
  const M3 Ra = body_R(C.X, a);
  const float3 axa = C.P.v3(T.o_axis + 6 * j);
  const float3 ua = S.v3(T.sm_ua + 3 * j);
  float ga[9], gb[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) ga[q] = gb[q] = 0.f;
  if (T.jtype[j] == 1) {
    const M3 Rb = loadR(C.X, 18 * b);
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
    wj = thdb * ua;
    const float u[3] = {wab.x, wab.y, wab.z}, r[3] = {refa.x, refa.y, refa.z};
    const float v[3] = {wbb.x, wbb.y, wbb.z}, s[3] = {refb.x, refb.y, refb.z};
#pragma unroll
    for (int q = 0; q < 9; ++q) { ga[q] = u[q / 3] * r[q % 3]; gb[q] = v[q / 3] * s[q % 3]; }
  }
  const float u[3] = {uab.x, uab.y, uab.z}, r[3] = {axa.x, axa.y, axa.z};
#pragma unroll
  for (int q = 0; q < 9; ++q) ga[q] = fmaf(u[q / 3], r[q % 3], ga[q]);
  const SL R = joint_rec(T, S, j);
  R.s3(HP_W, wj);
#pragma unroll
  for (int q = 0; q < 9; ++q) { R[HP_RA + q] = ga[q]; R[HP_RB + q] = gb[q]; }
}
__device__ __forceinline__ void hinge_reverse_body(const DevTopo& T, const RevCtx& C, int b) {
  const uint8_t* first = blk_bytes(T) + T.blk_inc0;
  const uint8_t* inc = blk_bytes(T) + T.blk_inc;
  float3 w = C.XB.v3(18 * b + 15);
  float gR[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) gR[q] = C.XB[18 * b + 3 + q];
  const int k1 = first[b + 1];
  for (int k = first[b]; k < k1 && inc[k] < 0x40; ++k) {
    const SL R = joint_rec(T, C.S, inc[k] & 31);
    const bool side = inc[k] & 0x20;
    const float3 c = R.v3(HP_W);
    w = side ? w + c : w - c;
#pragma unroll
    for (int q = 0; q < 9; ++q) gR[q] += R[(side ? HP_RB : HP_RA) + q];
  }
  C.XB.s3(18 * b + 15, w);
#pragma unroll
  for (int q = 0; q < 9; ++q) C.XB[18 * b + 3 + q] = gR[q];
}

// Every joint's hinge kinematics reversed (every warp calls; ends after a CTA barrier).
template <class Q>
__device__ __forceinline__ void blk_hinge_reverse(const DevTopo& T, const RevCtx& C, int warp) {
  if constexpr (Q::SEQ) {
    for (int j = warp; j < T.nj; j += blk_nw()) rx_hinge_item(T, C, j);
    cta_sync();
    for (int b = warp; b < T.nb; b += blk_nw()) rx_hinge_body(T, C, b);
  } else {
    for (int j = warp; j < T.nj; j += blk_nw()) hinge_reverse_item(T, C, j);
    cta_sync();
    for (int b = warp; b < T.nb; b += blk_nw()) hinge_reverse_body(T, C, b);
  }
  cta_sync();
}

// Features reversed, split: angle and rate adjoints to the joints of this warp; the rest (torso
// sensors, target vector) to the pose adjoint by warp 3, when no other warp writes it.
template <class AV>
__device__ __forceinline__ void features_reverse_joints(const DevTopo& T, const SL& S, const AV& sbar, int warp) {
  int k = 0;
  if (T.features & 1) {
    for (int m = 0; m < T.n_motors; ++m)
      if ((T.motor_joint[m] & (blk_nw() - 1)) == warp) S[T.sm_thb + T.motor_joint[m]] += sbar[k + m];
    k += T.n_motors;
  }
  if (T.features & 2)
    for (int m = 0; m < T.n_motors; ++m)
      if ((T.motor_joint[m] & (blk_nw() - 1)) == warp) S[T.sm_thdb + T.motor_joint[m]] += sbar[k + m];
}
template <class AV>
__device__ __forceinline__ void features_reverse_rest(const DevTopo& T, const RevCtx& C, const AV& sbar) {
  int k = 0;
  if (T.features & 1) k += T.n_motors;
  if (T.features & 2) k += T.n_motors;
  if (T.features & 4) k += 2;
  if (T.features & 8) {
    const int b = T.imu_body;
    const M3 R = loadR(C.X, 18 * b);
    const float3 w = C.X.v3(18 * b + 15);
    const float3 gb = f3(sbar[k], sbar[k + 1], sbar[k + 2]), wlb = f3(sbar[k + 3], sbar[k + 4], sbar[k + 5]);
    k += 6;
    // g = R^T (0,0,-1)  -> Rbar[2][c] -= gb_c ;  wl = R^T w -> Rbar += w wlb^T, wbar += R wlb
    C.XB[18 * b + 3 + 6] -= gb.x; C.XB[18 * b + 3 + 7] -= gb.y; C.XB[18 * b + 3 + 8] -= gb.z;
    add_outer(C.XB, 18 * b + 3, w, wlb);
    C.XB.a3(18 * b + 15, mv(R, wlb));
  }
  if (T.features & 16) {
    const int b = T.loss_body;
    const M3 R = loadR(C.X, 18 * b);
    const float3 c = C.P.v3(T.o_loss_point);
    const float3 qb = f3(sbar[k], sbar[k + 1], sbar[k + 2]);
    C.XB.a3(18 * b, qb);
    add_outer(C.XB, 18 * b + 3, qb, c);
    C.G.red3(T.o_loss_point, mtv(R, qb));
    C.G.red3(T.o_loss_target, -qb);
  }
}

// ------------------------------------------------------------------------------ controller
// Stores one 16-row tile's deltas: fp32 to the dump rows, hi + lo bfloat16 to the two planes.
template <int H, int NT>
__device__ __forceinline__ void store_delta(const float (&d)[NT][4], int mt, int n1, __nv_bfloat16* hi, __nv_bfloat16* lo,
                                            float* dump, size_t N) {
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
    const int c = n1 + nt * 8 + 2 * q, r0 = mt * 16 + g;
    float h[4], l[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      h[k] = __bfloat162float(__float2bfloat16_rn(d[nt][k]));
      l[k] = d[nt][k] - h[k];
    }
    *reinterpret_cast<uint32_t*>(hi + r0 * (H + 8) + c) = pack_bf16(h[0], h[1]);
    *reinterpret_cast<uint32_t*>(hi + (r0 + 8) * (H + 8) + c) = pack_bf16(h[2], h[3]);
    *reinterpret_cast<uint32_t*>(lo + r0 * (H + 8) + c) = pack_bf16(l[0], l[1]);
    *reinterpret_cast<uint32_t*>(lo + (r0 + 8) * (H + 8) + c) = pack_bf16(l[2], l[3]);
    dump[(size_t)c * N + r0] = d[nt][0];
    dump[(size_t)(c + 1) * N + r0] = d[nt][1];
    dump[(size_t)c * N + r0 + 8] = d[nt][2];
    dump[(size_t)(c + 1) * N + r0 + 8] = d[nt][3];
  }
}
// Zeroes the deltas of hidden units that were not positive (act: the layer's dump rows).
template <int NT>
__device__ __forceinline__ void mask_delta(float (&d)[NT][4], int mt, int n1, const float* act, size_t N) {
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
    const int c = n1 + nt * 8 + 2 * q, r0 = mt * 16 + g;
    if (!(act[(size_t)c * N + r0] > 0.f)) d[nt][0] = 0.f;
    if (!(act[(size_t)(c + 1) * N + r0] > 0.f)) d[nt][1] = 0.f;
    if (!(act[(size_t)c * N + r0 + 8] > 0.f)) d[nt][2] = 0.f;
    if (!(act[(size_t)(c + 1) * N + r0 + 8] > 0.f)) d[nt][3] = 0.f;
  }
}
// The tensor-core controller reversed on the CTA's warps: ub the output adjoint, sbar receives the
// input adjoint, col the step's dump column of lane 0. The planes (four of [32][H + 8] bfloat16) lie
// over the records, whose packages have been added up by then. Ends before a barrier.
template <int H, int NW>
__device__ __forceinline__ void ctrl_backward_nw(const DevTopo& T, const DevPtrs& D, const SL& ub, const SL& sbar, float* col,
                                                 int warp) {
  constexpr int NT = H / (8 * NW), KT = H / 16;
  constexpr CtrlTCLayout Lw = ctrl_tc_layout(H, H);
  const __nv_bfloat16* Wc = D.Wtc;
  const size_t N = (size_t)T.horizon * T.Bp;
  const int n1 = warp * (H / NW), no = T.widths[3], lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  __nv_bfloat16* p0 = reinterpret_cast<__nv_bfloat16*>(g_smem + T.sm_hbuf * 32);
  __nv_bfloat16 *h2 = p0, *l2 = p0 + 32 * (H + 8), *h1 = p0 + 64 * (H + 8), *l1 = p0 + 96 * (H + 8);
#pragma unroll
  for (int mt = 0; mt < 2; ++mt) {
    float d3[2][4];
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      const int c = nt * 8 + 2 * q, r0 = mt * 16 + g, r1 = r0 + 8;
      d3[nt][0] = c < no ? ub.lane_at(c, r0) : 0.f;
      d3[nt][1] = c + 1 < no ? ub.lane_at(c + 1, r0) : 0.f;
      d3[nt][2] = c < no ? ub.lane_at(c, r1) : 0.f;
      d3[nt][3] = c + 1 < no ? ub.lane_at(c + 1, r1) : 0.f;
    }
    uint32_t hi[1][4], lo[1][4];
    split_to_a<2>(d3, hi, lo);
    float d2[NT][4];
    zero_acc<NT>(d2);
    mma_acc_split<1, NT>(hi, lo, Wc + Lw.w3t, CTRL_TC_NOP, n1, 0, d2);
    mask_delta<NT>(d2, mt, n1, col + (size_t)T.dump_act[2] * N, N);
    store_delta<H, NT>(d2, mt, n1, h2, l2, col + (size_t)T.dump_del[1] * N, N);
  }
  cta_sync();
  {
    float d1[2][NT][4];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) zero_acc<NT>(d1[mt]);
#pragma unroll 2
    for (int kt = 0; kt < KT; ++kt) {
      uint32_t ah[2][4], al[2][4];
#pragma unroll
      for (int mt = 0; mt < 2; ++mt) {
        load_a_smem<H>(h2, mt, kt, ah[mt]);
        load_a_smem<H>(l2, mt, kt, al[mt]);
      }
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        uint32_t b0, b1;
        load_b(Wc + Lw.w2t, H, n1 + nt * 8, kt * 16, b0, b1);
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
          mma_bf16_16816(d1[mt][nt], ah[mt], b0, b1);
          mma_bf16_16816(d1[mt][nt], al[mt], b0, b1);
        }
      }
    }
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
      mask_delta<NT>(d1[mt], mt, n1, col + (size_t)T.dump_act[1] * N, N);
      store_delta<H, NT>(d1[mt], mt, n1, h1, l1, col + (size_t)T.dump_del[0] * N, N);
    }
  }
  cta_sync();
  if (warp < CTRL_TC_KP0 / 8) {  // eight inputs a warp
    float s[2][1][4];
    zero_acc<1>(s[0]);
    zero_acc<1>(s[1]);
#pragma unroll 2
    for (int kt = 0; kt < KT; ++kt) {
      uint32_t b0, b1;
      load_b(Wc + Lw.w1t, H, warp * 8, kt * 16, b0, b1);
#pragma unroll
      for (int mt = 0; mt < 2; ++mt) {
        uint32_t ah[4], al[4];
        load_a_smem<H>(h1, mt, kt, ah);
        load_a_smem<H>(l1, mt, kt, al);
        mma_bf16_16816(s[mt][0], ah, b0, b1);
        mma_bf16_16816(s[mt][0], al, b0, b1);
      }
    }
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
      store_c<1>(s[mt], mt, warp * 8, T.widths[0], [&](int f, int r, float v) { sbar.lane_at(f, r) = v; });
  }
}
template <int H, int NW>
__device__ __noinline__ void ctrl_backward_nw_call(const DevTopo& T, const DevPtrs& D, SL ub, SL sbar, float* col, int warp) {
  ctrl_backward_nw<H, NW>(T, D, ub, sbar, col, warp);
}
template <class Q>
__device__ __forceinline__ void ctrl_backward_blk(const DevTopo& T, const DevPtrs& D, const SL& ub, const SL& sbar, float* col,
                                                  int warp) {
  if constexpr (Q::CTRL_H == 128) {
    ctrl_backward_nw<128, Q::NW>(T, D, ub, sbar, col, warp);
  } else if constexpr (Q::CTRL_H == 256) {
    ctrl_backward_nw_call<256, Q::NW>(T, D, ub, sbar, col, warp);
  } else {
    if (T.widths[1] == 64) ctrl_backward_nw_call<64, Q::NW>(T, D, ub, sbar, col, warp);
    else if (T.widths[1] == 128) ctrl_backward_nw_call<128, Q::NW>(T, D, ub, sbar, col, warp);
    else ctrl_backward_nw_call<256, Q::NW>(T, D, ub, sbar, col, warp);
  }
}
// The fp32-arithmetic controller reversed (see controller_reverse), 8 inputs of a layer per warp and
// pass; ping-pong buffers z0, z1 over the records.
__device__ __forceinline__ void controller_reverse_nw(const DevTopo& T, const DevPtrs& D, const GW* act, const GW* del,
                                                      const SL& z0, const SL& z1, const SL& sbar, int warp) {
  const int L = T.n_layers;
  SL cur = z0, nxt = z1;
  for (int l = L - 1; l >= 0; --l) {
    const int ni = T.widths[l], no = T.widths[l + 1];
    const float* Wn = D.Wn + T.w_off[l];
    if (l > 0) {
      dense_bwd(Wn, ni, no, cur, act[l], nxt, true, false, 8 * warp, 8 * blk_nw());
      cta_sync();
      for (int k = warp; k < ni; k += blk_nw()) del[l - 1][k] = nxt[k];
      const SL tmp = cur;
      cur = nxt;
      nxt = tmp;
    } else {
      dense_bwd(Wn, ni, no, cur, act[0], sbar, false, false, 8 * warp, 8 * blk_nw());
    }
  }
  if (T.skip)
    dense_bwd(D.Wn + T.w_off[L], T.widths[0], T.widths[L], del[L - 1], act[0], sbar, false, true, 8 * warp, 8 * blk_nw());
}

// ------------------------------------------------------------------------------ one step
// Step t + 1's look-ahead: the tape record of step ts, its state and the controller's activations into
// L2 while step t + 1 is reversed.
__device__ __forceinline__ void rev_prefetch_step(const DevTopo& T, const DevPtrs& D, int t, int ts, const float* x) {
  const int Bp = T.Bp, nf = 18 * T.nb, base = blockIdx.x * 32;
  if (threadIdx.x < 32) prefetch_record_l2(T, tape_step(T, D, ts).rec);
  for (int f = threadIdx.x; f < nf; f += blockDim.x) prefetch_l2(x + (size_t)f * Bp + base);
  // the controller's activation rows (its delta rows are written, not read, by the reverse)
  if (T.n_layers == 0 || T.ext_ctrl) return;
  const size_t N = (size_t)T.horizon * Bp;
  const float* d = D.dump + (size_t)t * Bp + base;
  for (int l = 0; l <= T.n_layers; ++l)
    for (int r = threadIdx.x; r < T.widths[l]; r += blockDim.x) prefetch_l2(d + (size_t)(T.dump_act[l] + r) * N);
}

// Reverse of step t from its tape slot ts (every warp calls; ends after a CTA barrier). C.XB holds the
// adjoint of x_{t+1} on entry, that of x_t on exit; x_{t+1} is on chip in C.X (or copied there from
// x_t1 first when load_x1 is set), x_t is read from global memory and left in C.X.
template <class Q>
__device__ __forceinline__ void blk_reverse_step(const DevTopo& T, const DevPtrs& D, const RevCtx& C, int t, int ts,
                                                 const float* x_t, const float* x_t1, bool load_x1, int warp) {
  const int i = C.i, Bp = T.Bp, nf = 18 * T.nb, lane = threadIdx.x & 31;
  const size_t N = (size_t)T.horizon * Bp, n = (size_t)t * Bp + i;
  const uint32_t mine = blk_mine(warp);
  const SL& S = C.S;
  const TapeStep tp = tape_step(T, D, ts);
  const LaneT<SL> L{S, C.P, S, i};
  const BLaneT<SL> Bl{L, C.X, C.G, GC{tp.vminus, 32}};
  rev_stage_first<Q::SEQ>(T, tp);
  if (load_x1)
    for (int f = warp; f < nf; f += blk_nw()) C.X[f] = x_t1[(size_t)f * Bp + i];
  if (T.grad_decay != 1.f) {  // section 3.2: the adjoint from later steps shrinks by alpha per step
    for (int f = warp; f < nf; f += blk_nw()) C.XB[f] *= T.grad_decay;
    if (warp == 0)
      for (int k = 0; k < T.n_rec; ++k) S[T.sm_hb + k] *= T.grad_decay;  // and so does h's
  }
  cta_sync();
  // loss term (by the loss body's warp) and integrator, x_{t+1} on chip
  if ((T.loss_body & (blk_nw() - 1)) == warp) loss_reverse(T, Bl, C.X, C.XB, loss_weight(T, t + 1, D.hz[i]) * C.dl);
  integrate_reverse(T, GL{const_cast<float*>(x_t) + i, Bp}, C.X, C.XB, C.VB, mine);
  // x_t on chip, body by body (no other warp reads a body's x_{t+1}); accumulators zeroed
  for (int b = warp; b < T.nb; b += blk_nw()) {
#pragma unroll
    for (int f = 0; f < 18; ++f) C.X[18 * b + f] = x_t[(size_t)(18 * b + f) * Bp + i];
    S[T.sm_invmb + b] = 0.f;
    constexpr int n9 = Q::SEQ ? 9 : 6;
#pragma unroll
    for (int q = 0; q < n9; ++q) S[T.sm_iinvb + n9 * b + q] = 0.f;
  }
  for (int s = warp; s < T.nslots; s += blk_nw()) S[T.sm_lam + s] = 0.f;  // impulse adjoints
  inverse_inertia(T, L, C.X, mine);
  cta_sync();
  // the step's records, re-formed bit for bit
  hinge_kinematics(T, L, C.X, mine);
  const int u = T.n_layers > 0 ? T.n_layers : 0;
  const GW au = T.ext_ctrl ? GW{D.u_ext + n * T.ext_nop, 1} : GW{D.dump + (size_t)T.dump_act[u] * N + n, N};
  servo_targets(T, L, au, mine);
  blk_assemble<false>(T, S, C.P, C.X, VelTape{GS{tp.vminus}}, nullptr, warp);
  for (int j = warp; j < T.nj; j += blk_nw())
    for (int q = 0; q < (Q::SEQ ? JX_N : JA_N); ++q) joint_rec(T, S, j)[JR_N + q] = 0.f;
  for (int c = warp; c < T.ns; c += blk_nw())
    for (int q = 0; q < (Q::SEQ ? CX_N : CA_N); ++q) contact_rec(T, S, c)[CR_N + q] = 0.f;
  if constexpr (!Q::SEQ)
    for (int c = warp; c < T.np; c += blk_nw())
      for (int q = 0; q < PA_N; ++q) pair_rec(T, S, c)[PR_N + q] = 0.f;
  cta_sync();
  blk_stream(T, warp, true);
  blk_sweeps_rev<Q::SEQ>(T, S, tp, warp);
  const bool ws = T.ws != 0;
  if constexpr (Q::SEQ) {
    // the sweeps' staging buffers lay over x_t
    for (int f = warp; f < nf; f += blk_nw()) C.X[f] = x_t[(size_t)f * Bp + i];
    cta_sync();
    for (int j = warp; j < T.nj; j += blk_nw()) rx_joint_item(T, C, tp, ws, j);
    for (int q = warp; q < T.ns; q += blk_nw()) rx_contact_item(T, C, tp, ws, q);
  } else {
    for (int j = warp; j < T.nj; j += blk_nw()) joint_reverse(T, C, tp, ws, j);
    for (int q = warp; q < T.ns; q += blk_nw()) contact_reverse(T, C, tp, ws, q);
    for (int p = warp; p < T.np; p += blk_nw()) pair_reverse(T, C, tp, ws, p);
  }
  // servo targets: the joint's warp has its adjoint
  const SL zb = S.at(T.sm_zb);
  const int nout = T.n_layers > 0 ? T.widths[T.n_layers] : 0;
  for (int m = 0; m < T.n_motors; ++m) {
    const int j = T.motor_joint[m];
    if ((j & (blk_nw() - 1)) != warp) continue;
    const float g = S[T.sm_wstb + j], br = S[T.sm_wbr + j];
    float ub = 0.f;
    if (br == 0.f) {
      const float k = C.P[T.o_motor + 3 * j];
      const float um = m < nout ? au[m] : 0.f;
      ub = k * g;
      S[T.sm_thb + j] -= k * g;
      C.G.red(T.o_motor + 3 * j, (um - S[T.sm_th + j]) * g);
    } else {
      C.G.red(T.o_motor + 3 * j + 2, (br == 2.f ? 1.f : -1.f) * g);
    }
    if (m < nout) zb[m] = ub;
  }
  if (T.n_layers > 0 && warp == 3) {  // outputs that drive no servo; the recurrent ones: h^{t+1} = tanh(z)
    for (int o = T.n_motors; o < nout; ++o) zb[o] = 0.f;
    const int base = nout - T.n_rec;
    for (int k = 0; k < T.n_rec; ++k) {
      const float th = tanhf(au[base + k]);
      zb[base + k] = S[T.sm_hb + k] * (1.f - th * th);
    }
  }
  cta_sync();
  if constexpr (Q::SEQ) {
    for (int b = warp; b < T.nb; b += blk_nw()) rx_body(T, C, ws, b);
    external_reverse(T, Bl, C.XB, C.VB, mine);
  } else {
    for (int b = warp; b < T.nb; b += blk_nw()) body_reverse(T, C, b);
    if (T.np)
      for (int q = warp; q < T.ns; q += blk_nw()) sphere_reverse(T, C, q);
  }
  if (T.ext_ctrl) {
    // wide controller: the output adjoint goes to the batched products; the features' adjoint comes
    // back into the next launch
    float* ubx = D.ub_ext + (size_t)i * 16;
    for (int o = warp; o < 16; o += blk_nw()) {
      ubx[o] = o < nout ? zb[o] : 0.f;
      if (o < nout) D.dump[(size_t)(T.dump_del[T.n_layers - 1] + o) * N + n] = zb[o];  // output layer's delta
    }
    cta_sync();
  } else if (T.n_layers > 0) {
    GW act[DPK_MAXL + 1], del[DPK_MAXL + 1];
    for (int l = 0; l <= DPK_MAXL; ++l) {
      act[l] = GW{D.dump + (size_t)T.dump_act[l] * N + n, N};
      del[l] = GW{D.dump + (size_t)T.dump_del[l] * N + n, N};
    }
    for (int o = warp; o < nout; o += blk_nw()) del[T.n_layers - 1][o] = zb[o];
    cta_sync();  // the packages have been read: the controller's buffers may overwrite them
    const SL sbar = S.at(T.sm_sbar);
    if (T.mlp_tc) {
      ctrl_backward_blk<Q>(T, D, zb, sbar, D.dump + (n - lane), warp);
    } else {
      int maxw = 1;
      for (int l = 0; l <= T.n_layers; ++l) maxw = max(maxw, T.widths[l]);
      const SL z1 = S.at(T.sm_hbuf), z2 = S.at(T.sm_hbuf + maxw);
      for (int o = warp; o < nout; o += blk_nw()) z1[o] = zb[o];
      cta_sync();
      controller_reverse_nw(T, D, act, del, z1, z2, sbar, warp);
    }
    cta_sync();
    features_reverse_joints(T, S, sbar, warp);
    if (warp == 3) {
      features_reverse_rest(T, C, sbar);
      const int base = T.widths[0] - T.n_rec;
      for (int k = 0; k < T.n_rec; ++k) S[T.sm_hb + k] = sbar[base + k];  // adjoint of h^t
    }
  } else {
    cta_sync();
  }
  blk_hinge_reverse<Q>(T, C, warp);
}

__device__ __forceinline__ void blk_loss_initial_reverse(const DevTopo& T, const DevPtrs& D, const RevCtx& C) {
  const int b = T.loss_body;
  for (int f = 18 * b; f < 18 * b + 18; ++f) C.X[f] = D.ckpt[(size_t)f * T.Bp + C.i];
  const M3 R = loadR(C.X, 18 * b);
  const float3 c = C.P.v3(T.o_loss_point), a = C.P.v3(T.o_loss_target);
  const float3 gq = -C.dl * a;
  C.XB.a3(18 * b, gq);
  add_outer(C.XB, 18 * b + 3, gq, c);
  C.G.red3(T.o_loss_point, mtv(R, gq));
  C.G.red3(T.o_loss_target, -C.dl * (C.X.v3(18 * b) + mv(R, c)));
}
__device__ __forceinline__ RevCtx rev_ctx(const DevTopo& T, const DevPtrs& D, float* sm, int i) {
  return RevCtx{SL{sm}, SL{sm + T.sm_x * 32}, SL{sm + T.sm_xb * 32}, SL{sm + T.sm_vb * 32}, GC{D.prm + i, T.Bp},
                GL{D.grad_prm + i, T.Bp}, i, D.dloss[i]};
}

// Reverse mode through the last rollout, whole tape: every step from it, last first.
template <class Q>
__global__ void __launch_bounds__(32 * Q::NW, 1) k_backward_blk(const __grid_constant__ DevTopo T, const __grid_constant__ DevPtrs D) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane, Bp = T.Bp, nf = 18 * T.nb;
  const RevCtx C = rev_ctx(T, D, g_smem + lane, i);
  blk_load(T, D);
  for (int f = warp; f < nf; f += blk_nw()) C.XB[f] = 0.f;
  if (warp == 0)
    for (int k = 0; k < T.n_rec; ++k) C.S[T.sm_hb + k] = 0.f;  // no adjoint reaches h^T
  const size_t sb = (size_t)nf * Bp;
  const int Tw = warp_horizon(D, i);  // the rollout stepped this group to Tw
  for (int t = Tw - 1; t >= 0; --t) {
    if (t > 0) rev_prefetch_step(T, D, t - 1, t - 1, D.ckpt + (size_t)(t - 1) * sb);
    // x_{t+1} is on chip from the step reversed before, except for the first one
    blk_reverse_step<Q>(T, D, C, t, t, D.ckpt + (size_t)t * sb, D.state, t == Tw - 1, warp);
  }
  if (T.loss_kind == 3) {
    if (warp == 0) blk_loss_initial_reverse(T, D, C);
    cta_sync();
  }
  for (int f = warp; f < nf; f += blk_nw()) D.grad_state0[(size_t)f * Bp + i] = C.XB[f];
}

// Reverse mode from checkpoints: each segment (last first) is stepped again with its tape (layout Tf),
// then reversed (layout T). The state adjoint and that of h lie in front of both layouts.
template <class Q>
__global__ void __launch_bounds__(32 * Q::NW, 1) k_backward_seg_blk(const __grid_constant__ DevTopo T, const __grid_constant__ DevTopo Tf,
                                                             const __grid_constant__ DevPtrs D) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane, Bp = T.Bp, nf = 18 * T.nb;
  float* sm = g_smem + lane;
  const RevCtx C = rev_ctx(T, D, sm, i);
  const LaneT<SL> L{SL{sm}, GC{D.prm + i, Bp}, SL{sm}, i};
  const SL X{sm + Tf.sm_x * 32};
  SL act[DPK_MAXL + 1];
  for (int l = 0; l <= DPK_MAXL; ++l) act[l] = SL{sm + Tf.sm_act[l] * 32};
  for (int f = warp; f < nf; f += blk_nw()) C.XB[f] = 0.f;
  if (warp == 0)
    for (int k = 0; k < T.n_rec; ++k) C.S[T.sm_hb + k] = 0.f;  // no adjoint reaches h^T
  const size_t sb = (size_t)nf * Bp;
  const int Tw = warp_horizon(D, i), K = D.ckpt_every;
  for (int c = (Tw - 1) / K; c >= 0; --c) {
    const int ta = c * K, tb = min(Tw, ta + K);
    cta_sync();  // the layouts share their memory
    blk_load(Tf, D);
    for (int f = warp; f < nf; f += blk_nw()) X[f] = D.ckpt[(size_t)c * sb + (size_t)f * Bp + i];
    if (T.ws)  // the previous impulses the segment's first step started from
      for (int s = warp; s < T.nslots; s += blk_nw()) L.S[Tf.sm_lam + s] = D.ckpt_lam[((size_t)c * T.nslots + s) * Bp + i];
    if (warp == 0)
      for (int k = 0; k < T.n_rec; ++k)  // the controller's recurrent state at the segment's start
        L.S[Tf.sm_h + k] = D.ckpt_h[((size_t)c * T.n_rec + k) * Bp + i];
    cta_sync();
    for (int t = ta; t < tb; ++t) {
      for (int f = warp; f < nf; f += blk_nw()) D.seg[(size_t)(t - ta) * sb + (size_t)f * Bp + i] = X[f];
      blk_step<true, Q>(Tf, D, L, X, act, t, t - ta, nullptr, T.n_layers > 0 ? D.dump + (size_t)t * Bp + i : nullptr, warp);
    }
    for (int f = warp; f < nf; f += blk_nw()) D.seg[(size_t)(tb - ta) * sb + (size_t)f * Bp + i] = X[f];
    __threadfence();  // the reverse reads the tape through L2
    cta_sync();
    blk_load(T, D);
    cta_sync();
    for (int t = tb - 1; t >= ta; --t)
      blk_reverse_step<Q>(T, D, C, t, t - ta, D.seg + (size_t)(t - ta) * sb, D.seg + (size_t)(t - ta + 1) * sb, t == tb - 1,
                          warp);
  }
  if (T.loss_kind == 3) {
    if (warp == 0) blk_loss_initial_reverse(T, D, C);
    cta_sync();
  }
  for (int f = warp; f < nf; f += blk_nw()) D.grad_state0[(size_t)f * Bp + i] = C.XB[f];
}

// The wide controller's per-step reverse launches (see k_backward_ext in dp_steps.cuh): the feature
// adjoint of x_{t+1}, then the reverse of step t.
template <class Q>
__global__ void __launch_bounds__(32 * Q::NW, 1) k_backward_ext_blk(const __grid_constant__ DevTopo T, const __grid_constant__ DevPtrs D,
                                                             int t) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane, Bp = T.Bp, nf = 18 * T.nb;
  const RevCtx C = rev_ctx(T, D, g_smem + lane, i);
  const int Tw = warp_horizon(D, i);  // the same for the CTA's warps
  if (t >= Tw) return;                // this group's rollout ended before step t
  blk_load(T, D);
  const size_t sb = (size_t)nf * Bp;
  const uint32_t mine = blk_mine(warp);
  for (int f = warp; f < nf; f += blk_nw()) C.XB[f] = D.grad_state0[(size_t)f * Bp + i];
  const int tn = t + 1;
  if (t > 0) rev_prefetch_step(T, D, t, t, D.ckpt + (size_t)t * sb);
  if (tn < Tw) {  // adjoint of the features of x_{t+1}
    const float* xs = D.ckpt + (size_t)tn * sb;
    for (int f = warp; f < nf; f += blk_nw()) C.X[f] = xs[(size_t)f * Bp + i];
    cta_sync();
    const LaneT<SL> L{C.S, C.P, C.S, i};
    hinge_kinematics(T, L, C.X, mine);
    for (int j = warp; j < T.nj; j += blk_nw()) {
      C.S[T.sm_thb + j] = C.S[T.sm_thdb + j] = 0.f;
      C.S.s3(T.sm_uab + 3 * j, f3(0.f, 0.f, 0.f));
    }
    const GC sbar{D.sbar_ext + (size_t)i * T.ext_k0p, 1};
    features_reverse_joints(T, C.S, sbar, warp);
    if (warp == 3) features_reverse_rest(T, C, sbar);
    blk_hinge_reverse<Q>(T, C, warp);
  }
  if (t >= 0) {
    blk_reverse_step<Q>(T, D, C, t, t, D.ckpt + (size_t)t * sb, D.state, tn >= Tw, warp);
  } else {
    if (warp == 0 && T.loss_kind == 3) blk_loss_initial_reverse(T, D, C);
    cta_sync();
  }
  for (int f = warp; f < nf; f += blk_nw()) D.grad_state0[(size_t)f * Bp + i] = C.XB[f];
}

template <class Q>
static cudaError_t launch_backward_blk_t(const DevTopo& T, const DevTopo& Ts, const DevPtrs& D, cudaStream_t s) {
  cudaError_t e;
  if (D.tape_full) {
    const size_t smem = (size_t)T.sm_total * 128;
    e = cudaFuncSetAttribute(k_backward_blk<Q>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_backward_blk<Q><<<T.Bp / 32, 32 * T.blk_nw, smem, s>>>(T, D);
  } else {
    const size_t smem = (size_t)(T.sm_total > Ts.sm_total ? T.sm_total : Ts.sm_total) * 128;
    e = cudaFuncSetAttribute(k_backward_seg_blk<Q>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_backward_seg_blk<Q><<<T.Bp / 32, 32 * T.blk_nw, smem, s>>>(T, Ts, D);
  }
  return cudaGetLastError();
}
template <class Q>
static cudaError_t launch_backward_ext_blk_t(const DevTopo& T, const DevPtrs& D, int t, cudaStream_t s) {
  const size_t smem = (size_t)T.sm_total * 128;
  cudaError_t e = cudaFuncSetAttribute(k_backward_ext_blk<Q>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_backward_ext_blk<Q><<<T.Bp / 32, 32 * T.blk_nw, smem, s>>>(T, D, t);
  return cudaGetLastError();
}
