// One step of the engine on the warps of a CTA that share a group of 32 instances (a lane is an instance
// in every warp; eight warps for the compiled topologies, four else: plan_blocks), for any robot whose constraint rows fit on chip.
//
// The work of a step is cut into items: joints (the up to seven rows of one hinge or ball joint)
// and contacts (the three rows of one sphere). Outside the solver, item k (joints,
// contacts and pairs each counted from 0) belongs to warp k % blk_nw() and body b to warp b % blk_nw(); every quantity of an item (its lever arms, axes, effective masses) is
// formed once and kept in a compact record, from which the Jacobian of each row is a sign and a
// permutation. In the solver the rows of one item that are adjacent in the sweep order of both of
// its bodies form a block; the host schedules the blocks into levels of independent ones
// (plan_blocks in dp_plan.cu), a warp loads the two bodies' velocities from shared memory, runs
// the block's rows in registers and stores them back, and the warps meet at one CTA barrier per
// level that has a live block. Every body sees its rows in the order (colour, slot) of the sequential
// sweep. The compiled topologies' rollouts are its rollouts bit for bit; a row of another robot may be
// rounded otherwise in a last place.
//
// Why: one warp running the whole sweep (unrolled over the slots, velocities in registers) spent
// about 125 cycles per row update on one scheduler of four, with a straight-line body of some 70 KB
// of instructions per sweep that no instruction cache near the scheduler holds. The blocks share
// one small body of code, use the four schedulers, and leave the chain of the rows on the body
// with the most joints as the longest path.
#pragma once
#include "dp_adjoint.cuh"

extern __shared__ float g_smem[];

// CTA barrier 1 over all warps (each warp arrives from its own code path).
__device__ __forceinline__ void cta_sync() { asm volatile("bar.sync 1;" ::: "memory"); }
// Warps of the CTA (DevTopo.blk_nw), and the joints and bodies k of warp w (k % warps == w) as a mask.
__device__ __forceinline__ int blk_nw() { return blockDim.x >> 5; }
__device__ __forceinline__ uint32_t blk_mine(int warp) { return (blk_nw() == 8 ? 0x01010101u : 0x11111111u) << warp; }

// Compact records in shared memory ([field][32 lanes], DevTopo.sm_rows; stride rec_j, rec_c, rec_p),
// one per joint, contact sphere and sphere pair. The rollout keeps I^-1 J_w behind the first JR_N
// (CR_N, PR_N) fields; the reverse pass recomputes it in registers and has its accumulators there.
enum {
  JF_RA = 0,    // 3: lever arm on the parent (row k of the linear rows: J_wa = ra x e_k)
  JF_RB = 3,    // 3: lever arm on the child  (J_wb = -(rb x e_k))
  JF_T = 6,     // 6: the two angular directions t (J_wa = t, J_wb = -t)
  JF_ME = 12,   // 7: effective masses (3 linear, 2 angular, limit, servo; 0: inactive)
  JF_BI = 19,   // 7: biases
  JF_BND = 26,  // servo impulse bound
  JF_LS = 27,   // limit row's sign s: +1 at the lower bound, -1 at the upper
  JR_N = 28,
  JF_IAL = 28,  // 9: I_a^-1 J_wa of the linear rows (zero when the parent is the world)
  JF_IBL = 37,  // 9
  JF_IAT = 46,  // 6: of the angular rows
  JF_IBT = 52,  // 6
  JF_IAU = 58,  // 3: I_a^-1 u_a (limit and servo rows: J_wa = -s u_a, J_wb = s u_a)
  JF_IBU = 61,  // 3
  JF_N = 64
};
enum {
  CF_RA = 0,  // 3: lever arm (J_wa = ra x n, n = z, x, y)
  CF_ME = 3,  // 3
  CF_BI = 6,  // normal row's bias
  CF_MU = 7,
  CR_N = 8,
  CF_I = 8,   // 9: I^-1 J_wa of the normal, first and second friction row
  CF_N = 17
};
enum {
  PF_LIN = 0,   // 9: normal, t1, t2
  PF_ANGA = 9,  // 9
  PF_ANGB = 18, // 9
  PF_ME = 27,   // 3
  PF_BI = 30,
  PF_MU = 31,
  PR_N = 32,
  PF_IA = 32,   // 9
  PF_IB = 41,   // 9
  PF_N = 50
};
// Solver blocks (int4 descriptors of the program).
enum { BT_JOINT = 0, BT_LIMIT = 1, BT_MOTOR = 2, BT_GROUND = 3, BT_PAIR = 4 };
struct BlkOp {
  int4 v;
  __device__ __forceinline__ int type() const { return v.x & 0xff; }
  __device__ __forceinline__ int mask() const { return (v.x >> 8) & 0xff; }
  __device__ __forceinline__ int a() const { return (v.w & 0xff) - 1; }
  __device__ __forceinline__ int b() const { return ((v.w >> 8) & 0xff) - 1; }
  __device__ __forceinline__ int idx() const { return v.w >> 16; }      // joint, sphere or pair
  __device__ __forceinline__ int slot() const { return v.z & 0xffff; }  // slot of the item's first row
  __device__ __forceinline__ int live() const { return v.z >> 16; }     // live-flag index, -1: always live
};
// Stream entries (one byte): bit 7 a CTA barrier follows, bit 6 there is a block, low 6 bits it.
#define BS_BAR 0x80
#define BS_OP 0x40

__device__ __forceinline__ uint8_t* blk_bytes(const DevTopo& T) {
  return reinterpret_cast<uint8_t*>(g_smem + T.sm_prog * 32);
}
__device__ __forceinline__ uint8_t* blk_live(const DevTopo& T) { return blk_bytes(T) + T.blk_live; }
__device__ __forceinline__ BlkOp blk_op(const DevTopo& T, int k) {
  return BlkOp{reinterpret_cast<const int4*>(blk_bytes(T))[k]};
}
__device__ __forceinline__ SL joint_rec(const DevTopo& T, const SL& S, int j) { return S.at(T.sm_rows + T.rec_j * j); }
__device__ __forceinline__ SL contact_rec(const DevTopo& T, const SL& S, int q) {
  return S.at(T.sm_rows + T.rec_j * T.nj + T.rec_c * q);
}
__device__ __forceinline__ SL pair_rec(const DevTopo& T, const SL& S, int p) {
  return S.at(T.sm_rows + T.rec_j * T.nj + T.rec_c * T.ns + T.rec_p * p);
}
// Body velocities after the external impulses: on chip in the rollout, from the tape in reverse.
struct VelX {
  SL X;
  __device__ __forceinline__ float3 v(int b) const { return X.v3(18 * b + 12); }
  __device__ __forceinline__ float3 w(int b) const { return X.v3(18 * b + 15); }
};
struct VelTape {
  GS p;
  __device__ __forceinline__ float3 v(int b) const { return p.v3(6 * b); }
  __device__ __forceinline__ float3 w(int b) const { return p.v3(6 * b + 3); }
};

// The program into shared memory (once per launch, before the first barrier of the kernel).
__device__ __forceinline__ void blk_load(const DevTopo& T, const DevPtrs& D) {
  int* dst = reinterpret_cast<int*>(blk_bytes(T));
  for (int k = threadIdx.x; k < T.blk_words; k += blockDim.x) dst[k] = D.blk[k];
}

// This warp's stream of the step: the live blocks of each level in order, a barrier after every
// level that has a live block on some warp, and a zero at the end. Lane l handles level l; the
// streams of all warps hold the same number of barriers, so they cannot deadlock. reverse: the
// levels and the blocks of a level last first (the reverse sweeps).
__device__ __forceinline__ void blk_stream(const DevTopo& T, int warp, bool reverse = false) {
  const int lane = threadIdx.x & 31;
  const uint8_t* base = blk_bytes(T);
  const uint8_t* live = blk_live(T);
  unsigned lo = 0u, hi = 0u;  // live blocks
  {
    bool a = false;
    if (lane < T.blk_nops) { const int f = blk_op(T, lane).live(); a = f < 0 || live[f]; }
    lo = __ballot_sync(FULLMASK, a);
    if (T.blk_nops > 32) {
      a = false;
      if (32 + lane < T.blk_nops) { const int f = blk_op(T, 32 + lane).live(); a = f < 0 || live[f]; }
      hi = __ballot_sync(FULLMASK, a);
    }
  }
  const unsigned long long alive = ((unsigned long long)hi << 32) | lo;
  const int nl = T.blk_nlev;
  unsigned long long mine = 0ull;
  bool any = false;
  if (lane < nl) {
    const int level = reverse ? nl - 1 - lane : lane;
    for (int w = 0; w < blk_nw(); ++w) {
      const uint8_t* f = base + T.blk_lev + w * (nl + 1) + level;
      const unsigned long long m = ((1ull << f[1]) - 1ull) & ~((1ull << f[0]) - 1ull) & alive;
      any |= m != 0ull;
      if (w == warp) mine = m;
    }
  }
  // a level without a block of this warp still takes one entry, for its barrier
  const int n = any ? max(1, __popcll(mine)) : 0;
  int pos = n;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(FULLMASK, pos, o);
    if (lane >= o) pos += y;
  }
  const int total = __shfl_sync(FULLMASK, pos, 31);
  uint8_t* st = blk_bytes(T) + T.blk_stream + warp * T.blk_stream_len;
  int k = pos - n;
  const uint8_t bar = T.blk_single ? 0 : BS_BAR;
  if (any && mine == 0ull) st[k] = bar;
  while (mine) {
    const int o = reverse ? 63 - __clzll((long long)mine) : __ffsll((long long)mine) - 1;
    mine &= ~(1ull << o);
    st[k++] = (uint8_t)(BS_OP | o | (mine ? 0 : bar));
  }
  if (lane == 0) st[total] = 0;
  __syncwarp();
}

// ------------------------------------------------------------------------------ assembly
// v x e_k for a coordinate axis: the products with the axis' zeros are exact zeros.
template <int K>
__device__ __forceinline__ float3 cross_axis(float3 v) {
  if (K == 0) return f3(0.f, v.z, -v.y);
  if (K == 1) return f3(-v.z, 0.f, v.x);
  return f3(v.y, -v.x, 0.f);
}
// Products with an explicit order of rounding (the sums of dot3 and symv as the compiler fuses them
// for operands it knows nothing about; signs and zeros that it can see here would change the order).
__device__ __forceinline__ float dotx(float3 a, float3 b) {
  return fmaf(a.z, b.z, fmaf(a.x, b.x, __fmul_rn(a.y, b.y)));
}
__device__ __forceinline__ float3 symx(const float* s, float3 v) {
  return f3(fmaf(s[2], v.z, fmaf(s[0], v.x, __fmul_rn(s[1], v.y))),
            fmaf(s[4], v.z, fmaf(s[1], v.x, __fmul_rn(s[3], v.y))),
            fmaf(s[5], v.z, fmaf(s[4], v.y, __fmul_rn(s[2], v.x))));
}
__device__ __forceinline__ float3 axpy3(float s, float3 x, float3 y) {
  return f3(fmaf(s, x.x, y.x), fmaf(s, x.y, y.y), fmaf(s, x.z, y.z));
}
__device__ __forceinline__ void load6(const SL& S, int f, float (&o)[6]) {
#pragma unroll
  for (int q = 0; q < 6; ++q) o[q] = S[f + q];
}

// Record of joint j (hinge kinematics, servo target and world inverse inertias are on chip).
template <bool INV, class G>
__device__ __forceinline__ void joint_assemble(const DevTopo& T, const SL& S, const G& P, const SL& X, int j, uint8_t* ao) {
  const float bh = T.beta / T.dt;
  const int a = T.ja[j], b = T.jb[j], fl = T.jflags[j], s0 = T.jslot[j];
  const SL R = joint_rec(T, S, j);
  const M3 Rb = loadR(X, 18 * b);
  const M3 Ra = body_R(X, a);
  const float3 ra = a >= 0 ? mv(Ra, P.v3(T.o_anchor + 6 * j)) : P.v3(T.o_anchor + 6 * j);
  const float3 rb = mv(Rb, P.v3(T.o_anchor + 6 * j + 3));
  const float3 C = (body_p(X, a) + ra) - (X.v3(18 * b) + rb);
  float ia[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, ib[6];
  float ima = 0.f;
  if (a >= 0) { load6(S, T.sm_iinv + 6 * a, ia); ima = S[T.sm_invm + a]; }
  load6(S, T.sm_iinv + 6 * b, ib);
  const float imb = S[T.sm_invm + b];
  R.s3(JF_RA, ra);
  R.s3(JF_RB, rb);
  auto lin = [&](auto KI, float c) {
    constexpr int k = decltype(KI)::value;
    const float3 angA = cross_axis<k>(ra), angB = -cross_axis<k>(rb);
    float K = 0.f;
    float3 IA = f3(0.f, 0.f, 0.f);
    if (a >= 0) { IA = symx(ia, angA); K += ima + dotx(angA, IA); }
    const float3 IB = symx(ib, angB);
    K += imb + dotx(angB, IB);
    if (INV) { R.s3(JF_IAL + 3 * k, IA); R.s3(JF_IBL + 3 * k, IB); }
    R[JF_ME + k] = 1.f / (K + T.gamma);
    R[JF_BI + k] = bh * c;
  };
  lin(std::integral_constant<int, 0>{}, C.x);
  lin(std::integral_constant<int, 1>{}, C.y);
  lin(std::integral_constant<int, 2>{}, C.z);
  if (T.jtype[j] == 1) {
    float3 tau[2];
    onb3(P.v3(T.o_axis + 6 * j), tau[0], tau[1]);
    const float3 ub = mv(Rb, P.v3(T.o_axis + 6 * j + 3));
    const float3 ua = S.v3(T.sm_ua + 3 * j);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const float3 t = mv(Ra, tau[k]);
      float K = 0.f;
      float3 IA = f3(0.f, 0.f, 0.f);
      if (a >= 0) { IA = symx(ia, t); K += dotx(t, IA); }
      const float3 IB = symx(ib, -t);
      K += dotx(-t, IB);
      R.s3(JF_T + 3 * k, t);
      if (INV) { R.s3(JF_IAT + 3 * k, IA); R.s3(JF_IBT + 3 * k, IB); }
      R[JF_ME + 3 + k] = 1.f / (K + T.gamma);
      R[JF_BI + 3 + k] = bh * dot3(t, cross3(ub, ua));
    }
    if (fl) {
      float K = 0.f;
      float3 IA = f3(0.f, 0.f, 0.f);
      if (a >= 0) { IA = symx(ia, ua); K += dotx(ua, IA); }
      const float3 IB = symx(ib, ua);
      K += dotx(ua, IB);
      const float me = 1.f / (K + T.gamma);
      if (INV) { R.s3(JF_IAU, IA); R.s3(JF_IBU, IB); }
      if (fl & 1) {
        const float th = S[T.sm_th + j];
        const float lo = P[T.o_limit + 2 * j], hi = P[T.o_limit + 2 * j + 1];
        const bool low = th <= lo, high = !low && th >= hi, on = low || high;
        R[JF_ME + 5] = on ? me : 0.f;
        R[JF_BI + 5] = low ? bh * (th - lo) : (high ? bh * (hi - th) : 0.f);
        R[JF_LS] = low ? 1.f : -1.f;
        if (ao) ao[T.jlim[j]] = on ? 1 : 0;
        const bool any = __any_sync(FULLMASK, on && me != 0.f);
        if ((threadIdx.x & 31) == 0) blk_live(T)[j] = any ? 1 : 0;
      }
      if (fl & 2) {
        R[JF_ME + 6] = me;
        R[JF_BI + 6] = -S[T.sm_wst + j];
        R[JF_BND] = P[T.o_motor + 3 * j + 1] * T.dt;
        if (ao) ao[T.jmot[j]] = 1;
      }
    }
  }
  if (ao)
    for (int k = 0; k < (T.jtype[j] == 1 ? 5 : 3); ++k) ao[s0 + k] = 1;
}

// Record of ground contact q.
template <bool INV, class G, class VV>
__device__ __forceinline__ void contact_assemble(const DevTopo& T, const SL& S, const G& P, const SL& X, const VV& V,
                                                 int q, uint8_t* ao) {
  const float bh = T.beta / T.dt;
  const int a = T.sbody[q], s0 = T.cslot + 3 * q;
  const SL R = contact_rec(T, S, q);
  const float3 c = mv(loadR(X, 18 * a), P.v3(T.o_sph_off + 3 * q));
  const float rad = P[T.o_sph_rad + q];
  const float d = (X[18 * a + 2] + c.z) - rad - T.ground_z;
  const bool on = d <= 0.f;
  const bool any = __any_sync(FULLMASK, on);
  if ((threadIdx.x & 31) == 0) blk_live(T)[T.nj + q] = any ? 1 : 0;
  if (ao) ao[s0] = ao[s0 + 1] = ao[s0 + 2] = on ? 1 : 0;
  const float3 ra = f3(c.x, c.y, c.z - rad);
  float ia[6];
  load6(S, T.sm_iinv + 6 * a, ia);
  const float ima = S[T.sm_invm + a];
  const float3 an = cross_axis<2>(ra);
  const float vn = V.v(a).z + dotx(an, V.w(a));
  const float bias = bh * min0f(d + T.slop) + P[T.o_sph_e + q] * min0f(vn);
  R.s3(CF_RA, ra);
  auto row = [&](int k, float3 ang) {
    const float3 IA = symx(ia, ang);
    float K = 0.f;
    K += ima + dotx(ang, IA);
    if (INV) R.s3(CF_I + 3 * k, IA);
    R[CF_ME + k] = on ? 1.f / (K + T.gamma) : 0.f;
  };
  row(0, an);
  row(1, cross_axis<0>(ra));
  row(2, cross_axis<1>(ra));
  R[CF_BI] = on ? bias : 0.f;
  R[CF_MU] = P[T.o_sph_mu + q];
}

// Record of sphere pair p.
template <bool INV, class G, class VV>
__device__ __forceinline__ void pair_assemble(const DevTopo& T, const SL& S, const G& P, const SL& X, const VV& V,
                                                 int p, uint8_t* ao) {
  const float bh = T.beta / T.dt;
  const int k = T.pk[p], l = T.pl[p], a = T.sbody[k], b = T.sbody[l], s0 = T.cslot + 3 * (T.ns + p);
  const SL R = pair_rec(T, S, p);
  const float3 ck = mv(loadR(X, 18 * a), P.v3(T.o_sph_off + 3 * k));
  const float3 cl = mv(loadR(X, 18 * b), P.v3(T.o_sph_off + 3 * l));
  const float3 dl = (X.v3(18 * a) + ck) - (X.v3(18 * b) + cl);
  const float dist = sqrtf(dot3(dl, dl));
  const float3 n = dist > 1e-9f ? (1.f / dist) * dl : f3(0.f, 0.f, 1.f);
  const float rk = P[T.o_sph_rad + k], rl = P[T.o_sph_rad + l];
  const float d = dist - rk - rl;
  const bool on = d <= 0.f;
  const bool any = __any_sync(FULLMASK, on);
  if ((threadIdx.x & 31) == 0) blk_live(T)[T.nj + T.ns + p] = any ? 1 : 0;
  if (ao) ao[s0] = ao[s0 + 1] = ao[s0 + 2] = on ? 1 : 0;
  const float3 ra = ck - rk * n, rb = cl + rl * n;
  float3 t1, t2;
  onb3(n, t1, t2);
  float ia[6], ib[6];
  load6(S, T.sm_iinv + 6 * a, ia);
  load6(S, T.sm_iinv + 6 * b, ib);
  const float ima = S[T.sm_invm + a], imb = S[T.sm_invm + b];
  float bias = 0.f;
  auto row = [&](int r, float3 lin) {
    const float3 angA = cross3(ra, lin), angB = -cross3(rb, lin);
    if (r == 0) {
      const float vn = dot3(n, V.v(a) - V.v(b)) + dot3(angA, V.w(a)) + dot3(angB, V.w(b));
      const float ek = P[T.o_sph_e + k], el = P[T.o_sph_e + l];
      const float e = ek >= el ? ek : el;
      bias = bh * min0f(d + T.slop) + e * min0f(vn);
    }
    const float3 IA = symx(ia, angA), IB = symx(ib, angB);
    float K = 0.f;
    K += ima * dot3(lin, lin) + dotx(angA, IA);
    K += imb * dot3(lin, lin) + dotx(angB, IB);
    R.s3(PF_LIN + 3 * r, lin);
    R.s3(PF_ANGA + 3 * r, angA);
    R.s3(PF_ANGB + 3 * r, angB);
    if (INV) { R.s3(PF_IA + 3 * r, IA); R.s3(PF_IB + 3 * r, IB); }
    R[PF_ME + r] = on ? 1.f / (K + T.gamma) : 0.f;
  };
  row(0, n);
  row(1, t1);
  row(2, t2);
  R[PF_BI] = on ? bias : 0.f;
  R[PF_MU] = sqrtf(P[T.o_sph_mu + k] * P[T.o_sph_mu + l]);
}

// Every record, item k by warp k % blk_nw() (V: velocities after the external impulses; ao: the step's
// activity flags of this instance, or NULL; INV: with the I^-1 J_w fields).
template <bool INV, class G, class VV>
__device__ __forceinline__ void blk_assemble(const DevTopo& T, const SL& S, const G& P, const SL& X, const VV& V, uint8_t* ao,
                                             int warp) {
  for (int j = warp; j < T.nj; j += blk_nw()) joint_assemble<INV>(T, S, P, X, j, ao);
  for (int q = warp; q < T.ns; q += blk_nw()) contact_assemble<INV>(T, S, P, X, V, q, ao);
  for (int p = warp; p < T.np; p += blk_nw()) pair_assemble<INV>(T, S, P, X, V, p, ao);
}

// One row in full (the stages that walk slots: the learned warm start, the residual).
struct RowRec {
  float3 lin, angA, angB, IA, IB;
  float meff, bias, bnd;
};
static __device__ __noinline__ RowRec blk_row(const DevTopo& T, const SL S, int s) {
  const int kind = T.skind[s], idx = T.sidx[s], sub = T.ssub[s], a = T.sa[s];
  const float3 z = f3(0.f, 0.f, 0.f);
  RowRec r{z, z, z, z, z, 0.f, 0.f, 0.f};
  if (kind <= RK_MOTOR) {
    const SL R = joint_rec(T, S, idx);
    int m;
    if (kind == RK_JLIN) {
      m = sub;
      const float3 ra = R.v3(JF_RA), rb = R.v3(JF_RB);
      r.lin = f3(sub == 0 ? 1.f : 0.f, sub == 1 ? 1.f : 0.f, sub == 2 ? 1.f : 0.f);
      r.angA = sub == 0 ? cross_axis<0>(ra) : (sub == 1 ? cross_axis<1>(ra) : cross_axis<2>(ra));
      r.angB = -(sub == 0 ? cross_axis<0>(rb) : (sub == 1 ? cross_axis<1>(rb) : cross_axis<2>(rb)));
      r.IA = R.v3(JF_IAL + 3 * sub);
      r.IB = R.v3(JF_IBL + 3 * sub);
    } else if (kind == RK_JANG) {
      m = 3 + sub;
      r.angA = R.v3(JF_T + 3 * sub);
      r.angB = -r.angA;
      r.IA = R.v3(JF_IAT + 3 * sub);
      r.IB = R.v3(JF_IBT + 3 * sub);
    } else {
      m = kind == RK_LIMIT ? 5 : 6;
      const float sg = kind == RK_LIMIT ? R[JF_LS] : 1.f;
      r.angB = sg * S.v3(T.sm_ua + 3 * idx);
      r.angA = -r.angB;
      r.IA = -(sg * R.v3(JF_IAU));
      r.IB = sg * R.v3(JF_IBU);
      if (kind == RK_MOTOR) r.bnd = R[JF_BND];
    }
    if (a < 0) r.angA = z;
    r.meff = R[JF_ME + m];
    r.bias = R[JF_BI + m];
  } else if (kind <= RK_GT) {
    const SL R = contact_rec(T, S, idx);
    const float3 ra = R.v3(CF_RA);
    const int m = kind == RK_GN ? 0 : 1 + sub;
    r.lin = m == 0 ? f3(0.f, 0.f, 1.f) : (m == 1 ? f3(1.f, 0.f, 0.f) : f3(0.f, 1.f, 0.f));
    r.angA = m == 0 ? cross_axis<2>(ra) : (m == 1 ? cross_axis<0>(ra) : cross_axis<1>(ra));
    r.IA = R.v3(CF_I + 3 * m);
    r.meff = R[CF_ME + m];
    if (m == 0) r.bias = R[CF_BI];
    else r.bnd = R[CF_MU];
  } else {
    const SL R = pair_rec(T, S, idx);
    const int m = kind == RK_PN ? 0 : 1 + sub;
    r.lin = R.v3(PF_LIN + 3 * m);
    r.angA = R.v3(PF_ANGA + 3 * m);
    r.angB = R.v3(PF_ANGB + 3 * m);
    r.IA = R.v3(PF_IA + 3 * m);
    r.IB = R.v3(PF_IB + 3 * m);
    r.meff = R[PF_ME + m];
    if (m == 0) r.bias = R[PF_BI];
    else r.bnd = R[PF_MU];
  }
  return r;
}

// ------------------------------------------------------------------------------ forward sweeps
// One projected row update: lam becomes the new impulse, br its clamp branch (0 inside, 1 lower
// bound, 2 upper bound); returns the change. A row without bounds (EQ) never clamps.
template <bool EQ>
__device__ __forceinline__ float row_solve(const DevTopo& T, float Jv, float meff, float bias, float lo, float hi, float& lam,
                                           int& br) {
  const float l0 = lam;
  const float pre = fmaf(-meff, fmaf(T.gamma, l0, __fadd_rn(Jv, bias)), l0);
  br = EQ ? 0 : (pre < lo ? 1 : (pre > hi ? 2 : 0));
  lam = br == 1 ? lo : (br == 2 ? hi : pre);
  return lam - l0;
}
// A row's new impulse on chip and, with TAPE, to the tape with its clamp branch (only the one-warp
// reverse reads the branch of a row without bounds).
template <bool TAPE, bool EQ>
__device__ __forceinline__ void row_store(const DevTopo& T, const SL& S, const TapeStep& tp, int it, int slot, float lam,
                                          int br) {
  S[T.sm_lam + slot] = lam;
  if (TAPE) {
    const int o = (it * T.nslots + slot) * 32;
    tp.lam[o] = lam;
    if (!EQ || T.rec_rows) tp.br[o] = (uint8_t)br;
  }
}
template <int AX>
__device__ __forceinline__ float& axis_of(float3& v) {
  return AX == 0 ? v.x : (AX == 1 ? v.y : v.z);
}

// The parent's share of J v of a row along a coordinate axis.
template <bool SEQ>
__device__ __forceinline__ float jv_lin(float v, float3 ang, float3 w) {
  return SEQ ? fmaf(ang.z, w.z, fmaf(ang.y, w.y, fmaf(ang.x, w.x, v))) : __fadd_rn(v, dotx(ang, w));
}
// v +- dl im, fused (SEQ) or with the impulse's velocity rounded first.
template <bool SEQ>
__device__ __forceinline__ void lin_add(float& v, float dl, float im) {
  v = SEQ ? fmaf(dl, im, v) : __fadd_rn(v, __fmul_rn(dl, im));
}
template <bool SEQ>
__device__ __forceinline__ void lin_sub(float& v, float dl, float im) {
  v = SEQ ? fmaf(-dl, im, v) : __fsub_rn(v, __fmul_rn(dl, im));
}

// The blocks' bodies: va, wa, vb, wb are the velocities of the parent and the child (zeros for the
// world). Everything a block reads from the record is loaded before its first row and every result
// is stored after its last one: a store between the rows would keep the loads of the next row behind
// it, and each row would wait for shared memory (some 30 cycles) besides its own chain of products.
// ready() meets the barrier of the level before and loads the velocities: all that only this block
// changes (its record, its impulses) is loaded ahead of it, while the warp would wait there.
template <bool TAPE, bool SEQ, bool FULL, class RD>
__device__ __forceinline__ void joint_rows(const DevTopo& T, const SL& S, const TapeStep& tp, int it, const BlkOp& op,
                                           const SL& R, float ima, float imb, float3& va, float3& wa, float3& vb,
                                           float3& wb, const RD& ready) {
  const int mask = FULL ? 31 : op.mask(), s0 = op.slot();
  const float3 ra = R.v3(JF_RA), rb = R.v3(JF_RB);
  float lam[5], me[5], bi[5];
  float3 IA[5], IB[5], t[2];
#pragma unroll
  for (int k = 0; k < 5; ++k)
    if (mask >> k & 1) {
      lam[k] = S[T.sm_lam + s0 + k];
      me[k] = R[JF_ME + k];
      bi[k] = R[JF_BI + k];
      IA[k] = R.v3(k < 3 ? JF_IAL + 3 * k : JF_IAT + 3 * (k - 3));
      IB[k] = R.v3(k < 3 ? JF_IBL + 3 * k : JF_IBT + 3 * (k - 3));
      if (k >= 3) t[k - 3] = R.v3(JF_T + 3 * (k - 3));
    }
  ready();
  int br;
  auto lin = [&](auto KI) {
    constexpr int k = decltype(KI)::value;
    if (!(mask >> k & 1)) return;
    const float3 angA = cross_axis<k>(ra), angB = -cross_axis<k>(rb);
    const float Jv = jv_lin<SEQ>(axis_of<k>(va), angA, wa) + (dotx(angB, wb) - axis_of<k>(vb));
    const float dl = row_solve<true>(T, Jv, me[k], bi[k], 0.f, 0.f, lam[k], br);
    lin_add<SEQ>(axis_of<k>(va), dl, ima);
    wa = axpy3(dl, IA[k], wa);
    lin_sub<SEQ>(axis_of<k>(vb), dl, imb);
    wb = axpy3(dl, IB[k], wb);
  };
  lin(std::integral_constant<int, 0>{});
  lin(std::integral_constant<int, 1>{});
  lin(std::integral_constant<int, 2>{});
#pragma unroll
  for (int k = 3; k < 5; ++k) {
    if (!(mask >> k & 1)) continue;
    const float Jv = dotx(t[k - 3], wa) + dotx(-t[k - 3], wb);
    const float dl = row_solve<true>(T, Jv, me[k], bi[k], 0.f, 0.f, lam[k], br);
    wa = axpy3(dl, IA[k], wa);
    wb = axpy3(dl, IB[k], wb);
  }
#pragma unroll
  for (int k = 0; k < 5; ++k)
    if (mask >> k & 1) row_store<TAPE, true>(T, S, tp, it, s0 + k, lam[k], 0);
}
template <bool TAPE, class RD>
__device__ __forceinline__ void hinge_row(const DevTopo& T, const SL& S, const TapeStep& tp, int it, const BlkOp& op,
                                          const SL& R, float3& wa, float3& wb, const RD& ready) {
  const bool lim = op.type() == BT_LIMIT;
  const int m = lim ? 5 : 6, s = op.slot();
  const float sg = lim ? R[JF_LS] : 1.f;
  const int j = op.idx();
  const float3 angB = sg * S.v3(T.sm_ua + 3 * j), angA = -angB;
  float lam = S[T.sm_lam + s];
  const float me = R[JF_ME + m], bi = R[JF_BI + m];
  const float hi = lim ? __int_as_float(0x7f800000) : R[JF_BND], lo = lim ? 0.f : -hi;
  const float3 IA = -(sg * R.v3(JF_IAU)), IB = sg * R.v3(JF_IBU);
  ready();
  const float Jv = dotx(angA, wa) + dotx(angB, wb);
  int br;
  const float dl = row_solve<false>(T, Jv, me, bi, lo, hi, lam, br);
  wa = axpy3(dl, IA, wa);
  wb = axpy3(dl, IB, wb);
  row_store<TAPE, false>(T, S, tp, it, s, lam, br);
}
template <bool TAPE, bool SEQ, bool FULL, class RD>
__device__ __forceinline__ void contact_rows(const DevTopo& T, const SL& S, const TapeStep& tp, int it, const BlkOp& op,
                                             const SL& R, float ima, float3& va, float3& wa, const RD& ready) {
  const int mask = FULL ? 7 : op.mask(), s0 = op.slot();
  const float3 ra = R.v3(CF_RA);
  float lam[3], me[3];
  float3 IA[3];
  int br[3];
#pragma unroll
  for (int m = 0; m < 3; ++m)
    if (mask >> m & 1) {
      lam[m] = S[T.sm_lam + s0 + m];
      me[m] = R[CF_ME + m];
      IA[m] = R.v3(CF_I + 3 * m);
    }
  const float bias = R[CF_BI], mu = R[CF_MU];
  ready();
  if (!(mask & 1)) lam[0] = S[T.sm_lam + s0];  // the friction rows' bound: another block's impulse
  auto row = [&](auto MI, auto AI, float lo, float hi, float b) {
    constexpr int m = decltype(MI)::value, ax = decltype(AI)::value;
    const float3 angA = cross_axis<ax>(ra);
    const float Jv = jv_lin<SEQ>(axis_of<ax>(va), angA, wa);
    const float dl = row_solve<false>(T, Jv, me[m], b, lo, hi, lam[m], br[m]);
    lin_add<SEQ>(axis_of<ax>(va), dl, ima);
    wa = axpy3(dl, IA[m], wa);
  };
  using I0 = std::integral_constant<int, 0>;
  using I1 = std::integral_constant<int, 1>;
  using I2 = std::integral_constant<int, 2>;
  if (mask & 1) row(I0{}, I2{}, 0.f, __int_as_float(0x7f800000), bias);
  const float hi = mu * lam[0];
  if (mask & 2) row(I1{}, I0{}, -hi, hi, 0.f);
  if (mask & 4) row(I2{}, I1{}, -hi, hi, 0.f);
#pragma unroll
  for (int m = 0; m < 3; ++m)
    if (mask >> m & 1) row_store<TAPE, false>(T, S, tp, it, s0 + m, lam[m], br[m]);
}
template <bool TAPE, class RD>
__device__ __forceinline__ void pair_rows(const DevTopo& T, const SL& S, const TapeStep& tp, int it, const BlkOp& op,
                                          const SL& R, float ima, float imb, float3& va, float3& wa, float3& vb,
                                          float3& wb, const RD& ready) {
  const int mask = op.mask(), s0 = op.slot();
  ready();
  float ln = S[T.sm_lam + s0];
#pragma unroll 1
  for (int m = 0; m < 3; ++m) {
    if (!(mask >> m & 1)) continue;
    const float3 lin = R.v3(PF_LIN + 3 * m), angA = R.v3(PF_ANGA + 3 * m), angB = R.v3(PF_ANGB + 3 * m);
    float lam = S[T.sm_lam + s0 + m];
    float lo = 0.f, hi = __int_as_float(0x7f800000);
    if (m > 0) { hi = R[PF_MU] * ln; lo = -hi; }
    float Jv = 0.f;
    Jv += dotx(lin, va) + dotx(angA, wa);
    Jv += dotx(angB, wb) - dotx(lin, vb);
    int br;
    const float dl = row_solve<false>(T, Jv, R[PF_ME + m], m == 0 ? R[PF_BI] : 0.f, lo, hi, lam, br);
    row_store<TAPE, false>(T, S, tp, it, s0 + m, lam, br);
    if (m == 0) ln = lam;
    va = va + (dl * ima) * lin;
    wa = wa + dl * R.v3(PF_IA + 3 * m);
    vb = vb - (dl * imb) * lin;
    wb = wb + dl * R.v3(PF_IB + 3 * m);
  }
}

// The projected Gauss-Seidel sweeps of the step (every warp calls; ends after a CTA barrier). With
// TAPE the impulses and clamp branches of every update and the velocities after every sweep go to
// the tape.
template <bool TAPE, bool SEQ>
__device__ __forceinline__ void blk_sweeps(const DevTopo& T, const SL& S, const SL& X, const TapeStep& tp, int warp) {
  const uint8_t* st0 = blk_bytes(T) + T.blk_stream + warp * T.blk_stream_len;
  const int nv = 6 * T.nb;
  auto load = [&](int a, float3& v, float3& w, float& im) {
    v = w = f3(0.f, 0.f, 0.f);
    im = 0.f;
    if (a < 0) return;
    v = X.v3(18 * a + 12);
    w = X.v3(18 * a + 15);
    im = S[T.sm_invm + a];
  };
  auto store = [&](int a, float3 v, float3 w) {
    if (a < 0) return;
    X.s3(18 * a + 12, v);
    X.s3(18 * a + 15, w);
  };
  auto rows = [&](const BlkOp& op, int it, float ima, float imb, float3& va, float3& wa, float3& vb, float3& wb,
                  const auto& ready) {
    const int type = op.type(), idx = op.idx();
    const SL R = type == BT_GROUND ? contact_rec(T, S, idx) : (type == BT_PAIR ? pair_rec(T, S, idx) : joint_rec(T, S, idx));
    switch (type) {
      case BT_JOINT:
        if (op.mask() == 31) joint_rows<TAPE, SEQ, true>(T, S, tp, it, op, R, ima, imb, va, wa, vb, wb, ready);
        else joint_rows<TAPE, SEQ, false>(T, S, tp, it, op, R, ima, imb, va, wa, vb, wb, ready);
        break;
      case BT_GROUND:
        if (op.mask() == 7) contact_rows<TAPE, SEQ, true>(T, S, tp, it, op, R, ima, va, wa, ready);
        else contact_rows<TAPE, SEQ, false>(T, S, tp, it, op, R, ima, va, wa, ready);
        break;
      case BT_PAIR: pair_rows<TAPE>(T, S, tp, it, op, R, ima, imb, va, wa, vb, wb, ready); break;
      default: hinge_row<TAPE>(T, S, tp, it, op, R, wa, wb, ready); break;
    }
  };
  if (!SEQ && T.blk_single) {
    // one block (never a compiled topology): warp 0 keeps its bodies' velocities in registers over the sweeps
    if (warp == 0) {
      const bool on = st0[0] != 0;
      const BlkOp op = blk_op(T, 0);
      const int a = op.a(), b = op.b();
      float3 va, wa, vb, wb;
      float ima, imb;
      load(a, va, wa, ima);
      load(b, vb, wb, imb);
      for (int it = 0; it < T.iters; ++it) {
        if (on) rows(op, it, ima, imb, va, wa, vb, wb, [] {});
        if (TAPE)
          for (int c = 0; c < T.nb; ++c) {
            float* vi = tp.viter + (it * nv + 6 * c) * 32;
            const float3 v = c == a ? va : (c == b ? vb : X.v3(18 * c + 12));
            const float3 w = c == a ? wa : (c == b ? wb : X.v3(18 * c + 15));
            vi[0] = v.x; vi[32] = v.y; vi[64] = v.z;
            vi[96] = w.x; vi[128] = w.y; vi[160] = w.z;
          }
      }
      store(a, va, wa);
      store(b, vb, wb);
    }
    cta_sync();
    return;
  }
  bool pend = false;  // a barrier to meet before the next velocities are read
  for (int it = 0; it < T.iters; ++it) {
    const uint8_t* st = st0;
    int e = *st++;
    BlkOp nop = blk_op(T, e & 63);
    while (e) {
      const int nxt = *st++;  // (a stream ends with a zero; one more byte is allocated)
      const BlkOp op = nop;
      nop = blk_op(T, nxt & 63);  // the next entry's block while this one runs
      if (e & BS_OP) {
        const int a = op.a(), b = op.b();
        float3 va = f3(0.f, 0.f, 0.f), wa = va, vb = va, wb = va;
        const float ima = a >= 0 ? S[T.sm_invm + a] : 0.f, imb = b >= 0 ? S[T.sm_invm + b] : 0.f;
        rows(op, it, ima, imb, va, wa, vb, wb, [&] {
          if (pend) cta_sync();
          if (a >= 0) { va = X.v3(18 * a + 12); wa = X.v3(18 * a + 15); }
          if (b >= 0) { vb = X.v3(18 * b + 12); wb = X.v3(18 * b + 15); }
        });
        store(a, va, wa);
        store(b, vb, wb);
      } else if (pend) {
        cta_sync();
      }
      pend = e & BS_BAR;
      e = nxt;
    }
    if (TAPE) {
      if (pend) cta_sync();
      float* vi = tp.viter + it * nv * 32;
      for (int b = warp; b < T.nb; b += blk_nw())
#pragma unroll
        for (int k = 0; k < 6; ++k) vi[(6 * b + k) * 32] = X[18 * b + 12 + k];
      pend = true;
    }
  }
  cta_sync();
}
