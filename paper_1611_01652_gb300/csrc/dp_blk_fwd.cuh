// The rollout kernel on blocks, one CTA per group of 32 instances (stages of dp_blk.cuh).
#pragma once
#include "dp_blk.cuh"

// What a kernel is built for: CTRL_H the hidden width of the tensor-core controller it carries (0:
// every supported width, dispatched at run time); SEQ the order of the sums in a row update. With
// SEQ the parent's share of J v is one chain of multiply-adds from the linear velocity on and the
// linear update is fused (the quadruped's and the arms' worlds); without it the angular product is
// summed by itself and the linear impulse is rounded first (every other robot). Each keeps the
// rounding its worlds have always had. NW: the warps of a CTA (plan_blocks in dp_plan.cu).
struct BlkQuad {
  static constexpr int CTRL_H = 128, NW = 8;
  static constexpr bool SEQ = true;
};
struct BlkArm {
  static constexpr int CTRL_H = 256, NW = 8;
  static constexpr bool SEQ = true;
};
struct BlkDyn {
  static constexpr int CTRL_H = 0, NW = 4;
  static constexpr bool SEQ = false;
};

// ------------------------------------------------------------------------------ controller
// bfloat16 hidden activations in shared memory: [32 instances][H + 8] per layer. The padding puts
// the eight rows of an A fragment in different banks.
template <int H>
__device__ __forceinline__ __nv_bfloat16* ctrl_hidden(const DevTopo& T, int l) {
  return reinterpret_cast<__nv_bfloat16*>(g_smem + T.sm_hbuf * 32) + (l - 1) * 32 * (H + 8);
}
template <int H>
__device__ __forceinline__ void load_a_smem(const __nv_bfloat16* h, int mt, int kt, uint32_t (&a)[4]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  const uint32_t* p = reinterpret_cast<const uint32_t*>(h + (mt * 16 + g) * (H + 8) + kt * 16 + 2 * q);
  a[0] = p[0];
  a[1] = p[4 * (H + 8)];
  a[2] = p[4];
  a[3] = p[4 * (H + 8) + 4];
}
// ReLU and bfloat16 storage of one 16-row tile's NT column tiles (first column n1) into a hidden
// layer's buffer, and fp32 into the dump (feature-major) when given.
template <int H, int NT>
__device__ __forceinline__ void store_hidden(const float (&acc)[NT][4], int mt, int n1, __nv_bfloat16* h, float* dump,
                                             size_t N) {
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
    const int c = n1 + nt * 8 + 2 * q, r0 = mt * 16 + g;
    float v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = __bfloat162float(__float2bfloat16_rn(fmaxf(acc[nt][k], 0.f)));
    *reinterpret_cast<uint32_t*>(h + r0 * (H + 8) + c) = pack_bf16(v[0], v[1]);
    *reinterpret_cast<uint32_t*>(h + (r0 + 8) * (H + 8) + c) = pack_bf16(v[2], v[3]);
    if (dump) {
      dump[(size_t)c * N + r0] = v[0];
      dump[(size_t)(c + 1) * N + r0] = v[1];
      dump[(size_t)c * N + r0 + 8] = v[2];
      dump[(size_t)(c + 1) * N + r0 + 8] = v[3];
    }
  }
}

// The tensor-core controller on the CTA's warps: each hidden layer's columns are split over
// the warps (both 16-row tiles of a weight fragment are multiplied with one load of it), the
// output layer's two row tiles over warps 0 and 1. Every output's sum runs over k in increasing
// order. in: the features, out: the outputs, dump: the step's dump column of lane 0 (or NULL).
// Called by every warp with the features complete; the outputs are complete after the caller's
// next barrier.
template <int H, int NW>
__device__ __forceinline__ void ctrl_forward_nw(const DevTopo& T, const DevPtrs& D, const SL& in, const SL& out,
                                                float* dump, int warp) {
  constexpr int NT = H / (8 * NW), KT = H / 16, KT0 = CTRL_TC_KP0 / 16;
  constexpr CtrlTCLayout Lw = ctrl_tc_layout(H, H);
  const __nv_bfloat16* Wc = D.Wtc;
  const size_t N = (size_t)T.horizon * T.Bp;
  const int n1 = warp * (H / NW), K0 = T.widths[0], no = T.widths[3];
  __nv_bfloat16 *h1 = ctrl_hidden<H>(T, 1), *h2 = ctrl_hidden<H>(T, 2);
  {
    float acc[2][NT][4];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) bias_init<NT>(D.bias + T.w_off[0], n1, H, acc[mt]);
#pragma unroll
    for (int kt = 0; kt < KT0; ++kt) {
      uint32_t a[2][4];
      auto x = [&](int f, int r) { return in.lane_at(f, r); };
#pragma unroll
      for (int mt = 0; mt < 2; ++mt) load_a_lanes(x, K0, mt, kt, a[mt]);
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        uint32_t b0, b1;
        load_b(Wc + Lw.w1, CTRL_TC_KP0, n1 + nt * 8, kt * 16, b0, b1);
        mma_bf16_16816(acc[0][nt], a[0], b0, b1);
        mma_bf16_16816(acc[1][nt], a[1], b0, b1);
      }
    }
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
      store_hidden<H, NT>(acc[mt], mt, n1, h1, dump ? dump + (size_t)T.dump_act[1] * N : nullptr, N);
  }
  cta_sync();
  {
    float acc[2][NT][4];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) bias_init<NT>(D.bias + T.w_off[1], n1, H, acc[mt]);
#pragma unroll 4
    for (int kt = 0; kt < KT; ++kt) {
      uint32_t a[2][4];
      load_a_smem<H>(h1, 0, kt, a[0]);
      load_a_smem<H>(h1, 1, kt, a[1]);
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        uint32_t b0, b1;
        load_b(Wc + Lw.w2, H, n1 + nt * 8, kt * 16, b0, b1);
        mma_bf16_16816(acc[0][nt], a[0], b0, b1);
        mma_bf16_16816(acc[1][nt], a[1], b0, b1);
      }
    }
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
      store_hidden<H, NT>(acc[mt], mt, n1, h2, dump ? dump + (size_t)T.dump_act[2] * N : nullptr, N);
  }
  cta_sync();
  if (warp < 2) {
    float acc[2][4];
    bias_init<2>(D.bias + T.w_off[2], 0, no, acc);
#pragma unroll 4
    for (int kt = 0; kt < KT; ++kt) {
      uint32_t a[4];
      load_a_smem<H>(h2, warp, kt, a);
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) {
        uint32_t b0, b1;
        load_b(Wc + Lw.w3, H, nt * 8, kt * 16, b0, b1);
        mma_bf16_16816(acc[nt], a, b0, b1);
      }
    }
    store_c<2>(acc, warp, 0, no, [&](int f, int r, float v) { out.lane_at(f, r) = v; });
  }
}
template <int H, int NW>
__device__ __noinline__ void ctrl_forward_nw_call(const DevTopo& T, const DevPtrs& D, SL in, SL out, float* dump, int warp) {
  ctrl_forward_nw<H, NW>(T, D, in, out, dump, warp);
}
template <class Q>
__device__ __forceinline__ void ctrl_forward_blk(const DevTopo& T, const DevPtrs& D, const SL& in, const SL& out,
                                                 float* dump, int warp) {
  if constexpr (Q::CTRL_H == 128) {
    ctrl_forward_nw<128, Q::NW>(T, D, in, out, dump, warp);
  } else if constexpr (Q::CTRL_H == 256) {
    ctrl_forward_nw_call<256, Q::NW>(T, D, in, out, dump, warp);
  } else {
    if (T.widths[1] == 64) ctrl_forward_nw_call<64, Q::NW>(T, D, in, out, dump, warp);
    else if (T.widths[1] == 128) ctrl_forward_nw_call<128, Q::NW>(T, D, in, out, dump, warp);
    else ctrl_forward_nw_call<256, Q::NW>(T, D, in, out, dump, warp);
  }
}

// The fp32-arithmetic controller on the CTA's warps: 8 outputs of a layer per warp and pass.
__device__ __forceinline__ void controller_forward_nw(const DevTopo& T, const DevPtrs& D, const SL* act, int warp) {
  for (int l = 0; l < T.n_layers; ++l) {
    dense_fwd(D.Wt + T.w_off[l], D.bias + T.w_off[l], T.widths[l], T.widths[l + 1], act[l], act[l + 1],
              l + 1 < T.n_layers, false, T.ctrl_round != 0, 8 * warp, 8 * blk_nw());
    if (l + 1 < T.n_layers) cta_sync();
  }
  if (T.skip) {  // a warp adds to the outputs it wrote
    const int l = T.n_layers;
    dense_fwd(D.Wt + T.w_off[l], D.bias + T.w_off[l], T.widths[0], T.widths[l], act[0], act[l], false, true, false,
              8 * warp, 8 * blk_nw());
  }
}

// Hinge kinematics of this warp's joints, and the controller's inputs: joint angles and rates by
// the joint's warp, the rest by warp 3 (the clock from the table made at creation).
__device__ __forceinline__ void blk_features(const DevTopo& T, const DevPtrs& D, const LaneT<SL>& L, const SL& X, int t,
                                             const SL& act0, int warp) {
  const SL& S = L.S;
  int k = 0;
  if (T.features & 1) {
    for (int m = 0; m < T.n_motors; ++m) {
      const int j = T.motor_joint[m];
      if ((j & (blk_nw() - 1)) == warp) act0[k + m] = qz(T, S[T.sm_th + j]);
    }
    k += T.n_motors;
  }
  if (T.features & 2) {
    for (int m = 0; m < T.n_motors; ++m) {
      const int j = T.motor_joint[m];
      if ((j & (blk_nw() - 1)) == warp) act0[k + m] = qz(T, S[T.sm_thd + j]);
    }
    k += T.n_motors;
  }
  if (warp != 3) return;
  if (T.features & 4) {
    float s, c;
    if (t < T.horizon) {
      s = __ldg(D.clk + 2 * t);
      c = __ldg(D.clk + 2 * t + 1);
    } else {
      clock_features(T, t, s, c);
    }
    act0[k++] = qz(T, s);
    act0[k++] = qz(T, c);
  }
  if (T.features & 8) {
    const int b = T.imu_body;
    const M3 R = loadR(X, 18 * b);
    const float3 g = mtv(R, f3(0.f, 0.f, -1.f));
    const float3 wl = mtv(R, X.v3(18 * b + 15));
    act0[k++] = qz(T, g.x); act0[k++] = qz(T, g.y); act0[k++] = qz(T, g.z);
    act0[k++] = qz(T, wl.x); act0[k++] = qz(T, wl.y); act0[k++] = qz(T, wl.z);
  }
  if (T.features & 16) {
    const float3 d = loss_point(T, L, X) - L.P.v3(T.o_loss_target);
    act0[k++] = qz(T, d.x); act0[k++] = qz(T, d.y); act0[k++] = qz(T, d.z);
  }
  for (; k < T.widths[0]; ++k) act0[k] = 0.f;
  if (T.n_rec) {  // recurrent state h^t: the last inputs (a bfloat16 storage point like the sensors)
    const int base = T.widths[0] - T.n_rec;
    for (int q = 0; q < T.n_rec; ++q) act0[base + q] = qz(T, S[T.sm_h + q]);
  }
}

// ------------------------------------------------------------------------------ warm start
// The damped previous-impulse start of this warp's items: alpha times the impulses the rows ended
// the previous step with, projected on the rows' bounds; limits start cold.
__device__ __forceinline__ void blk_damped_start(const DevTopo& T, const SL& S, int warp) {
  const SL lam = S.at(T.sm_lam);
  for (int j = warp; j < T.nj; j += blk_nw()) {
    const SL R = joint_rec(T, S, j);
    const int s0 = T.jslot[j], n = T.jtype[j] == 1 ? 5 : 3;
    for (int k = 0; k < n; ++k) lam[s0 + k] = R[JF_ME + k] != 0.f ? T.ws_alpha * lam[s0 + k] : 0.f;
    if (T.jlim[j] >= 0) lam[T.jlim[j]] = 0.f;
    if (T.jmot[j] >= 0) {
      const int s = T.jmot[j];
      const float y = R[JF_ME + 6] != 0.f ? T.ws_alpha * lam[s] : 0.f, hi = R[JF_BND];
      lam[s] = fminf(fmaxf(y, -hi), hi);
    }
  }
  auto touch = [&](int s0, float me, float mu) {
    float l[3] = {0.f, 0.f, 0.f};
    if (me != 0.f) {
      l[0] = fmaxf(T.ws_alpha * lam[s0], 0.f);
      const float hi = mu * l[0];
      l[1] = fminf(fmaxf(T.ws_alpha * lam[s0 + 1], -hi), hi);
      l[2] = fminf(fmaxf(T.ws_alpha * lam[s0 + 2], -hi), hi);
    }
    for (int k = 0; k < 3; ++k) lam[s0 + k] = l[k];
  };
  // (the warp that has formed the record: there is no barrier in between)
  for (int q = warp; q < T.ns; q += blk_nw()) {
    const SL R = contact_rec(T, S, q);
    touch(T.cslot + 3 * q, R[CF_ME], R[CF_MU]);
  }
  for (int p = warp; p < T.np; p += blk_nw()) {
    const SL R = pair_rec(T, S, p);
    touch(T.cslot + 3 * (T.ns + p), R[PF_ME], R[PF_MU]);
  }
}

// v += M^-1 J^T lambda0 for the bodies of this warp, each body's rows in slot order.
__device__ __forceinline__ void blk_apply_start(const DevTopo& T, const SL& S, const SL& X, int warp) {
  const SL lam = S.at(T.sm_lam);
  const uint8_t* first = blk_bytes(T) + T.blk_inc0;
  const uint8_t* inc = blk_bytes(T) + T.blk_inc;
  for (int b = warp; b < T.nb; b += blk_nw()) {
    float3 v = X.v3(18 * b + 12), w = X.v3(18 * b + 15);
    const float im = S[T.sm_invm + b];
    const int k0 = first[b], k1 = first[b + 1];
    auto put = [&](float l, int ax, float sg, float3 I) {
      const float c = __fmul_rn(l, im) * sg;
      if (ax == 0) v.x = __fadd_rn(v.x, c);
      if (ax == 1) v.y = __fadd_rn(v.y, c);
      if (ax == 2) v.z = __fadd_rn(v.z, c);
      w = f3(fmaf(l, I.x, w.x), fmaf(l, I.y, w.y), fmaf(l, I.z, w.z));
    };
    for (int k = k0; k < k1 && inc[k] < 0x40; ++k) {
      const int j = inc[k] & 31, s0 = T.jslot[j];
      const bool sb = inc[k] & 0x20;
      const SL R = joint_rec(T, S, j);
      const float sg = sb ? -1.f : 1.f;
#pragma unroll
      for (int q = 0; q < 3; ++q) put(lam[s0 + q], q, sg, R.v3((sb ? JF_IBL : JF_IAL) + 3 * q));
      if (T.jtype[j] == 1)
#pragma unroll
        for (int q = 0; q < 2; ++q) put(lam[s0 + 3 + q], -1, sg, R.v3((sb ? JF_IBT : JF_IAT) + 3 * q));
    }
    for (int k = k0; k < k1 && inc[k] < 0x40; ++k) {  // servo rows (limit rows start cold)
      const int j = inc[k] & 31;
      if (T.jmot[j] < 0) continue;
      const SL R = joint_rec(T, S, j);
      const float3 I = inc[k] & 0x20 ? R.v3(JF_IBU) : -R.v3(JF_IAU);
      put(lam[T.jmot[j]], -1, 1.f, I);
    }
    for (int k = k0; k < k1; ++k) {
      if (inc[k] < 0x40) continue;
      const int c = inc[k] & 31;
      if (inc[k] < 0x80) {
        const SL R = contact_rec(T, S, c);
        const int s0 = T.cslot + 3 * c;
        put(lam[s0], 2, 1.f, R.v3(CF_I));
        put(lam[s0 + 1], 0, 1.f, R.v3(CF_I + 3));
        put(lam[s0 + 2], 1, 1.f, R.v3(CF_I + 6));
      } else {
        const bool sb = inc[k] & 0x20;
        const SL R = pair_rec(T, S, c);
        const int s0 = T.cslot + 3 * (T.ns + c);
        for (int m = 0; m < 3; ++m) {
          const float l = lam[s0 + m], c1 = (sb ? -1.f : 1.f) * __fmul_rn(l, im);
          v = v + c1 * R.v3(PF_LIN + 3 * m);
          w = w + l * R.v3((sb ? PF_IB : PF_IA) + 3 * m);
        }
      }
    }
    X.s3(18 * b + 12, v);
    X.s3(18 * b + 15, w);
  }
}

__device__ __forceinline__ float rec_jv(const RowRec& R, const SL& X, int a, int b) {
  float Jv = 0.f;
  if (a >= 0) Jv += dot3(R.lin, X.v3(18 * a + 12)) + dot3(R.angA, X.v3(18 * a + 15));
  if (b >= 0) Jv += dot3(R.angB, X.v3(18 * b + 15)) - dot3(R.lin, X.v3(18 * b + 12));
  return Jv;
}

// The learned start and the harvest of training rows (see warm_start in dp_forward.cuh), the row
// groups split over the warps: features, the network on the tensor cores, projection. Called
// after the records are complete; the application is blk_apply_start's.
static __device__ __noinline__ void blk_network_start(const DevTopo& T, const DevPtrs& D, const LaneT<SL> L, const SL X,
                                                      int warp) {
  const SL S = L.S, lam = S.at(T.sm_lam);
  const bool harvest = D.harvest != nullptr;
  float mtot = 0.f;
  float3 pc = f3(0.f, 0.f, 0.f);
  int nact = 0;
  for (int b = 0; b < T.nb; ++b) {
    const float m = L.P[T.o_mass + b];
    mtot += m;
    pc += m * X.v3(18 * b);
  }
  pc = (1.f / mtot) * pc;
  for (int c = 0; c < T.ns + T.np; ++c)
    if ((c < T.ns ? contact_rec(T, S, c)[CF_ME] : pair_rec(T, S, c - T.ns)[PF_ME]) != 0.f) ++nact;
  const float gn = sqrtf(T.gravity[0] * T.gravity[0] + T.gravity[1] * T.gravity[1] + T.gravity[2] * T.gravity[2]);
  const float share = mtot * gn * T.dt / (float)max(1, nact);
  const SL F = S.at(T.sm_ws + 19 * warp), Y = S.at(T.sm_ws + 19 * warp + 16), H = S.at(T.sm_ws + 19 * blk_nw());
  const int lane = threadIdx.x & 31;
  for (int g = warp; g < T.n_wsg; g += blk_nw()) {
    const int type = T.wsg_type[g];
    const int s0 = T.wsg_slot[g][0], s1 = T.wsg_slot[g][1], s2 = T.wsg_slot[g][2];
    const bool contact = type == WSG_GROUND || type == WSG_PAIR;
    float lp[3], bnd[3];
    bool act0 = false;
    for (int k = 0; k < 3; ++k) {
      const int s = T.wsg_slot[g][k];
      lp[k] = s >= 0 ? lam[s] : 0.f;
      RowRec R{};
      if (s >= 0) R = blk_row(T, S, s);
      const bool on = s >= 0 && R.meff != 0.f;  // rows of inactive slots contribute zeros
      F[k] = on ? rec_jv(R, X, T.sa[s], T.sb[s]) : 0.f;
      F[3 + k] = on ? R.bias : 0.f;
      F[6 + k] = on ? R.meff : 0.f;
      bnd[k] = s >= 0 ? R.bnd : 0.f;
      if (k == 0) act0 = on;
    }
    float3 q;  // the group's point: contact point on body a, or the joint's anchor on its child
    if (type == WSG_GROUND) {
      const int qi = T.sidx[s0], a = T.sa[s0];
      q = X.v3(18 * a) + mv(loadR(X, 18 * a), L.P.v3(T.o_sph_off + 3 * qi)) - L.P[T.o_sph_rad + qi] * f3(0.f, 0.f, 1.f);
    } else if (type == WSG_PAIR) {
      const int k = T.pk[T.sidx[s0]], a = T.sa[s0];
      q = X.v3(18 * a) + mv(loadR(X, 18 * a), L.P.v3(T.o_sph_off + 3 * k)) -
          L.P[T.o_sph_rad + k] * pair_rec(T, S, T.sidx[s0]).v3(PF_LIN);
    } else {
      const int j = T.sidx[s0], b = T.sb[s0];
      q = X.v3(18 * b) + mv(loadR(X, 18 * b), L.P.v3(T.o_anchor + 6 * j + 3));
    }
    F[9] = contact ? bnd[1] : (type == WSG_HINGE && s2 >= 0 ? bnd[2] : 0.f);
    F[10] = q.x - pc.x;
    F[11] = q.y - pc.y;
    F[12] = (float)nact;
    F[13] = share;
    F[14] = q.z - T.ground_z;
    F[15] = (float)type;
    if (harvest) {  // padded lanes (copies of the last instance) harvest nothing
      const unsigned m = __ballot_sync(FULLMASK, act0 && L.i < T.B);
      unsigned long long base = 0;
      if (lane == 0 && m) base = atomicAdd(D.harvest_count, (unsigned long long)__popc(m));
      base = __shfl_sync(FULLMASK, base, 0);
      const long long id = (m >> lane) & 1u ? (long long)(base + __popc(m & ((1u << lane) - 1u))) : -1;
      const bool keep = id >= 0 && id < D.harvest_max;
      H[g] = __int_as_float(keep ? (int)id : -1);
      if (keep) {
        for (int k = 0; k < 16; ++k) D.harvest[id * 19 + k] = F[k];
        for (int k = 0; k < 3; ++k) D.harvest[id * 19 + 16 + k] = lp[k];  // replaced after the solve
      }
    }
    if (T.ws) {
      float z[3];
      if (T.ws_net) {
        __syncwarp();
        mlp3_forward<WsTC::K0, WsTC::H1, WsTC::H2, WsTC::NO>(
            WsTC::K0, WsTC::NO,
            [&](int f, int r) { return F.lane_at(f, r); }, D.ws_tc + WsTC::W1, D.ws_b + WsTC::B1, D.ws_tc + WsTC::W2,
            D.ws_b + WsTC::B2, D.ws_tc + WsTC::W3, D.ws_b + WsTC::B3,
            [&](int f, int r, float v) { Y.lane_at(f, r) = v; }, [](int, int, int, float) {});
        __syncwarp();
        for (int k = 0; k < 3; ++k) z[k] = T.ws_alpha * lp[k] + F[6 + k] * Y[k];
      } else {
        for (int k = 0; k < 3; ++k) z[k] = T.ws_alpha * lp[k];
      }
      if (contact) {
        float l0[3] = {0.f, 0.f, 0.f};
        if (act0) {
          l0[0] = fmaxf(z[0], 0.f);
          const float hi = bnd[1] * l0[0];
          l0[1] = fminf(fmaxf(z[1], -hi), hi);
          l0[2] = fminf(fmaxf(z[2], -hi), hi);
        }
        lam[s0] = l0[0];
        lam[s1] = l0[1];
        lam[s2] = l0[2];
      } else {
        for (int k = 0; k < 3; ++k) {
          const int s = T.wsg_slot[g][k];
          if (s < 0) continue;
          float y = F[6 + k] != 0.f ? z[k] : 0.f;
          if (T.skind[s] == RK_MOTOR) y = fminf(fmaxf(y, -bnd[k]), bnd[k]);
          lam[s] = y;
        }
      }
      __syncwarp();
    }
  }
  if (T.ws)
    for (int j = warp; j < T.nj; j += blk_nw())
      if (T.jlim[j] >= 0) lam[T.jlim[j]] = 0.f;  // limits start cold
}

// Harvest: per reserved group, the network's ideal output (see harvest_finish in dp_forward.cuh).
static __device__ __noinline__ void blk_harvest_finish(const DevTopo& T, const DevPtrs& D, const SL S, int warp) {
  const SL H = S.at(T.sm_ws + 19 * blk_nw());
  for (int g = warp; g < T.n_wsg; g += blk_nw()) {
    const int id = __float_as_int(H[g]);
    if (id < 0) continue;
    float* row = D.harvest + (long long)id * 19;
    for (int k = 0; k < 3; ++k) {
      const int s = T.wsg_slot[g][k];
      const float me = row[6 + k];
      row[16 + k] = me != 0.f ? ((s >= 0 ? S[T.sm_lam + s] : 0.f) - T.ws_alpha * row[16 + k]) / me : 0.f;
    }
  }
}

// RMS complementarity residual of the solve (see solve_residual in dp_forward.cuh).
static __device__ __noinline__ float blk_residual(const DevTopo& T, const SL S, const SL X) {
  float ss = 0.f;
  int na = 0;
  for (int s = 0; s < T.nslots; ++s) {
    const RowRec R = blk_row(T, S, s);
    if (R.meff == 0.f) continue;
    const int kind = T.skind[s];
    const float l = S[T.sm_lam + s];
    const float w = rec_jv(R, X, T.sa[s], T.sb[s]) + R.bias + T.gamma * l;
    float e;
    if (kind == RK_JLIN || kind == RK_JANG) {
      e = w;
    } else if (kind == RK_LIMIT || kind == RK_GN || kind == RK_PN) {
      e = fminf(l, w);
    } else {
      const float hi = (kind == RK_MOTOR) ? R.bnd : R.bnd * S[T.sm_lam + T.snormal[s]];
      e = l - fminf(fmaxf(l - w, -hi), hi);
    }
    ss += e * e;
    ++na;
  }
  return na ? sqrtf(ss / (float)na) : 0.f;
}

// ------------------------------------------------------------------------------ one step
// x_t -> x_{t+1} in place on X (every warp calls; ends after a CTA barrier). With TAPE the solver
// tape goes to slot ts and, when D.dump is used (dump_col), the controller activations to the
// dump. X must be complete on entry (a barrier after its last writes).
template <bool TAPE, class Q>
__device__ __forceinline__ void blk_step(const DevTopo& T, const DevPtrs& D, const LaneT<SL>& L, const SL& X, const SL* act,
                                         int t, int ts, uint8_t* ao, float* dump_col, int warp) {
  const SL& S = L.S;
  const int Bp = T.Bp, lane = threadIdx.x & 31;
  const uint32_t mine = blk_mine(warp);
  hinge_kinematics(T, L, X, mine);
  const int u = T.n_layers > 0 ? T.n_layers : 0;
  if (T.ext_ctrl) {
    // wide controller: its output for this step was computed between launches
    const float* ue = D.u_ext + ((size_t)t * Bp + L.i) * T.ext_nop;
    for (int m = warp; m < T.widths[u]; m += blk_nw()) act[u][m] = ue[m];
    cta_sync();
  } else if (T.n_layers > 0) {
    blk_features(T, D, L, X, t, act[0], warp);
    cta_sync();
    if (T.mlp_tc)
      ctrl_forward_blk<Q>(T, D, act[0], act[u], dump_col ? dump_col - lane : nullptr, warp);
    else
      controller_forward_nw(T, D, act, warp);
    cta_sync();
    if (T.n_rec && warp == 0) {  // h^{t+1} = tanh of the last outputs
      const int base = T.widths[u] - T.n_rec;
      for (int k = 0; k < T.n_rec; ++k) S[T.sm_h + k] = tanhf(act[u][base + k]);
    }
    if (D.u_noise) {  // perturbed controller output (harvest of training rows)
      const float* nz = D.u_noise + ((size_t)t * T.B + min(L.i, T.B - 1)) * T.n_motors;  // [T][B][n_motors]
      if (warp == 0)
        for (int m = 0; m < T.n_motors && m < T.widths[u]; ++m) act[u][m] += nz[m];
      cta_sync();
    }
    if (dump_col) {
      const size_t N = (size_t)T.horizon * Bp;
      for (int l = 0; l <= T.n_layers; ++l) {
        if (T.mlp_tc && l > 0 && l < T.n_layers) continue;  // hidden layers went straight to the dump
        for (int k = warp; k < T.widths[l]; k += blk_nw()) dump_col[(size_t)(T.dump_act[l] + k) * N] = act[l][k];
      }
    }
  } else {
    cta_sync();
  }
  servo_targets(T, L, act[u], mine);
  external_impulses(T, L, X, mine);
  TapeStep tp{};
  if (TAPE) {
    tp = tape_step(T, D, ts);
    for (int b = warp; b < T.nb; b += blk_nw())
#pragma unroll
      for (int k = 0; k < 6; ++k) tp.vminus[(6 * b + k) * 32] = X[18 * b + 12 + k];
  }
  cta_sync();
  blk_assemble<true>(T, S, L.P, X, VelX{X}, ao, warp);
  const bool net = D.harvest || (T.ws && T.ws_net);
  if (!T.ws) {
    if (!net)  // (the harvest reads the previous impulses first)
      for (int s = warp; s < T.nslots; s += blk_nw()) S[T.sm_lam + s] = 0.f;
  } else if (!net) {
    blk_damped_start(T, S, warp);
  }
  cta_sync();
  if (net) {
    blk_network_start(T, D, L, X, warp);
    cta_sync();
    if (!T.ws) {
      for (int s = warp; s < T.nslots; s += blk_nw()) S[T.sm_lam + s] = 0.f;
      cta_sync();
    }
  }
  if (T.ws) {
    blk_apply_start(T, S, X, warp);
    if (TAPE)
      for (int s = warp; s < T.nslots; s += blk_nw()) tp.lam0[s * 32] = S[T.sm_lam + s];
  }
  if (TAPE && T.rec_rows)
    for (int s = warp; s < T.nslots; s += blk_nw()) {
      const RowRec r = blk_row(T, S, s);
      const GS R = GS{tp.rows + s * RF_N * 32};
      R.s3(RF_LIN, r.lin); R.s3(RF_ANGA, r.angA); R.s3(RF_ANGB, r.angB); R.s3(RF_IA, r.IA); R.s3(RF_IB, r.IB);
      R[RF_MEFF] = r.meff; R[RF_BIAS] = r.bias; R[RF_BND] = r.bnd;
    }
  blk_stream(T, warp);
  cta_sync();
  blk_sweeps<TAPE, Q::SEQ>(T, S, X, tp, warp);
  if (D.harvest) blk_harvest_finish(T, D, S, warp);
  if (D.resid) {
    if (warp == 0) D.resid[L.i] += blk_residual(T, S, X);
    cta_sync();
  }
  integrate(T, X, mine);
  cta_sync();
}

// Rollouts and steps (see k_forward in dp_steps.cuh for rollout's values) on blocks, one CTA per group of
// 32 instances.
template <bool REC, class Q>
__global__ void __launch_bounds__(32 * Q::NW, 1) k_forward_blk(const __grid_constant__ DevTopo T, const __grid_constant__ DevPtrs D,
                                                        const float* __restrict__ x0, int t0, int nsteps, int rollout) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane;
  const int Bp = T.Bp, B = T.B, nf = 18 * T.nb;
  float* sm = g_smem + lane;
  const LaneT<SL> L{SL{sm}, GC{D.prm + i, Bp}, SL{sm}, i};
  const SL X{sm + T.sm_x * 32};
  SL act[DPK_MAXL + 1];
  for (int l = 0; l <= DPK_MAXL; ++l) act[l] = SL{sm + T.sm_act[l] * 32};
  const bool fresh = rollout == 1 || (rollout == 2 && t0 == 0);
  const float* xs = fresh ? x0 : D.state;
  blk_load(T, D);
  for (int f = warp; f < nf; f += blk_nw()) X[f] = xs[(size_t)f * Bp + i];
  for (int s = warp; s < T.nslots; s += blk_nw()) L.S[T.sm_lam + s] = fresh ? 0.f : D.lam_prev[(size_t)s * Bp + i];
  if (warp == 0)
    for (int k = 0; k < T.n_rec; ++k) L.S[T.sm_h + k] = fresh ? 0.f : D.hrec[(size_t)k * Bp + i];
  cta_sync();
  float loss = (rollout == 2 && !fresh) ? D.loss[i] : 0.f;  // warp 0's copy is the one kept
  if (fresh && T.loss_kind == 3) loss = -dot3(L.P.v3(T.o_loss_target), loss_point(T, L, X));
  const int hz = D.hz[i];
  // a rollout steps the group to the largest horizon among its instances
  const int nrun = rollout ? max(0, min(nsteps, warp_horizon(D, i) - t0)) : nsteps;
  const size_t N = (size_t)T.horizon * Bp;
  for (int k = 0; k < nrun; ++k) {
    const int t = t0 + k;
    if (rollout) {
      if (t % D.ckpt_every == 0) {
        const size_t c = (size_t)(t / D.ckpt_every);
        for (int f = warp; f < nf; f += blk_nw()) D.ckpt[(c * nf + f) * Bp + i] = X[f];
        if (D.ckpt_lam)
          for (int s = warp; s < T.nslots; s += blk_nw()) D.ckpt_lam[(c * T.nslots + s) * Bp + i] = L.S[T.sm_lam + s];
        if (D.ckpt_h && warp == 0)
          for (int q = 0; q < T.n_rec; ++q) D.ckpt_h[(c * T.n_rec + q) * Bp + i] = L.S[T.sm_h + q];
      }
      if (D.traj && i < B)
        for (int f = warp; f < nf; f += blk_nw()) D.traj[((size_t)t * B + i) * nf + f] = X[f];
    }
    // the activity log is per rollout step (rollout parts) or per call step (dp_step)
    uint8_t* ao = (D.active && i < B) ? D.active + ((size_t)(rollout == 2 ? t : k) * B + i) * T.nslots : nullptr;
    blk_step<REC, Q>(T, D, L, X, act, t, t, ao, REC && T.n_layers > 0 && !T.ext_ctrl ? D.dump + (size_t)t * Bp + i : nullptr,
                     warp);
    if (warp == 0) {
      const float w = loss_weight(T, t + 1, hz);
      if (w != 0.f) {
        const float l = loss_value(T, L, X);
        if (Q::SEQ) loss += w * l;
        else loss = __fadd_rn(loss, __fmul_rn(w, l));
      }
    }
  }
  if (rollout && D.traj && i < B)
    for (int f = warp; f < nf; f += blk_nw()) D.traj[((size_t)(t0 + nrun) * B + i) * nf + f] = X[f];
  if (T.ext_ctrl && t0 + nrun < T.horizon) {
    // wide controller: input features of the next step, bf16 for the products, and the
    // activation dump column for the weight gradient
    const int tn = t0 + nrun;
    hinge_kinematics(T, L, X, blk_mine(warp));
    blk_features(T, D, L, X, tn, act[0], warp);
    cta_sync();
    __nv_bfloat16* sx = D.s_ext + (size_t)i * T.ext_k0p;
    for (int q = warp; q < T.ext_k0p; q += blk_nw()) {
      const float v = q < T.widths[0] ? act[0][q] : 0.f;
      sx[q] = __float2bfloat16_rn(v);
      if (REC && q < T.widths[0]) D.dump[(size_t)(T.dump_act[0] + q) * N + (size_t)tn * Bp + i] = v;
    }
  }
  for (int s = warp; s < T.nslots; s += blk_nw()) D.lam_prev[(size_t)s * Bp + i] = L.S[T.sm_lam + s];
  if (warp == 0)
    for (int q = 0; q < T.n_rec; ++q) D.hrec[(size_t)q * Bp + i] = L.S[T.sm_h + q];
  bool bad = false;
  for (int f = warp; f < nf; f += blk_nw()) {
    D.state[(size_t)f * Bp + i] = X[f];
    bad |= !isfinite(X[f]);
  }
  if (warp == 0) {
    bad |= !isfinite(loss);
    if (rollout) D.loss[i] = loss;
  }
  if (bad && i < B) atomicOr(D.status + i, DPK_ST_NAN_STATE);
}

template <bool REC, class Q>
static cudaError_t launch_forward_blk_t(const DevTopo& T, const DevPtrs& D, const float* x0, int t0, int nsteps,
                                        int rollout, cudaStream_t s) {
  const size_t smem = (size_t)T.sm_total * 32 * sizeof(float);
  cudaError_t e = cudaFuncSetAttribute(k_forward_blk<REC, Q>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_forward_blk<REC, Q><<<T.Bp / 32, 32 * T.blk_nw, smem, s>>>(T, D, x0, t0, nsteps, rollout);
  return cudaGetLastError();
}
