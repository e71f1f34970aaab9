// D3Q19 step kernel on pairs of nodes: every thread owns two nodes, neighbours along y, of a
// 32 x TY tile and marches z (FP32 and 16-bit storage; the colour-gradient, Shan-Chen
// multiphase and two-component models; any nx up to 512, any ny and nz, walls).
//
// Same step and densities as the other step kernels (lbm_step.cuh); what differs is the
// work per instruction.  One node per thread, this structure issued 848 (Shan-Chen) to 1403 (colour
// gradient) instructions per node, at 43-58% of the issue slots, with DRAM at 46% of its
// peak: both nodes' FP32 arithmetic runs as packed f32x2 instructions (lbm_vec.cuh), the
// collision is written with the fewest operations (below), and a store address is one
// multiply-add of a constant base and a 32-bit node index.  That is 474 (SC) and 745 (CG)
// instructions per node at 41% and 32% of the issue slots, with DRAM at 56% and 68%: what is left
// above the bytes is the latency of a plane's chain (copy, fields, barrier, neighbours' columns,
// collision, stores) with 16 and 8 warps per SM to hide it.  At 128^3: CG FP32 177 -> 135 us, SC
// FP32 84 -> 65 us, SC FP16 82 -> 57 us; at 256^3 CG FP32 runs at 5.2 TB/s of algorithmic bytes.
//
// Per plane J of a block's sequence, every thread
//   1. reads its two nodes of plane J from the raw plane buffer (a TMA copy of the tile's
//      TY rows and one halo row above and below), forms the component densities and
//      writes the stencil fields into field slot J; one warp, another for every plane,
//      does the same for the two halo rows;
//   2. passes the block barrier; the threads of the tile's first and last column send
//      their fields to the x-neighbours' halo columns in distributed shared memory (a
//      cluster spans a full x-row of tiles, so the periodic wrap in x stays inside it) as
//      asynchronous remote stores that complete on the receiver's mbarrier of slot J;
//   3. collides its nodes of plane J-1 from the sums t_i it kept (CG: both colours'
//      deviations added, since the CG collision acts on the total; SC: the deviations of each component) and
//      the field slots J-2, J-1, J, and pushes the results.  The wait for the neighbours'
//      columns of plane J comes after the part of the collision that does not read them
//      (moments, relaxation rate, in-plane differences): at 128^3 (clusters of 4) 152 ->
//      143 us.
// With EARLY the sums of plane J are kept while staging and the raw buffer is handed back
// after the block barrier, so one buffer per block suffices (CG, two blocks per SM: with
// two buffers and one block of 16 rows 140 us, three blocks and late sums 151 us); otherwise
// they are read again after the collision, which needs fewer registers (SC: 16 warps per
// SM).
//
// Slots and barriers: no thread releases at cluster scope (such a release waits for the
// thread's own stores to reach L2; measured at a third of the step); the remote columns are
// ordered by the mbarrier's transaction count.  Field slot J (last read by the collision
// of plane J-3, in iteration J-2) is written locally after the block barrier of iteration
// J-1, and remotely by a neighbour only after that neighbour has received this block's
// columns of plane J-1, which are sent after this block's barrier of iteration J-1: four
// slots.  Every wait is bounded (lbm_step_tma.cuh).
#pragma once

#include "lbm_rules.h"
#include "lbm_step_tma.cuh"
#include "lbm_vec.cuh"

namespace lbm {

// Per-component densities of both nodes (CompState; in FP32 the density is the reference q).
struct Comp2 {
  F2 q, dq, d;
};
template <class L>
__device__ __forceinline__ Comp2 comp_state2(const F2* g, const F2& r_old) {
  Comp2 c;
  const F2 delta = tree_sum2<L::Q>(g);
  c.q = two_sum2(r_old, delta, c.dq);
  c.d = c.dq - delta;
  return c;
}

// Reciprocal by one Newton-Raphson step, x (2 - a x), from rcp.approx (relative error below 2^-22):
// within 0.501 ulp for 2^-126 <= |a| <= 2^126, which holds for the densities, viscosities and
// gradients it is taken of; NaN for 0 and for infinities, which a collision does not survive
// either way.  Six calls for a pair of nodes: with __frcp_rn in its place 101 x 75 x 67 CG FP32 takes
// 57.0 us instead of 51.4 and 128^3 with 15% walls 225 instead of 208; 128^3 without walls is level.
__device__ __forceinline__ float rcp_newton(float a) {
  float x;
  asm("rcp.approx.f32 %0, %1;" : "=f"(x) : "f"(a));
  return fmaf(fmaf(-a, x, 1.f), x, x);
}

// c_q . a for the positive member of pair q (its first non-zero component is +1)
template <class L>
__device__ __forceinline__ F2 dot2(int q, const F2 (&a)[3]) {
  const int c[3] = {L::pcx(q), L::pcy(q), L::pcz(q)};
  F2 r;
  bool first = true;
#pragma unroll
  for (int k = 0; k < 3; k++) {
    if (c[k] == 0) continue;
    r = first ? a[k] : (c[k] > 0 ? r + a[k] : r - a[k]);
    first = false;
  }
  return r;
}

// sum_q c_q d_q over the opposite pairs; axis pairs (ax) and diagonal pairs (dg) apart, as
// they carry different weights
template <class L>
struct PairSum {
  F2 ax[3], dg[3];
  bool has[3] = {false, false, false};
  __device__ __forceinline__ PairSum() {}
  __device__ __forceinline__ void add(int q, const F2& d) {
    const int c[3] = {L::pcx(q), L::pcy(q), L::pcz(q)};
#pragma unroll
    for (int k = 0; k < 3; k++) {
      if (c[k] == 0) continue;
      if (L::pgrp(q) == 1) {
        ax[k] = d;
      } else {
        dg[k] = !has[k] ? (c[k] > 0 ? d : F2(0.f) - d) : (c[k] > 0 ? dg[k] + d : dg[k] - d);
        has[k] = true;
      }
    }
  }
};

// CG collision (the equations of cg_collide, lbm_step.cuh) of a thread's two nodes.  t[i]:
// sums g^R_i + g^B_i of the stored deviations; nb(f, i, j): field f (0 q_R, 1 q_B, 2 rho^N,
// 3 rho) at neighbour i of node j, the plane above only after ready(); emit(i, g^R_i,
// g^B_i) takes the results.  The total post-collision population of a pair (i, j = opp(i))
// is formed as (1 - omega) t + E +- O with the even and odd parts E = K0 + cu (K1 cu + K2
// c.grad rho) + K3 (c.grad rho^N)^2 and O = K4 cu, whose group constants K hold the relaxed
// equilibrium (Eqs. BGK, equiliCG), the perturbation (Eq. perturbationOp) and the change of
// reference, with S0, S1 the Guo source (Eq. source) of a body force.
// REP: the nodes' repulsion forces fr come on top of the body force.
template <class L, bool REP, class NB, class READY, class EMIT>
__device__ __forceinline__ void cg_collide_pair(const StepParams<float>& p, const F2 (&t)[L::Q], const Comp2& cr,
                                                const Comp2& cb, const F2 (&fr)[3], const NB& nb, const READY& ready,
                                                const EMIT& emit) {
  const F2 qR = cr.q, qB = cb.q;
  PairSum<L> sj;
#pragma unroll
  for (int q = 0; q < L::NP; q++) sj.add(q, t[2 * q + 1] - t[2 * q + 2]);
  auto rcp = [](float a) { return rcp_newton(a); };
  const F2 rho = qR + qB;
  const F2 inv = each(rho, rcp);
  F2 u[3], F[3];
  bool forced = p.has_body;
  if constexpr (REP) {  // away from interfaces every force of the warp is 0
    const bool any = fr[0][0] != 0.f || fr[0][1] != 0.f || fr[1][0] != 0.f || fr[1][1] != 0.f || fr[2][0] != 0.f ||
                     fr[2][1] != 0.f;
    forced = forced || __any_sync(0xffffffffu, any);
  }
#pragma unroll
  for (int k = 0; k < 3; k++) {
    F2 jm = k < L::D ? sj.ax[k] + sj.dg[k] : F2(0.f);
    F[k] = F2(p.body[k]);
    if constexpr (REP) F[k] = F[k] + fr[k];
    if (forced) jm = REP ? fma(F2(0.5f), F[k], jm) : jm + F2(0.5f * p.body[k]);
    u[k] = jm * inv;
  }
  const F2 sv = fma(qR, F2(p.inv_nu_r), qB * F2(p.inv_nu_b));
  const F2 nubar = rho * each(sv, rcp);
  const F2 omega = F2(2.f) * each(fma(F2(6.f), nubar, F2(1.f)), rcp);
  const F2 om1 = F2(1.f) - omega;
  const F2 en = p.enhanced ? nubar : F2(0.f);
  PairSum<L> sr, sn;
  auto grads = [&](bool inplane) {
#pragma unroll
    for (int q = 0; q < L::NP; q++) {
      if ((L::pcz(q) == 0) != inplane) continue;
      F2 dr, dn;
#pragma unroll
      for (int j = 0; j < 2; j++) {
        const int i1 = 2 * q + 1, i2 = 2 * q + 2;
        dr.set(j, nb(3, i1, j) - nb(3, i2, j));
        dn.set(j, nb(2, i1, j) - nb(2, i2, j));
      }
      sr.add(q, dr);
      sn.add(q, dn);
    }
  };
  grads(true);
  ready();
  grads(false);
  F2 gr[3], gn[3];
#pragma unroll
  for (int k = 0; k < 3; k++) {
    if (k < L::D) {
      const float w1 = float(3.0 * L::w(1)), w2 = float(3.0 * L::w(2));
      gr[k] = fma(F2(w2), sr.dg[k], F2(w1) * sr.ax[k]);
      gn[k] = fma(F2(w2), sn.dg[k], F2(w1) * sn.ax[k]);
    } else {
      gr[k] = gn[k] = F2(0.f);
    }
  }
  const F2 uu = fma(u[0], u[0], fma(u[1], u[1], u[2] * u[2]));
  const F2 ugr = fma(u[0], gr[0], fma(u[1], gr[1], u[2] * gr[2]));
  const F2 gg = fma(gn[0], gn[0], fma(gn[1], gn[1], gn[2] * gn[2]));
  const F2 gabs = each(gg, [](float a) { return sqrtf(a); });
  const float eps = p.grad_eps;
  const F2 inv_g = each(gabs, [&](float a) { return a > eps ? rcp_newton(a) : 0.f; });
  const F2 Ag = each(gabs, [&](float a) { return a > eps ? p.A * a : 0.f; });
  const F2 cR = qR * inv;
  const F2 qRB = cR * qB;
  const F2 rec = F2(p.beta) * qRB * inv;
  const F2 wrho = omega * rho;
  const F2 kg = fma(F2(-0.5f), omega, F2(1.f));
  const F2 uF = fma(u[0], F[0], fma(u[1], F[1], u[2] * F[2]));
  F2 K0[3], K1[3], K2[3], K3[3], K4[3], base[3], rcg[3], S0[3], S1[3];
  const F2 pe = Ag * inv_g * inv_g;
  // 3 w_i and 3/2 w_i in FP32 with the sums over the directions that conserve momentum (3 w_1
  // * 2 + 3 w_2 * 8 = 1) and mass (to 3/2) exactly.  Rounded to nearest, 3 w_i gains 3e-8 of
  // the momentum every step, the same way at every node.
  const float w3[3] = {1.f, 11184810.f / 67108864.f, 11184811.f / 134217728.f};
  const float w32[3] = {16777215.f / 33554432.f, 11184811.f / 134217728.f, 11184811.f / 268435456.f};
#pragma unroll
  for (int g = 0; g <= 2; g++) {
    const float wg = float(L::w(g)), phR = p.phi[0][g], phB = p.phi[1][g];
    // (1 - omega) k_g + omega (phi dq + psi en u.grad - 3/2 w rho uu) - A|grad| B
    const F2 kgs = fma(F2(phR), cr.d, F2(phB) * cb.d);
    F2 e = fma(F2(phR), cr.dq, F2(phB) * cb.dq);
    e = fma(F2(float(L::psi(g))) * en, ugr, e);
    e = fma(F2(-w32[g]) * rho, uu, e);
    K0[g] = fma(om1, kgs, fma(omega, e, F2(float(-L::B(g))) * Ag));
    if (forced) K0[g] = fma(F2(-3.f * wg) * kg, uF, K0[g]);
    if (g > 0) {
      K1[g] = F2(4.5f * wg) * wrho;
      K2[g] = F2(float(2.0 * L::xi(g))) * (omega * en);
      K3[g] = F2(wg) * pe;
      K4[g] = F2(w3[g]) * wrho;
      rcg[g] = rec * fma(qR, F2(phR), qB * F2(phB)) * inv_g * F2(g == 1 ? 1.f : 0.70710678118654752440f);
      S0[g] = F2(9.f * wg) * kg;
      S1[g] = F2(w3[g]) * kg;
    }
  }
  // (rho_R phi^B q_B - rho_B phi^R q_R) / rho with q = rho.  The rest direction takes what
  // makes the sum over the directions vanish: the rounded constants' own sum is off by up to
  // 3e-8, the same way at every node and step, and would move that much of one colour to the
  // other (velocity error after 40 steps 1.9e-6, against 8e-7).
  base[1] = qRB * F2(p.phi[1][1] - p.phi[0][1]);
  base[2] = qRB * F2(p.phi[1][2] - p.phi[0][2]);
  base[0] = fma(F2(-12.f), base[2], F2(-6.f) * base[1]);
  {
    const F2 Gs = fma(om1, t[0], K0[0]);
    const F2 gR = fma(cR, Gs, base[0]);
    emit(0, gR, Gs - gR);
  }
  auto pairs = [&](auto with_force) {
    constexpr bool FORCE = decltype(with_force)::value;
#pragma unroll
    for (int q = 0; q < L::NP; q++) {
      const int g = L::pgrp(q);
      const F2 cu = dot2<L>(q, u), cg = dot2<L>(q, gr), cn = dot2<L>(q, gn);
      F2 E = fma(cu, fma(K2[g], cg, K1[g] * cu), K0[g]);
      E = fma(K3[g] * cn, cn, E);
      F2 O = K4[g] * cu;
      if constexpr (FORCE) {
        const F2 cF = dot2<L>(q, F);
        E = fma(S0[g] * cu, cF, E);
        O = fma(S1[g], cF, O);
      }
      const F2 Gi = fma(om1, t[2 * q + 1], E + O);
      const F2 Gj = fma(om1, t[2 * q + 2], E - O);
      const F2 rc = rcg[g] * cn;
      const F2 Ri = fma(cR, Gi, base[g] + rc);
      const F2 Rj = fma(cR, Gj, base[g] - rc);
      emit(2 * q + 1, Ri, Gi - Ri);
      emit(2 * q + 2, Rj, Gj - Rj);
    }
  };
  if (forced)
    pairs(std::true_type{});
  else
    pairs(std::false_type{});
}

// SC multiphase collision (Eqs. interactionforceMP, collisSC, equiliSC, guoforce2, source) of
// a thread's two nodes; nb(f, i, j): field 0 psi, 1 q.  With a = 3 omega rho u + 3 k F and
// b = 4.5 omega rho u + 9 k F (k = 1 - omega/2) a pair's results are
// (1 - omega) t + w [K0 + (c.u)(c.b) +- c.a].
template <class L, class NB, class READY, class EMIT>
__device__ __forceinline__ void scmp_collide_pair(const StepParams<float>& p, const F2 (&t)[L::Q], const Comp2& c,
                                                  const F2& psic, const NB& nb, const READY& ready, const EMIT& emit) {
  PairSum<L> sp, sj;
#pragma unroll
  for (int q = 0; q < L::NP; q++) sj.add(q, t[2 * q + 1] - t[2 * q + 2]);
  auto psis = [&](bool inplane) {
#pragma unroll
    for (int q = 0; q < L::NP; q++) {
      if ((L::pcz(q) == 0) != inplane) continue;
      F2 d;
#pragma unroll
      for (int j = 0; j < 2; j++) d.set(j, nb(0, 2 * q + 1, j) - nb(0, 2 * q + 2, j));
      sp.add(q, d);
    }
  };
  psis(true);
  ready();
  psis(false);
  const F2 inv = each(c.q, [](float a) { return rcp_newton(a); });
  const F2 gp = F2(-p.G) * psic;
  const float omega = p.omega_r, kg = 1.f - 0.5f * omega;
  const F2 om1 = F2(1.f - omega);
  F2 u[3], F[3], av[3], bv[3];
#pragma unroll
  for (int k = 0; k < 3; k++) {
    F[k] = F2(p.has_body ? p.body[k] : 0.f);
    F2 jm = F2(0.f);
    if (k < L::D) {
      F[k] = fma(gp, fma(F2(float(L::w(2))), sp.dg[k], F2(float(L::w(1))) * sp.ax[k]), F[k]);
      jm = sj.ax[k] + sj.dg[k];
    }
    u[k] = fma(F2(0.5f), F[k], jm) * inv;
  }
  const F2 uu = fma(u[0], u[0], fma(u[1], u[1], u[2] * u[2]));
  const F2 uF = fma(u[0], F[0], fma(u[1], F[1], u[2] * F[2]));
  const F2 wr = F2(omega) * c.q;
#pragma unroll
  for (int k = 0; k < 3; k++) {
    av[k] = fma(F2(3.f) * wr, u[k], F2(3.f * kg) * F[k]);
    bv[k] = fma(F2(4.5f) * wr, u[k], F2(9.f * kg) * F[k]);
  }
  F2 K0 = fma(om1, c.d, F2(omega) * c.dq);
  K0 = fma(F2(-1.5f) * wr, uu, K0);
  K0 = fma(F2(-3.f * kg), uF, K0);
  emit(0, fma(om1, t[0], F2(float(L::w(0))) * K0));
#pragma unroll
  for (int q = 0; q < L::NP; q++) {
    const F2 wg = F2(float(L::w(L::pgrp(q))));
    const F2 cu = dot2<L>(q, u), ca = dot2<L>(q, av), cbv = dot2<L>(q, bv);
    const F2 E = fma(cu, cbv, K0);
    emit(2 * q + 1, fma(wg, E + ca, om1 * t[2 * q + 1]));
    emit(2 * q + 2, fma(wg, E - ca, om1 * t[2 * q + 2]));
  }
}

// Two-component SC collision (Eqs. doublebeltrepulsionforce2, guoforce2, collisSC, equiliSC,
// source) of a thread's two nodes; t[0..Q) and t[Q..2Q): the components' deviations; nb(f,
// i, j): field f = q_1, q_2; per component as in scmp_collide_pair, with the common velocity.
template <class L, class NB, class READY, class EMIT>
__device__ __forceinline__ void sc2c_collide_pair(const StepParams<float>& p, const F2 (&t)[2 * L::Q],
                                                  const Comp2 (&c)[2], const NB& nb, const READY& ready,
                                                  const EMIT& emit) {
  constexpr int Q = L::Q;
  PairSum<L> s1, s2, sj;
#pragma unroll
  for (int q = 0; q < L::NP; q++)
    sj.add(q, (t[2 * q + 1] - t[2 * q + 2]) + (t[Q + 2 * q + 1] - t[Q + 2 * q + 2]));
  auto diffs = [&](bool inplane) {
#pragma unroll
    for (int q = 0; q < L::NP; q++) {
      if ((L::pcz(q) == 0) != inplane) continue;
      F2 d1, d2;
#pragma unroll
      for (int j = 0; j < 2; j++) {
        d1.set(j, nb(0, 2 * q + 1, j) - nb(0, 2 * q + 2, j));
        d2.set(j, nb(1, 2 * q + 1, j) - nb(1, 2 * q + 2, j));
      }
      s1.add(q, d1);
      s2.add(q, d2);
    }
  };
  diffs(true);
  ready();
  diffs(false);
  const F2 inv = each(c[0].q + c[1].q, [](float a) { return rcp_newton(a); });
  F2 u[3], F[2][3];
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const F2 w1 = F2(float(L::w(1))), w2 = F2(float(L::w(2)));
    F[0][k] = F2(-p.G) * c[0].q * fma(w2, s2.dg[k], w1 * s2.ax[k]);
    F[1][k] = F2(-p.G) * c[1].q * fma(w2, s1.dg[k], w1 * s1.ax[k]);
    if (p.has_body) {
      const F2 b = F2(p.body[k]) * inv;
      F[0][k] = fma(b, c[0].q, F[0][k]);
      F[1][k] = fma(b, c[1].q, F[1][k]);
    }
    u[k] = fma(F2(0.5f), F[0][k] + F[1][k], sj.ax[k] + sj.dg[k]) * inv;
  }
  const F2 uu = fma(u[0], u[0], fma(u[1], u[1], u[2] * u[2]));
#pragma unroll
  for (int s = 0; s < 2; s++) {
    const float omega = s == 0 ? p.omega_r : p.omega_b, kg = 1.f - 0.5f * omega;
    const F2 om1 = F2(1.f - omega), wr = F2(omega) * c[s].q;
    const F2 uF = fma(u[0], F[s][0], fma(u[1], F[s][1], u[2] * F[s][2]));
    F2 av[3], bv[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
      av[k] = fma(F2(3.f) * wr, u[k], F2(3.f * kg) * F[s][k]);
      bv[k] = fma(F2(4.5f) * wr, u[k], F2(9.f * kg) * F[s][k]);
    }
    F2 K0 = fma(om1, c[s].d, F2(omega) * c[s].dq);
    K0 = fma(F2(-1.5f) * wr, uu, K0);
    K0 = fma(F2(-3.f * kg), uF, K0);
    emit(s, 0, fma(om1, t[s * Q], F2(float(L::w(0))) * K0));
#pragma unroll
    for (int q = 0; q < L::NP; q++) {
      const F2 wg = F2(float(L::w(L::pgrp(q))));
      const F2 cu = dot2<L>(q, u), ca = dot2<L>(q, av), cb = dot2<L>(q, bv);
      const F2 E = fma(cu, cb, K0);
      emit(s, 2 * q + 1, fma(wg, E + ca, om1 * t[s * Q + 2 * q + 1]));
      emit(s, 2 * q + 2, fma(wg, E - ca, om1 * t[s * Q + 2 * q + 2]));
    }
  }
}

template <int MODEL>
struct PairTraits;
template <>
struct PairTraits<kCG> {
  // q_R, q_B, rho^N, and their sum rho: the gradient reads rho 18 times per node, which as
  // q_R + q_B would take two loads and an addition each
  static constexpr int NV = 4;
  static constexpr int NH = 1;  // held values per direction: the colours' sum
  static constexpr bool EARLY = true;
};
template <>
struct PairTraits<kSCMP> {
  static constexpr int NV = 2;  // psi, q
  static constexpr int NH = 1;
  static constexpr bool EARLY = false;
};
template <>
struct PairTraits<kSC2C> {
  static constexpr int NV = 2;  // q_1, q_2
  static constexpr int NH = 2;
  static constexpr bool EARLY = false;
};

// The planes a cluster stages: the lattice's (tile row, plane) pairs, tile row by tile row,
// are cut into nblk runs of equal length; a run is split where it passes into the next tile
// row, and every piece [z0, z1) is staged with its two halo planes (which are not
// collided).  Equal runs keep every cluster busy to the end whatever the lattice (128^3
// with 110 resident clusters: 208 units of 9.8 planes took two rounds, 155 us; runs of 18.6
// planes 138 us), and neighbouring tile rows are still marched within a few planes of each
// other, so that their shared rows hit L2.
struct PlaneRun {
  long long next, end;  // positions tile row * nz + z
  int nz, z;
  Segment sg;
  bool valid;
  __device__ PlaneRun(long long begin, long long end_, int nz_) : next(begin), end(end_), nz(nz_) { pop(); }
  __device__ void pop() {
    valid = next < end;
    if (!valid) return;
    sg.col = (int)(next / nz);
    sg.z0 = (int)(next - (long long)sg.col * nz);
    const long long stop = min(end, (long long)(sg.col + 1) * nz);
    sg.z1 = sg.z0 + (int)(stop - next);
    next = stop;
    z = sg.z0 - 1;
  }
  __device__ void advance() {
    if (++z > sg.z1) pop();
  }
  __device__ bool last() const { return z == sg.z1 && next >= end; }
};

__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// shared::cluster address of the same shared-memory offset in block `rank` of the cluster
__device__ __forceinline__ uint32_t mapa_shared(uint32_t addr, uint32_t rank) {
  uint32_t d;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(addr), "r"(rank));
  return d;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile(
      "barrier.cluster.arrive.release.aligned;\n\t"
      "barrier.cluster.wait.acquire.aligned;" ::
          : "memory");
}
// Asynchronous 32-bit store into another block's shared memory (addresses from mapa);
// completion is counted, in bytes, on that block's mbarrier `bar`.
__device__ __forceinline__ void st_async_f32(uint32_t cluster_addr, float v, uint32_t cluster_bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(cluster_addr),
               "r"(__float_as_uint(v)), "r"(cluster_bar)
               : "memory");
}

constexpr int kPairFields = 4;       // field slots
constexpr int kPairHeader = 128;     // mbarriers, then 128-byte aligned plane buffers

template <class L, class S, class RT, int MODEL, int TY>
__host__ __device__ constexpr size_t pair_smem_bytes(int raw) {
  using Lay = TmaLayout<L, S, RT, MODEL, kPairTX, TY>;
  return kPairHeader + size_t(raw) * Lay::BUF_MAIN + size_t(kPairFields) * PairTraits<MODEL>::NV * Lay::NE * 4;
}
// Raw plane buffers: as many (1 to 3) as the block's share of the SM's 228 KB holds.
template <class L, class S, class RT, int MODEL, int TY, int MB>
__host__ __device__ constexpr int pair_raw() {
  constexpr size_t budget = MB == 1 ? 232448 : 233472 / MB - 1024;
  return pair_smem_bytes<L, S, RT, MODEL, TY>(3) <= budget   ? 3
         : pair_smem_bytes<L, S, RT, MODEL, TY>(2) <= budget ? 2
                                                             : 1;
}

// Destination arrays of a step.  As kernel constants they make a store address one
// multiply-add (base + index), where an array base computed in the kernel costs three more
// integer instructions per store.
template <class S, class RT, int KQ, int K>
struct OutArrays {
  S* f[KQ];
  RT* r[K];
};

// Walls: a 64-bit word for every row of a tile, (z * ny + y) * tiles + tile.  Bit b: column
// x0 - 1 + b (periodic) is a wall, b = 0 to the tile's width + 1; kWallAny: there is one within
// rows y - 1 to y + 2 of planes z - 1 to z + 1, all that the nodes of rows y and y + 1 can see.
constexpr unsigned long long kWallAny = 1ULL << 63;
// A walled lattice runs two collisions: where a plane of a tile row has walls in sight of any of
// its nodes, the whole row of tiles (a cluster) takes the one that looks at them, which is half as
// long again: 128^3 CG FP32 134 us without walls, 149 between two planes, 208 with 15% of the
// nodes solid at random (SC FP32 65, 75, 101).  One collision for all nodes takes 163 between two
// planes; a choice by warp 169 and, with single columns of walls, 282 against 195: both
// collisions together do not fit the instruction cache.  So clusters whose runs are shorter than
// kShortRun planes, and would change over every few of them, take the walled one throughout (64^3
// CG FP32 31.5 -> 26.5; the smaller SC code gains at the shortest runs only).
// Runs are cut by cost: entry g of ncuts + 1 cuts is the (tile row, plane) position before which the
// share g / ncuts of the work lies, a plane counting kWallCost or kPlainCost.
constexpr int kPlainCost = 2, kWallCost = 3, kMaxCuts = 16384;
constexpr int kShortRun = 16, kShortRunSC = 2;

// Forms of the kernel: every tile full (nx % 32 == 0, ny % TY == 0); any size; any size with
// walls.  The tests for partial tiles cost the full ones 4% (CG 128^3 FP32) to 16% (FP16).
enum PairForm : int { kFull = 0, kRagged = 1, kWalls = 2 };

// Launch: cluster dims (C, 1, 1) with C = p.ncx = ceil(nx / 32) <= kPairMaxCluster; grid =
// p.nblk clusters * C blocks of 16 TY threads, MB blocks per SM; p.ncol = ceil(ny / TY) tile
// rows.  Rows are p.px nodes apart (a multiple of 16 bytes, which a tensor map needs), the
// last tile of a row or column may be partial.  Every index within an array fits 31 bits.
// REP (colour gradient): the repulsion force rep [3][n] of lbm_rep.cuh is added.
// With walls (kWalls) a wall neighbour's stencil values are the centre's, and what would be
// pushed into it comes back (halfway bounce-back).
template <class L, class T, class S, class RT, int MODEL, int FORM, int TY, int MB, bool REP = false>
__global__ void __launch_bounds__(16 * TY, MB)
    step_kernel_pair(const __grid_constant__ TmaMaps maps,
                     const __grid_constant__ OutArrays<S, RT, ModelTraits<MODEL>::K * L::Q, ModelTraits<MODEL>::K> out,
                     const unsigned long long* __restrict__ walls, const uint8_t* __restrict__ rows_walled,
                     const int* __restrict__ cuts, const T* __restrict__ rep, int* __restrict__ status,
                     const __grid_constant__ StepParams<T> p) {
  static_assert(sizeof(T) == 4 && sizeof(RT) == 4, "fields are exchanged as 32-bit words");
  static_assert(TY == 8 || TY == 16, "tile rows with a tensor map");
  constexpr int TX = kPairTX, kWarps = TY / 2;
  constexpr int RAW = pair_raw<L, S, RT, MODEL, TY, MB>();
  constexpr bool EARLY = PairTraits<MODEL>::EARLY;
  static_assert(EARLY || RAW >= 2, "late sums keep a plane's buffer through the next copy");
  using Lay = TmaLayout<L, S, RT, MODEL, TX, TY>;
  constexpr int Q = L::Q, K = Lay::K;
  constexpr int NV = PairTraits<MODEL>::NV, NH = PairTraits<MODEL>::NH;
  constexpr int EX = Lay::EX, NE = Lay::NE;
  constexpr int FS = kPairFields;
  extern __shared__ __align__(128) unsigned char smem[];
  uint64_t* raw_full = reinterpret_cast<uint64_t*>(smem);     // [RAW]
  uint64_t* fld_full = raw_full + RAW;                         // [FS]: the neighbours' columns
  unsigned char* bufs = smem + kPairHeader;                    // [RAW][BUF_MAIN]
  float* fld = reinterpret_cast<float*>(bufs + RAW * Lay::BUF_MAIN);  // [FS][NV][NE]

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int C = p.ncx;
  const uint32_t rank = cluster_ctarank();
  const uint32_t left = (rank + C - 1) % C, right = (rank + 1) % C;
  const int x0 = (int)rank * TX;
  constexpr bool FULL = FORM == kFull, WALLS = FORM == kWalls;
  const int width = FULL ? TX : min(TX, p.nx - x0);                                // columns of this tile
  const int left_width = FULL || rank != 0 ? TX : p.nx - (C - 1) * TX;  // and of the left neighbour's
  const int cid = blockIdx.x / C;
  const int plane_n = p.px * p.ny;

  if (tid == 0) {
    for (int s = 0; s < RAW; s++) mbar_init(&raw_full[s], 1);
    for (int s = 0; s < FS; s++) mbar_init(&fld_full[s], 1);  // the expect-tx arrival
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  cluster_sync_all();  // barriers of every block initialised before any remote store
  await_previous_step();
  // A blown-up (or timed-out) state stops stepping; the cluster barriers are still passed.
  const bool skip = *status != 0;
  // copy destinations must be 128-byte aligned; a misaligned base stops the work (every
  // block of the cluster sees the same offset) but not the barriers
  const bool layout_ok = (smem_addr(bufs) & 127u) == 0;
  if (!layout_ok && tid == 0) atomicOr(status, kStatusLayout);
  bool alive = !skip && layout_ok;
  auto wait = [&](uint64_t* bar, int phase) {  // one decision per warp
    if (!__all_sync(0xffffffffu, mbar_wait_bounded(bar, phase & 1))) {
      if (lane == 0) atomicOr(status, kStatusTimeout);
      alive = false;
    }
  };

  // TMA copy of one plane into raw buffer s: top halo row, TY rows, bottom halo row
  auto issue = [&](const PlaneRun& pr, int s) {
    const int y0 = pr.sg.col * TY;
    const int yt = y0 == 0 ? p.ny - 1 : y0 - 1, yb = y0 + TY >= p.ny ? 0 : y0 + TY;
    const int gz = wrap(pr.z, p.nz);
    unsigned char* b = bufs + s * Lay::BUF_MAIN;
    uint64_t* bar = &raw_full[s];
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    mbar_arrive_expect_tx(bar, Lay::TX_BYTES);
#pragma unroll
    for (int g = 0; g < 3; g++) {
      const bool mid = g == 1;
      const int y = g == 0 ? yt : (g == 1 ? y0 : yb);
      const CUtensorMap* pop = mid ? (TY == 16 ? &maps.pop_main_mid16 : &maps.pop_main_mid) : &maps.pop_main_row;
      const CUtensorMap* ref = mid ? (TY == 16 ? &maps.ref_main_mid16 : &maps.ref_main_mid) : &maps.ref_main_row;
      tma_load_4d(b + Lay::PM::group(g), pop, x0, 0, y, gz, bar);
      tma_load_4d(b + Lay::OFF_RM + Lay::RMR::group(g), ref, x0, 0, y, gz, bar);
    }
  };

  const long long total = (long long)p.ncol * p.nz;
  // with walls and short runs, every plane takes the walled collision (kShortRun)
  [[maybe_unused]] const bool one_form = total < (MODEL == kSCMP ? kShortRunSC : kShortRun) * (long long)p.nblk;
  auto cut = [&](int b) -> long long {  // where run b begins
    if constexpr (WALLS)
      if (!one_form) return cuts[(long long)b * p.ncuts / p.nblk];
    return total * b / p.nblk;
  };
  const long long begin = cut(cid), end = cut(cid + 1);
  PlaneRun ahead(begin, end, p.nz);  // the next plane to copy
  PlaneRun cur(begin, end, p.nz);    // the plane being staged
  int issued = 0;                              // planes whose copy was issued
  auto issue_next = [&]() {
    if (tid == 0 && alive && ahead.valid) {
      issue(ahead, issued % RAW);
      issued++;
    }
    ahead.advance();
  };
  for (int j = 0; j < (EARLY ? RAW : RAW - 1); j++) issue_next();

  // state of the plane staged last, collided one plane later
  F2 hold[NH * Q], next_hold[EARLY ? Q : 1];
  Comp2 hcs[K];
  int prev_z = 0, prev_y0 = 0;
  int near[2] = {0, 0};
  [[maybe_unused]] bool walled = false;
  bool prev_interior = false;

  for (int J = 0; cur.valid; J++) {
    const int y0 = cur.sg.col * TY;
    const int z = cur.z;
    const bool interior = z >= cur.sg.z0 && z < cur.sg.z1;  // plane J is collided in iteration J+1
    if (!REP && p.admit_early && cur.last()) admit_next_step();
    const int fs = J % FS;
    const unsigned char* b = bufs + (J % RAW) * Lay::BUF_MAIN;
    const int halo_warp = J % kWarps;  // stages the halo rows too
    const int rows = FULL ? TY : min(TY, p.ny - y0);
    Comp2 cs[K];
    // 1: the node is a wall or outside the lattice; otherwise bit i: its neighbour i is a wall
    int next_near[2] = {0, 0};
    [[maybe_unused]] bool next_walled = false;
    if constexpr (WALLS) {
      const int gy = y0 + 2 * warp;
      next_walled = interior && rows_walled[cur.sg.col * p.nz + z] != 0;
      if (next_walled && gy < p.ny) {
        auto word = [&](int y, int zz) { return walls[unsigned(zz * p.ny + y) * unsigned(C) + rank]; };
        if (word(gy, z) & kWallAny) {
          unsigned v[3][4];  // columns x-1 .. x+1 of planes z-1 .. z+1, rows gy-1 .. gy+2
#pragma unroll
          for (int r = 0; r < 4; r++) {
            const int y = gy - 1 + r, yw = y < 0 ? p.ny - 1 : y < p.ny ? y : min(y - p.ny, p.ny - 1);
            v[0][r] = unsigned(word(yw, z == 0 ? p.nz - 1 : z - 1) >> lane);
            v[1][r] = unsigned(word(yw, z) >> lane);
            v[2][r] = unsigned(word(yw, z + 1 >= p.nz ? 0 : z + 1) >> lane);
          }
#pragma unroll
          for (int j = 0; j < 2; j++)
#pragma unroll
            for (int i = 0; i < Q; i++)
              next_near[j] |= int((v[cz<L>(i) + 1][cy<L>(i) + 1 + j] >> (cx<L>(i) + 1)) & 1u) << i;
        }
      }
    }
    if constexpr (!FULL) {
#pragma unroll
      for (int j = 0; j < 2; j++)
        if (lane >= width || y0 + 2 * warp + j >= p.ny || (next_near[j] & 1)) next_near[j] = 1;
    }
    // ---- stage plane J ----
    if (alive) wait(&raw_full[J % RAW], J / RAW);
    // bytes of the two halo columns (rows + 2 rows, NV fields) the x-neighbours send
    if (alive && tid == 0) mbar_arrive_expect_tx(&fld_full[fs], 2u * (rows + 2) * NV * 4u);
    if (alive) {
      // densities and fields of the raw rows ey0, ey1, into field rows fy0, fy1 (negative:
      // none); the sums too when `own`
      auto stage_rows = [&](int ey0, int ey1, int fy0, int fy1, bool own, Comp2 (&c)[K]) {
        const S* p0 = reinterpret_cast<const S*>(b + Lay::PM::row(ey0)) + lane;
        const S* p1 = reinterpret_cast<const S*>(b + Lay::PM::row(ey1)) + lane;
        const RT* r0 = reinterpret_cast<const RT*>(b + Lay::OFF_RM + Lay::RMR::row(ey0)) + lane;
        const RT* r1 = reinterpret_cast<const RT*>(b + Lay::OFF_RM + Lay::RMR::row(ey1)) + lane;
#pragma unroll
        for (int k = 0; k < K; k++) {
          F2 g[Q], r;
#pragma unroll
          for (int i = 0; i < Q; i++) {
            g[i].set(0, ld_s<S, T>(p0[(k * Q + i) * TX]));
            g[i].set(1, ld_s<S, T>(p1[(k * Q + i) * TX]));
          }
          r.set(0, r0[k * TX]);
          r.set(1, r1[k * TX]);
          c[k] = comp_state2<L>(g, r);
          if (EARLY && own) {
#pragma unroll
            for (int i = 0; i < Q; i++) next_hold[i] = k == 0 ? g[i] : next_hold[i] + g[i];
          }
        }
        float* f = fld + fs * NV * NE + lane + 1;
#pragma unroll
        for (int j = 0; j < 2; j++) {
          const int fy = j == 0 ? fy0 : fy1, e = fy * EX;
          if (!FULL && (fy < 0 || lane >= width)) continue;
          float fields[2];
          node_fields<MODEL, float>(p, c[0].q[j], K == 2 ? c[K - 1].q[j] : 0.f, fields);
          if constexpr (MODEL == kCG) {
            f[e] = c[0].q[j];
            f[NE + e] = c[1].q[j];
            f[2 * NE + e] = fields[1];
            f[3 * NE + e] = fields[0];
          } else if constexpr (MODEL == kSC2C) {
            f[e] = c[0].q[j];
            f[NE + e] = c[1].q[j];
          } else {
            f[e] = fields[0];
            f[NE + e] = c[0].q[j];
          }
        }
      };
      if (FULL || 2 * warp < rows)
        stage_rows(2 * warp + 1, 2 * warp + 2, 2 * warp + 1, FULL || 2 * warp + 1 < rows ? 2 * warp + 2 : -1, true, cs);
      if (warp == halo_warp) {
        Comp2 unused[K];
        stage_rows(0, TY + 1, 0, rows + 1, false, unused);
      }
    }
    // repulsion forces of the nodes collided below, on their way during the barrier
    [[maybe_unused]] F2 fr[3];
    if constexpr (REP) {
#pragma unroll
      for (int k = 0; k < 3; k++)
#pragma unroll
        for (int j = 0; j < 2; j++) {
          const bool own = prev_interior && (FULL || !(near[j] & 1));
          const unsigned n = x0 + lane + p.nx * (prev_y0 + 2 * warp + j + p.ny * prev_z);
          fr[k].set(j, own ? rep[k * p.n + n] : 0.f);
        }
    }
    __syncthreads();  // local fields of plane J complete; iteration J-1 retired
    issue_next();     // into this plane's buffer (EARLY), else into plane J-1's
    if (alive && (lane == 0 || lane == width - 1)) {
      // the tile's first column is the left neighbour's right halo column, its last
      // column the right neighbour's left one
      auto send_column = [&](uint32_t peer, int exd) {
        const uint32_t bar = mapa_shared(smem_addr(&fld_full[fs]), peer);
        auto send = [&](int ey) {  // the fields this thread staged in row ey
#pragma unroll
          for (int f = 0; f < NV; f++) {
            const float* src = &fld[(fs * NV + f) * NE + ey * EX];
            st_async_f32(mapa_shared(smem_addr(src + exd), peer), src[lane + 1], bar);
          }
        };
        if (FULL || 2 * warp < rows) send(2 * warp + 1);
        if (FULL || 2 * warp + 1 < rows) send(2 * warp + 2);
        if (warp == halo_warp) {
          send(0);
          send(rows + 1);
        }
      };
      if constexpr (FULL) {
        send_column(lane == 0 ? left : right, lane == 0 ? TX + 1 : 0);
      } else {
        if (lane == 0) send_column(left, left_width + 1);
        if (lane == width - 1) send_column(right, 0);
      }
    }
    auto ready = [&]() { wait(&fld_full[fs], J / FS); };  // the neighbours' columns of plane J
    if (alive && !prev_interior) ready();
    // ---- collide plane J-1 ----
    const bool any_live = FULL || __any_sync(0xffffffffu, !(near[0] & near[1] & 1));
    if (alive && prev_interior && !any_live) ready();  // walls, or rows beyond a partial tile
    if (alive && prev_interior && any_live) {
      const int slm = (J + FS - 2) % FS, sl0 = (J + FS - 1) % FS;
      const int e0 = (2 * warp + 1) * EX + (lane + 1);
      const float* f_m = fld + slm * NV * NE + e0;
      const float* f_0 = fld + sl0 * NV * NE + e0;
      const float* f_p = fld + fs * NV * NE + e0;
      // storage indices: columns x-1 .. x+1, rows y-1 .. y+2, planes z-1 .. z+1 (periodic)
      const int gx = x0 + lane, gy = prev_y0 + 2 * warp, zz = prev_z;
      auto row = [&](int y) { return unsigned((y >= p.ny ? y - p.ny : y) * p.px); };
      const unsigned xo[3] = {unsigned(gx == 0 ? p.nx - 1 : gx - 1), unsigned(gx), unsigned(gx + 1 >= p.nx ? 0 : gx + 1)};
      const unsigned yo[4] = {row(gy == 0 ? p.ny - 1 : gy - 1), row(gy), row(gy + 1), row(gy + 2)};
      const unsigned zo[3] = {unsigned((zz == 0 ? p.nz - 1 : zz - 1) * plane_n), unsigned(zz * plane_n),
                              unsigned((zz + 1 >= p.nz ? 0 : zz + 1) * plane_n)};
      auto dest = [&](int i, int j) -> unsigned {
        return xo[cx<L>(i) + 1] + yo[cy<L>(i) + 1 + j] + zo[cz<L>(i) + 1];
      };
#pragma unroll
      for (int k = 0; k < K; k++)
#pragma unroll
        for (int j = 0; j < 2; j++)
          if (FULL || !(near[j] & 1)) out.r[k][dest(0, j)] = hcs[k].q[j];
      auto collide = [&](auto with_walls) {
        constexpr bool WALLED = decltype(with_walls)::value;
        // field f at neighbour i of node j; at a wall, of the node itself
        auto nb = [&](int f, int i, int j) -> float {
          const float* base = cz<L>(i) == 0 ? f_0 : (cz<L>(i) > 0 ? f_p : f_m);
          const float* at = base + (cy<L>(i) + j) * EX + cx<L>(i);
          if constexpr (WALLED) at = (near[j] >> i) & 1 ? f_0 + j * EX : at;
          return at[f * NE];
        };
        // a result of component k, re-referenced to the destination's density (field f), out;
        // what runs into a wall comes back into the opposite direction's array, ns elements off
        auto push = [&](int k, int f, int i, const F2& v) {
          F2 o = v;
          if (i != 0) {
            F2 n;
#pragma unroll
            for (int j = 0; j < 2; j++) n.set(j, nb(f, i, j));
            o = fma(F2(p.phi[k][grp<L>(i)]), hcs[k].q - n, v);
          }
#pragma unroll
          for (int j = 0; j < 2; j++) {
            // (chosen first and stored under one predicate, the walled form takes no branches)
            int to = int(dest(i, j));
            if (WALLED && i != 0) {
              const int back = int(dest(0, j)) + (opp<L>(i) > i ? plane_n * p.nz : -plane_n * p.nz);
              to = (near[j] >> i) & 1 ? back : to;
            }
            S* const at = WALLED ? out.f[k * Q + i] + to : out.f[k * Q + i] + dest(i, j);
            if (FULL || !(near[j] & 1)) *at = st_s<S, T>(o[j]);
          }
        };
        if constexpr (MODEL == kCG) {
          auto emit = [&](int i, const F2& vR, const F2& vB) {
            push(0, 0, i, vR);
            push(1, 1, i, vB);
          };
          cg_collide_pair<L, REP>(p, hold, hcs[0], hcs[1], fr, nb, ready, emit);
        } else if constexpr (MODEL == kSC2C) {
          auto emit = [&](int k, int i, const F2& v) { push(k, k, i, v); };
          sc2c_collide_pair<L>(p, hold, hcs, nb, ready, emit);
        } else {
          F2 psic;
#pragma unroll
          for (int j = 0; j < 2; j++) psic.set(j, nb(0, 0, j));
          auto emit = [&](int i, const F2& v) { push(0, 1, i, v); };
          scmp_collide_pair<L>(p, hold, hcs[0], psic, nb, ready, emit);
        }
      };
      if constexpr (WALLS) {
        if (walled || one_form)
          collide(std::true_type{});
        else
          collide(std::false_type{});
      } else {
        collide(std::false_type{});
      }
    }
    if constexpr (EARLY) {
#pragma unroll
      for (int i = 0; i < Q; i++) hold[i] = next_hold[i];
    } else if (alive) {
      // the deviations of plane J again, from its raw buffer (intact until the copy issued
      // after the next block barrier)
      const S* p0 = reinterpret_cast<const S*>(b + Lay::PM::row(2 * warp + 1)) + lane;
      const S* p1 = reinterpret_cast<const S*>(b + Lay::PM::row(2 * warp + 2)) + lane;
#pragma unroll
      for (int i = 0; i < NH * Q; i++) {
        hold[i].set(0, ld_s<S, T>(p0[i * TX]));
        hold[i].set(1, ld_s<S, T>(p1[i * TX]));
      }
    }
#pragma unroll
    for (int k = 0; k < K; k++) hcs[k] = cs[k];
    near[0] = next_near[0];
    near[1] = next_near[1];
    walled = next_walled;
    prev_interior = interior;
    prev_z = z;
    prev_y0 = y0;
    cur.advance();
  }
  if (!REP) admit_next_step();  // (a plain launch follows: the next step's force)
  // the copies this block issued have landed before its shared memory is released
  if (tid == 0)
    for (int j = max(0, issued - RAW); j < issued; j++) mbar_wait_bounded(&raw_full[j % RAW], (j / RAW) & 1);
  __syncwarp();
  cluster_sync_all();  // no block leaves while a neighbour may still write to it
}

}  // namespace lbm
