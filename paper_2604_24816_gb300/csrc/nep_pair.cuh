// nep_pair.cuh -- one pair's share of the forces from an atom's own adjoint row (sm_103a), shared by the fused
// kernels (one thread per atom, nep_force.cu) and the wide kernels (several lanes per atom, nep_wide.cu).
#pragma once

#include "nep_descriptor.cuh"

namespace nep {

// The adjoint row of an atom as angular_pair_solid reads it, four components of every channel at a time.
template <class S>
struct RowTmem {
  uint32_t trow;
  __device__ __forceinline__ void load(int k, float (&h)[S::NA][4]) const { tm_load<S>(trow, k, h); }
};
template <class S>
struct RowReg {
  const float (&g)[S::NA][S::NLM];
  __device__ __forceinline__ void load(int k, float (&h)[S::NA][4]) const {
#pragma unroll
    for (int a = 0; a < S::NA; ++a)
#pragma unroll
      for (int c = 0; c < 4; ++c) h[a][c] = g[a][4 * k + c];
  }
};

// The same force part for a row over the solid harmonics (G' = solid_norm G): with f_lm = R_lm(u), homogeneous
// of degree l in u, d/dd [g(r) f(u)] = g' f u + (g / r) (grad f - u (u . grad f)), so no factor l appears:
// al = sum_lm A_lm R_lm and gv = sum_lm B_lm grad R_lm (SolidGrad) give the force (al - u . gv / r) u + gv / r.
// The zonal weights come first (their chunk is the row's last), since each degree's gradient needs its own.
template <class S, class Row>
__device__ __forceinline__ void angular_pair_solid(const Model<S> &P, const Row &row, bool si, float r, float ir,
                                                   float dx, float dy, float dz, float &coef, float &vx, float &vy,
                                                   float &vz) {
  constexpr int NP = solid_pairs(S::NLM), NC = S::NLM / 4;
  const float ar = si ? 1.f : r;
  const float ux = si ? 1.f : dx * ir, uy = si ? 0.f : dy * ir, uz = si ? 0.f : dz * ir;
  float g[S::NA], dg[S::NA];
  radial_channels_d<S>(P, ar, g, dg);
  const Solid<S::NLM> H(ux, uy, uz);
  SolidGrad G;
  float2 al = bc2(0.f), b[NP];
  float b0[S::LMAX + 1];
#pragma unroll
  for (int kk = 0; kk < NC; ++kk) {
    const int k = kk == 0 ? NC - 1 : kk - 1;
    float h[S::NA][4];
    row.load(k, h);
    float2 a01 = mul2(pr(h[0][0], h[0][1]), bc2(dg[0])), a23 = mul2(pr(h[0][2], h[0][3]), bc2(dg[0]));
    float2 b01 = mul2(pr(h[0][0], h[0][1]), bc2(g[0])), b23 = mul2(pr(h[0][2], h[0][3]), bc2(g[0]));
#pragma unroll
    for (int a = 1; a < S::NA; ++a) {
      const float2 h01 = pr(h[a][0], h[a][1]), h23 = pr(h[a][2], h[a][3]);
      const float2 dg2 = bc2(dg[a]), g2 = bc2(g[a]);
      a01 = fma2(h01, dg2, a01);
      a23 = fma2(h23, dg2, a23);
      b01 = fma2(h01, g2, b01);
      b23 = fma2(h23, g2, b23);
    }
    float2 y01, y23;
    H.chunk(k, y01, y23);
    al = fma2(a01, y01, al);
    al = fma2(a23, y23, al);
    if (2 * k < NP) b[2 * k < NP ? 2 * k : 0] = b01;
    else { b0[4 * k - 2 * NP + 1] = b01.x; b0[4 * k - 2 * NP + 2] = b01.y; }
    if (2 * k + 1 < NP) b[2 * k + 1 < NP ? 2 * k + 1 : 0] = b23;
    else { b0[4 * k - 2 * NP + 3] = b23.x; b0[4 * k - 2 * NP + 4] = b23.y; }
    // the degrees whose pairs are complete after this chunk
    if constexpr (S::NLM == 24) {
      if (k == 0) G.template add<1>(H, b, b0[1]);
      if (k == 1) G.template add<2>(H, b + 1, b0[2]);
      if (k == 2) G.template add<3>(H, b + 3, b0[3]);
      if (k == 4) G.template add<4>(H, b + 6, b0[4]);
    } else {
      if (k == 0) {
        G.template add<1>(H, b, b0[1]);
        G.template add<2>(H, b + 1, b0[2]);
      }
    }
  }
  float gx, gy, gz;
  G.get(gx, gy, gz);
  coef = (hsum(al) - ir * fmaf(ux, gx, fmaf(uy, gy, uz * gz))) * ir;
  vx = gx * ir; vy = gy * ir; vz = gz * ir;
}

// Radial and LJ part of one active pair's force coefficient (d = coef * r_ij + angular part): the
// radial adjoint (the two cubics c0, c1 of radial_tail_cubics) against the basis derivatives, plus half of the shifted-force LJ pair force.  INSIDE_RC: the caller knows that
// r < rc_R (an angular pair: rc_A <= rc_R is checked by nep_create).  LJ = false: without
// the pair term.  e2: gets the pair's LJ energy added.
template <class S, bool INSIDE_RC = false, bool LJ = true>
__device__ __forceinline__ float radial_lj_coef(const Model<S> &P, float4 c0, float4 c1, float r2, float r, float ir,
                                                float *e2 = nullptr) {
  float coef = 0.f;
  if (INSIDE_RC || r2 < P.rcR2) coef = cubics_deriv(c0, c1, r, P.inv_rcR) * ir;
  if (LJ && P.lj_on != 0.f && r2 < P.lj_rc2) {
    float el, dl;
    lj_pair<S>(P, r2, r, ir, el, dl);
    coef = fmaf(0.5f * dl, ir, coef);
    if (e2 != nullptr) *e2 += el;
  }
  return coef;
}

}  // namespace nep
