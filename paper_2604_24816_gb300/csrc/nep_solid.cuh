// nep_solid.cuh -- solid harmonics of the fused kernels, and their weighted gradient without gradient
// polynomials (sm_103a).
//
// The rotation-invariant descriptors q_nl = sum_m s_nlm^2 (Section III.B) do not depend on the basis chosen
// inside each l, so the fused kernels keep the angular sums and the adjoint row over the regular solid
// harmonics R_lm(u) = r^l P_lm(cos theta) e^(i m phi) / (l + m)! (P_lm without the (-1)^m phase), as real
// components C_lm = Re R_lm (m = 0..l) and S_lm = Im R_lm (m = 1..l).  They are linked by
//   dR_lm/dz = R_(l-1)m,   (d/dx + i d/dy) R_lm = -R_(l-1)(m+1),   (d/dx - i d/dy) R_lm = R_(l-1)(m-1)
// (the standard relations of the regular solid harmonics), so that the gradient of sum_lm b_lm R_lm is a
// sum over the lower degree's values with sums and differences of the weights: solid_grad below needs 38
// (paired) instructions for 24 components where gradient polynomials and their accumulation took about 100
// (the teacher's fused kernel, issue-bound: 1.114 -> 1.060 ms at 1,048,576 atoms and no spills; the student's,
// which has 8 components and waits on its walk, unchanged).
// The normalised harmonics of the addition theorem are Yh_lm = solid_norm R_lm; a sum kept over R is
// s' = s / norm and an adjoint row over R is G' = norm G, scaled once per atom.
//
// Order of the NLM components (LMAX = 4: 24, LMAX = 2: 8): the pairs (C_lm, S_lm), m = 1..l, degree by
// degree, then the C_l0.  Pair index l(l-1)/2 + m - 1; pairs sit at even positions, so a pair is one float2.
#pragma once

#include "nep_common.cuh"

namespace nep {

__host__ __device__ constexpr int solid_pairs(int nlm) { return nlm == 24 ? 10 : 3; }
__host__ __device__ constexpr int solid_pair_l(int k) { return k < 1 ? 1 : (k < 3 ? 2 : (k < 6 ? 3 : 4)); }
__host__ __device__ constexpr int solid_pair_m(int k) { return k - solid_pair_l(k) * (solid_pair_l(k) - 1) / 2 + 1; }
__host__ __device__ constexpr int solid_l(int nlm, int p) {
  return p < 2 * solid_pairs(nlm) ? solid_pair_l(p / 2) : p - 2 * solid_pairs(nlm) + 1;
}
__host__ __device__ constexpr int solid_m(int nlm, int p) {
  return p < 2 * solid_pairs(nlm) ? solid_pair_m(p / 2) : 0;
}
// l! for m = 0, sqrt(2 (l - m)! (l + m)!) otherwise.
__host__ __device__ constexpr float solid_norm(int nlm, int p) {
  const int l = solid_l(nlm, p), m = solid_m(nlm, p);
  if (m == 0) return l == 1 ? 1.f : (l == 2 ? 2.f : (l == 3 ? 6.f : 24.f));
  if (l == 1) return 2.f;
  if (l == 2) return m == 1 ? 3.4641016151377546f : 6.928203230275509f;            // sqrt 12, sqrt 48
  if (l == 3) return m == 1 ? 9.797958971132712f : (m == 2 ? 15.491933384829668f   // sqrt 96, sqrt 240
                                                            : 37.94733192202055f);   // sqrt 1440
  return m == 1 ? 37.94733192202055f : (m == 2 ? 53.66563145999495f : (m == 3 ? 100.39920318408906f
                                                                               : 283.97183031300545f));
}
// The l = 2 component at position p in the order of the 4-body tensor (xy, yz, z^2, xz, x^2 - y^2), -1 for
// another degree.
__host__ __device__ constexpr int solid_quadrupole(int nlm, int p) {
  if (solid_l(nlm, p) != 2) return -1;
  const int m = solid_m(nlm, p);
  return m == 0 ? 2 : (m == 1 ? (p % 2 == 0 ? 3 : 1) : (p % 2 == 0 ? 4 : 0));
}

// Values at a unit vector: the sectoral pairs R_mm, from which R_lm = R_mm f_lm(z).
template <int NLM>
struct Solid {
  float z, z2;
  float2 r[NLM == 24 ? 4 : 2];       // R_mm, m = 1..LMAX
  __host__ __device__ __forceinline__ static float2 scaled(float2 v, float c) { return mul2(v, bc2(c)); }
  __host__ __device__ __forceinline__ Solid(float x, float y, float z_) : z(z_), z2(z_ * z_) {
    r[0] = make_float2(0.5f * x, 0.5f * y);
    r[1] = make_float2(0.5f * fmaf(r[0].x, r[0].x, -(r[0].y * r[0].y)), r[0].x * r[0].y);
    if constexpr (NLM == 24) {
      const float2 a = scaled(r[0], 1.f / 3.f), b = scaled(r[0], 0.25f);
      r[2] = make_float2(fmaf(a.x, r[1].x, -(a.y * r[1].y)), fmaf(a.x, r[1].y, a.y * r[1].x));
      r[3] = make_float2(fmaf(b.x, r[2].x, -(b.y * r[2].y)), fmaf(b.x, r[2].y, b.y * r[2].x));
    }
  }
  // (C, S) of pair k (a compile-time constant after unrolling)
  __host__ __device__ __forceinline__ float2 pair(int k) const {
    switch (k) {
      case 0: return r[0];
      case 1: return scaled(r[0], z);
      case 2: return r[1];
      case 3: return scaled(r[0], fmaf(0.625f, z2, -0.125f));
      case 4: return scaled(r[1], z);
      case 5: return r[NLM == 24 ? 2 : 0];
      case 6: return scaled(r[0], z * fmaf(7.f / 24.f, z2, -0.125f));
      case 7: return scaled(r[1], fmaf(7.f / 12.f, z2, -1.f / 12.f));
      case 8: return scaled(r[NLM == 24 ? 2 : 0], z);
      default: return r[NLM == 24 ? 3 : 0];
    }
  }
  // C_l0
  __host__ __device__ __forceinline__ float zonal(int l) const {
    switch (l) {
      case 1: return z;
      case 2: return fmaf(0.75f, z2, -0.25f);
      case 3: return z * fmaf(5.f / 12.f, z2, -0.25f);
      default: return fmaf(fmaf(35.f / 192.f, z2, -30.f / 192.f), z2, 3.f / 192.f);
    }
  }
  // components 4c..4c+3 as two pairs
  __host__ __device__ __forceinline__ void chunk(int c, float2 &a, float2 &b) const {
    constexpr int NP = solid_pairs(NLM);
    a = 2 * c < NP ? pair(2 * c) : make_float2(zonal(4 * c - 2 * NP + 1), zonal(4 * c - 2 * NP + 2));
    b = 2 * c + 1 < NP ? pair(2 * c + 1) : make_float2(zonal(4 * c - 2 * NP + 3), zonal(4 * c - 2 * NP + 4));
  }
};

// Gradient of sum_lm b_lm R_lm at the point of H, degree by degree: add<l> takes the weights of degree l (b: the
// pairs m = 1..l, b0: the zonal one) and sums over the values of degree l - 1.
struct SolidGrad {
  float2 c, s, zp;                   // sums over C and S values; z over pairs
  float z0;                          // z over zonal values
  __host__ __device__ __forceinline__ SolidGrad() : c(bc2(0.f)), s(bc2(0.f)), zp(bc2(0.f)), z0(0.f) {}
  template <int L, int NLM>
  __host__ __device__ __forceinline__ void add(const Solid<NLM> &H, const float2 *b, float b0) {
    if constexpr (L == 1) {
      c = add2(c, b[0]);             // C_00 = 1
      z0 += b0;
    } else {
      const float q0 = H.zonal(L - 1);
      c = fma2(bc2(q0), b[0], c);
      z0 = fmaf(q0, b0, z0);
#pragma unroll
      for (int m = 1; m < L; ++m) {
        const float2 v = H.pair((L - 1) * (L - 2) / 2 + m - 1);   // (C, S) of degree L - 1, order m
        const float2 up = b[m];                                   // weights of order m + 1
        float2 xc, xs;
        if (m == 1) {
          xc = make_float2(fmaf(-2.f, b0, up.x), up.y);
          xs = make_float2(fmaf(2.f, b0, up.x), up.y);
        } else {
          const float2 dn = b[m - 2];                             // weights of order m - 1
          xc = fma2(make_float2(-1.f, 1.f), dn, up);
          xs = fma2(make_float2(1.f, -1.f), dn, up);
        }
        c = fma2(bc2(v.x), xc, c);
        s = fma2(bc2(v.y), xs, s);
        zp = fma2(v, b[m - 1], zp);
      }
    }
  }
  __host__ __device__ __forceinline__ void get(float &gx, float &gy, float &gz) const {
    gx = 0.5f * (c.x + s.y);
    gy = 0.5f * (c.y - s.x);
    gz = hsum(zp) + z0;
  }
};

}  // namespace nep
