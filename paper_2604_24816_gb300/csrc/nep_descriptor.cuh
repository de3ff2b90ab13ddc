// nep_descriptor.cuh -- per-atom descriptor pieces shared by the float32 and the mixed-precision
// descriptor kernels: the neighbour walk that accumulates the radial sums q_n, the LJ energy and the
// angular sums s_nlm (Section III.B; the geometry of each neighbour is computed once and reused for all
// channels, Algorithm 1 with one tile), the rotation invariants q_nl and q4_n, and the adjoint row
// G_nlm = dU/ds_nlm built from the network gradient.
#pragma once

#include <cuda_fp16.h>

#include "nep_common.cuh"
#include "nep_solid.cuh"
#include "nep_tc.cuh"

namespace nep {

// Adjoint rows in memory are float32 (the teacher's separate kernels) or float16 (the mixed student's); the force
// kernel reads them W values per 16-byte load.
template <class GT>
struct GTraits;
template <>
struct GTraits<float> {
  static constexpr int W = 4;
};
template <>
struct GTraits<__half> {
  static constexpr int W = 8;
};

__device__ __forceinline__ void load_vec(const float *p, float (&v)[4]) {
  const float4 t = __ldg(reinterpret_cast<const float4 *>(p));
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void load_vec(const __half *p, float (&v)[8]) {
  const uint4 t = __ldg(reinterpret_cast<const uint4 *>(p));
  const uint32_t w[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&w[k]));
    v[2 * k] = f.x; v[2 * k + 1] = f.y;
  }
}
// The 8 values at the tail of a row (dU/dq_n of the radial descriptors and padding).
template <class GT>
__device__ __forceinline__ void load_tail8(const GT *row, int off, float (&v)[8]) {
  constexpr int W = GTraits<GT>::W;
#pragma unroll
  for (int b = 0; b < 8; b += W) {
    float t[W];
    load_vec(row + off + b, t);
#pragma unroll
    for (int k = 0; k < W; ++k) v[b + k] = t[k];
  }
}

// Per-atom fallback to another model (the teacher) for atoms whose scaled descriptors leave a box:
// an atom is flagged when some q~_nu = q_scale_nu q_nu lies outside [lo_nu, hi_nu].  Flagged atoms
// get a zero adjoint row and no site energy from this model; their indices are appended to `list`
// (order of arrival: the consumers only use integer atomics, so results do not depend on it).
struct Fallback {
  int on;
  int cap;                 // capacity of list
  int *list, *count;       // flagged atoms (cell-sorted indices), number flagged
  float lo[16], hi[16];
};

template <class S>
__device__ __forceinline__ bool out_of_range(const Fallback &fb, const Model<S> &P, const float (&q)[S::NDES]) {
  bool out = false;
  if constexpr (S::NDES <= 16) {       // the range box holds up to 16 descriptors (the student's 12)
#pragma unroll
    for (int v = 0; v < S::NDES; ++v) {
      const float t = q[v] * P.qs[v];
      out |= (t < fb.lo[v]) | (t > fb.hi[v]);
    }
  }
  return out;
}

// Append atom i to the fallback list (status bit ST_FB_OVERFLOW when the list is full).
__device__ __forceinline__ void flag_atom(const Fallback &fb, int i, int *status) {
  const int slot = atomicAdd(fb.count, 1);
  if (slot < fb.cap) fb.list[slot] = i;
  else atomicOr(status, ST_FB_OVERFLOW);
}

template <class S>
struct AtomSums {
  float QR[S::KR];        // radial basis sums sum_j f_k(r_ij); q_n = sum_k cR_nk QR_k
  static_assert(S::KR <= 8, "the radial adjoint in basis space lives in the 8-element row tail");
  float s[S::NA][S::NLM];
  float elj;
  int nrad, nang, nact, cnt;
};

// Walk atom i's full neighbour row and accumulate q_n, s_nlm and the LJ energy.  REC: every active pair
// is also recorded as (dx, dy, dz, j) at rec[off + slot * BLOCK], angular pairs from slot 0 up and the
// other active pairs from slot pmax - 1 down (the layout of accumulate_atom_tm's records).
// SOLID: the sums over the solid harmonics (s' = s / solid_norm, in the order of nep_solid.cuh).
template <class S, int DE, int DP, int BLOCK, bool REC = false, bool SOLID = false>
__device__ __forceinline__ void accumulate_atom(const Model<S> &P, const float4 *shift, int i, int n,
                                                const float4 *__restrict__ pos, const int32_t *__restrict__ nbr,
                                                RowSpan sp, uint32_t *ring_e, float4 *ring_p, AtomSums<S> &A,
                                                float4 *__restrict__ rec = nullptr, unsigned off = 0, int pmax = 0) {
  const int cnt = sp.c;
  const float4 pi = pos[i];
  static_assert(S::KR == 8, "eight basis functions");
  float2 Q[4] = {bc2(0.f), bc2(0.f), bc2(0.f), bc2(0.f)};
#pragma unroll
  for (int a = 0; a < S::NA; ++a)
#pragma unroll
    for (int c = 0; c < S::NLM; ++c) A.s[a][c] = 0.f;
  A.elj = 0.f;
  A.nrad = 0; A.nang = 0; A.nact = 0; A.cnt = cnt;
  NbrPipe<DE, DP, BLOCK> pipe;
  pipe.start(ring_e, ring_p, nbr + i, (size_t)n, pos, sp);
  const unsigned last = off + (unsigned)(pmax - 1) * BLOCK;
  unsigned oa = off, oo = last;                        // REC: where the next angular and the next other record go
  for (int k = 0; k < cnt; ++k) {
    uint32_t e;
    float4 pj;
    pipe.get(k, e, pj);
    const float4 o = shift[e >> J_BITS];
    const float dx = pj.x - pi.x + o.x, dy = pj.y - pi.y + o.y, dz = pj.z - pi.z + o.z;
    const float r2 = dx * dx + dy * dy + dz * dz;
    if (r2 >= P.rmax2) continue;
    if constexpr (REC) {
      const bool in_a = r2 < P.rcA2;
      rec[in_a ? oa : oo] = make_float4(dx, dy, dz, __int_as_float((int)(e & J_MASK)));
      if (in_a) oa += BLOCK;
      else oo -= BLOCK;
    } else {
      ++A.nact;
    }
    const float ir = rsqrtf(r2);
    const float r = r2 * ir;
    if (REC || r2 < P.rcR2) {                          // (the pair term's cutoff is at most rc_R: nep_create)
      cheb_accumulate(r, P.inv_rcR, Q);
      if (!REC) ++A.nrad;
    }
    if (!REC && P.lj_on != 0.f && r2 < P.lj_rc2) {
      float el, dl;
      lj_pair<S>(P, r2, r, ir, el, dl);
      A.elj = fmaf(0.5f, el, A.elj);
    }
    if (r2 < P.rcA2) {
      float g[S::NA];
      radial_channels<S>(P, r, true, g);
      float Y[S::NLM];
      if constexpr (SOLID) {
        const Solid<S::NLM> H(dx * ir, dy * ir, dz * ir);
#pragma unroll
        for (int k = 0; k < S::NLM / 4; ++k) {
          float2 y01, y23;
          H.chunk(k, y01, y23);
          Y[4 * k] = y01.x; Y[4 * k + 1] = y01.y; Y[4 * k + 2] = y23.x; Y[4 * k + 3] = y23.y;
        }
      } else {
        harmonics<S::NLM>(dx * ir, dy * ir, dz * ir, Y);
      }
#pragma unroll
      for (int a = 0; a < S::NA; ++a)
#pragma unroll
        for (int c = 0; c < S::NLM; ++c) A.s[a][c] = fmaf(g[a], Y[c], A.s[a][c]);
      if (!REC) ++A.nang;
    }
  }
  if constexpr (REC) {
    A.nang = (int)((oa - off) / BLOCK);
    A.nact = A.nrad = A.nang + (int)((last - oo) / BLOCK);
  }
  pipe.finish();
  cheb_sums(Q, A.QR);
}
// Traceless 4-body tensors T_n rebuilt from the l = 2 sums (components 3..7 = m -2..2).
template <class S>
struct FourBody {
  float xx[S::NA], yy[S::NA], zz[S::NA], xy[S::NA], yz[S::NA], xz[S::NA];
};

// Traceless T_n from the l = 2 sums s2[n][m] (components 3..7 of s_nl m, m = -2..2) and the 4-body
// descriptors q4_n = tr(T_n^3) = 3 det T_n, written to q[NR + NA LMAX + n].
template <class S>
__device__ __forceinline__ void fourbody_tensors(const float (&s2)[S::NA][5], FourBody<S> &T, float (&q)[S::NDES]) {
  const float i3 = 0.57735026918962576f, third = 1.f / 3.f;
#pragma unroll
  for (int a = 0; a < S::NA; ++a) {
    T.xy[a] = s2[a][0] * i3;
    T.yz[a] = s2[a][1] * i3;
    T.xz[a] = s2[a][3] * i3;
    T.xx[a] = s2[a][4] * i3 - s2[a][2] * third;
    T.yy[a] = -s2[a][4] * i3 - s2[a][2] * third;
    T.zz[a] = 2.f * s2[a][2] * third;
    const float det = T.xx[a] * (T.yy[a] * T.zz[a] - T.yz[a] * T.yz[a]) -
                      T.xy[a] * (T.xy[a] * T.zz[a] - T.yz[a] * T.xz[a]) +
                      T.xz[a] * (T.xy[a] * T.yz[a] - T.yy[a] * T.xz[a]);
    q[S::NR + S::NA * S::LMAX + a] = 3.f * det;
  }
}

// Descriptors [q_n | q_nl (n-major, l = 1..LMAX) | q4_n = tr(T_n^3) = 3 det T_n (teacher shape only)].
// SOLID: A holds s' (accumulate_atom<.., SOLID>), scaled by solid_norm here.
template <class S, bool SOLID = false>
__device__ __forceinline__ void descriptors_of(const Model<S> &P, const AtomSums<S> &A, float (&q)[S::NDES],
                                               FourBody<S> &T) {
#pragma unroll
  for (int a = 0; a < S::NR; ++a) {
    float t = 0.f;
#pragma unroll
    for (int k = 0; k < S::KR; ++k) t = fmaf(P.cR[a][k], A.QR[k], t);
    q[a] = t;
  }
#pragma unroll
  for (int a = 0; a < S::NA; ++a) {
#pragma unroll
    for (int l = 1; l <= S::LMAX; ++l) q[S::NR + a * S::LMAX + (l - 1)] = 0.f;
#pragma unroll
    for (int c = 0; c < S::NLM; ++c) {
      const float sc = SOLID ? solid_norm(S::NLM, c) * A.s[a][c] : A.s[a][c];
      float &ql = q[S::NR + a * S::LMAX + (SOLID ? solid_l(S::NLM, c) : lm_l(c)) - 1];
      ql = fmaf(sc, sc, ql);
    }
  }
  if constexpr (S::FOURBODY) {
    static_assert(!SOLID, "the register-resident solid-harmonic rows have no 4-body term");
    float s2[S::NA][5];
#pragma unroll
    for (int a = 0; a < S::NA; ++a)
#pragma unroll
      for (int m = 0; m < 5; ++m) s2[a][m] = A.s[a][3 + m];
    fourbody_tensors<S>(s2, T, q);
  }
}

// The one-hidden-layer network (Section III.B equation): U = sum_mu w1_mu tanh(sum_nu W0_mu,nu q~_nu -
// b0_mu) - b1 with q~ = q_scale q; returns U and Fp_nu = dU/dq_nu (zero for an atom flagged for the
// fallback model, whose site energy comes from the other model).
// MT: the operands of its two products are rounded to that type (W0 by the host already), sums in float32.
template <class S, class MT = float>
__device__ __forceinline__ float network(const Model<S> &P, const float (&q)[S::NDES], bool flagged,
                                         float (&Fp)[S::NDES]) {
  float qt[S::NDES], dq[S::NDES];
#pragma unroll
  for (int v = 0; v < S::NDES; ++v) { qt[v] = round_to<MT>(q[v] * P.qs[v]); dq[v] = 0.f; }
  float U = -P.b1;
  // The teacher's 30 x 30 network, fully unrolled, is ~2k instructions of straight-line code that the
  // row-walk loops share the instruction cache with; one neuron per iteration (weights read from the
  // constant bank with a register offset) measured 2 % faster in the fused kernel.
  constexpr int UNROLL = S::NNEU * S::NDES > 400 ? 1 : S::NNEU;
#pragma unroll UNROLL
  for (int mu = 0; mu < S::NNEU; ++mu) {
    float z = -P.b0[mu];
#pragma unroll
    for (int v = 0; v < S::NDES; ++v) z = fmaf(P.W0[mu][v], qt[v], z);
    const float h = tanhf(z);
    U = fmaf(P.w1[mu], h, U);
    const float t = round_to<MT>(P.w1[mu] * (1.f - h * h));
#pragma unroll
    for (int v = 0; v < S::NDES; ++v) dq[v] = fmaf(t, P.W0[mu][v], dq[v]);
  }
#pragma unroll
  for (int v = 0; v < S::NDES; ++v) Fp[v] = flagged ? 0.f : dq[v] * P.qs[v];
  return U;
}

// Radial adjoint in basis space, stored in the row tail: tail_k = dU/dQR_k = sum_n Fp_n cR_nk, so the
// force kernel contracts it directly with the basis derivatives f_k'(r) of each pair.
template <class S>
__device__ __forceinline__ void radial_tail(const Model<S> &P, const float (&Fp)[S::NDES], float (&tail)[8]) {
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    float t = 0.f;
    if (k < S::KR) {
#pragma unroll
      for (int a = 0; a < S::NR; ++a) t = fmaf(Fp[a], P.cR[a][k], t);
    }
    tail[k] = t;
  }
}

// The radial tail as the fused kernels' force pass contracts it (cubics_deriv): the two cubics of
// cheb_to_cubics, (e0, o0, e1, o1) in c0 and (e2, o2, e3, o3) in c1.
__device__ __forceinline__ void radial_tail_cubics(const float (&tail)[8], float4 &c0, float4 &c1) {
  float e[4], o[4];
  cheb_to_cubics(tail, e, o);
  c0 = make_float4(e[0], o[0], e[1], o[1]);
  c1 = make_float4(e[2], o[2], e[3], o[3]);
}

// 4-body part of the adjoint of channel a for the l = 2 components 3..7, per unit dU/dq4_a:
// d tr(T^3)/d s_m = 3 (T^2) : dT/ds_m.
template <class S>
__device__ __forceinline__ void fourbody_adjoint(int a, const FourBody<S> &T, float (&g4)[5]) {
  const float Mxx = T.xx[a] * T.xx[a] + T.xy[a] * T.xy[a] + T.xz[a] * T.xz[a];
  const float Myy = T.xy[a] * T.xy[a] + T.yy[a] * T.yy[a] + T.yz[a] * T.yz[a];
  const float Mzz = T.xz[a] * T.xz[a] + T.yz[a] * T.yz[a] + T.zz[a] * T.zz[a];
  const float Mxy = T.xx[a] * T.xy[a] + T.xy[a] * T.yy[a] + T.xz[a] * T.yz[a];
  const float Myz = T.xy[a] * T.xz[a] + T.yy[a] * T.yz[a] + T.yz[a] * T.zz[a];
  const float Mxz = T.xx[a] * T.xz[a] + T.xy[a] * T.yz[a] + T.xz[a] * T.zz[a];
  const float s3 = 1.7320508075688772f;
  g4[0] = 2.f * s3 * Mxy;
  g4[1] = 2.f * s3 * Myz;
  g4[2] = 2.f * Mzz - Mxx - Myy;
  g4[3] = 2.f * s3 * Mxz;
  g4[4] = s3 * (Mxx - Myy);
}

// Adjoint of channel a: gl[c] = dU/ds_{a,c} = 2 Fp_{a,l(c)} s_{a,c} (+ 4-body gradient for l = 2:
// d tr(T^3)/d s_m = 3 (T^2) : dT/ds_m).
// SOLID: A holds s' and the row is G' = solid_norm G, over the solid harmonics (adjoint_chunk).
template <class S, bool SOLID = false>
__device__ __forceinline__ void adjoint_channel(int a, const AtomSums<S> &A, const FourBody<S> &T,
                                                const float (&Fp)[S::NDES], float (&gl)[S::NLM]) {
#pragma unroll
  for (int c = 0; c < S::NLM; ++c) {
    const float h = SOLID ? solid_norm(S::NLM, c) : 1.f;
    gl[c] = (2.f * h * h) * Fp[S::NR + a * S::LMAX + (SOLID ? solid_l(S::NLM, c) : lm_l(c)) - 1] * A.s[a][c];
  }
  if constexpr (S::FOURBODY) {
    static_assert(!SOLID, "the register-resident solid-harmonic rows have no 4-body term");
    const float f4 = Fp[S::NR + S::NA * S::LMAX + a];
    float g4[5];
    fourbody_adjoint<S>(a, T, g4);
#pragma unroll
    for (int m = 0; m < 5; ++m) gl[3 + m] = fmaf(f4, g4[m], gl[3 + m]);
  }
}

// ---------------------------------------------------------------------------------------------------
// Teacher shape with the 120 angular sums s_nlm in tensor memory (TMEM) instead of registers, in the chunked layout
// of tm_col (chunk k = components 4k..4k+3 of every channel: one x16 access for channels 0..3 and one x4
// access for channel 4), which the force pass's adjoint row shares.  All TMEM accesses are
// warp-collective, so the neighbour walk runs to the warp's longest row (threads past their own row, or
// past the last atom, idle with a predicate) and the angular update is made by whole warps, lanes
// without an angular pair adding g = 0.
constexpr int TMEM_W = 4;

// Chunk k of every channel into v (one statement, waited for), and v into it.
template <class S>
__device__ __forceinline__ void tm_load(uint32_t trow, int k, float (&v)[S::NA][TMEM_W]) {
  tmem_ld_chunk<S::NLM>(trow, k, v);
}
template <class S>
__device__ __forceinline__ void tm_store(uint32_t trow, int k, const float (&v)[S::NA][TMEM_W]) {
  tmem_st_chunk<S::NLM>(trow, k, v);
}

// Zero the sums, then walk atom ii's row (cnt entries; cnt = 0 for threads past the last atom):
// radial basis sums QR and the LJ energy in registers, s_nlm in TMEM.
// The accumulations run in float2 pairs (two basis functions, or two (l, m) components, per instruction).
// REC: every active pair is also recorded as (dx, dy, dz, j) at rec[off + slot * BLOCK] (off: this
// thread's column of a [pmax][BLOCK] array): angular pairs (r < rc_A) from
// slot 0 up in walk order, the other active pairs from slot pmax - 1 down (pmax >= the row length, so
// the two never meet).
template <class S, int DE, int DP, int BLOCK, bool REC = false, bool SOLID = false>
__device__ __forceinline__ void accumulate_atom_tm(const Model<S> &P, const float4 *shift, uint32_t trow, int ii,
                                                   int n, const float4 *__restrict__ pos,
                                                   const int32_t *__restrict__ nbr, RowSpan sp, uint32_t *ring_e,
                                                   float4 *ring_p, float (&QR)[S::KR],
                                                   float &elj, int &nrad, int &nang, int &nact,
                                                   float4 *__restrict__ rec = nullptr, unsigned off = 0, int pmax = 0) {
  static_assert(S::NA == 5 && S::NLM == 24, "teacher shape");
  static_assert(S::KR == 8, "eight basis functions");
  constexpr int W = TMEM_W;
  constexpr int NC = S::NLM / W;
  {
    float z[S::NA][W];
#pragma unroll
    for (int a = 0; a < S::NA; ++a)
#pragma unroll
      for (int c = 0; c < W; ++c) z[a][c] = 0.f;
#pragma unroll
    for (int k = 0; k < NC; ++k) tm_store<S>(trow, k, z);
    tmem_wait_st();
  }
  float2 Q[4] = {bc2(0.f), bc2(0.f), bc2(0.f), bc2(0.f)};
  elj = 0.f;
  nrad = 0; nang = 0; nact = 0;
  const float4 pi = pos[ii];
  const int cnt = sp.c;
  NbrPipe<DE, DP, BLOCK> pipe;
  pipe.start(ring_e, ring_p, nbr + ii, (size_t)n, pos, sp);
  const int trip = __reduce_max_sync(0xffffffffu, cnt);
  const unsigned last = off + (unsigned)(pmax - 1) * BLOCK;
  unsigned oa = off, oo = last;                        // REC: where the next angular and the next other record go
  for (int k = 0; k < trip; ++k) {
    const bool valid = k < cnt;
    uint32_t e;
    float4 pj;
    // past the end of the row the ring slots are stale: act below is false for them, and e = 0 keeps
    // the shift-table index in range
    pipe.get(k, e, pj);
    e = valid ? e : 0u;
    const float4 o = shift[e >> J_BITS];
    const float dx = pj.x - pi.x + o.x, dy = pj.y - pi.y + o.y, dz = pj.z - pi.z + o.z;
    const float r2 = dx * dx + dy * dy + dz * dz;
    const bool act = valid && r2 < P.rmax2;
    const float ir = rsqrtf(r2);
    const float r = r2 * ir;
    if (act) {
      if constexpr (REC) {
        const bool in_a = r2 < P.rcA2;
        rec[in_a ? oa : oo] = make_float4(dx, dy, dz, __int_as_float((int)(e & J_MASK)));
        if (in_a) oa += BLOCK;
        else oo -= BLOCK;
      } else {
        ++nact;
      }
      if (REC || r2 < P.rcR2) {                        // (the pair term's cutoff is at most rc_R: nep_create)
        cheb_accumulate(r, P.inv_rcR, Q);
        if (!REC) ++nrad;
      }
      if (!REC && P.lj_on != 0.f && r2 < P.lj_rc2) {
        float el, dl;
        lj_pair<S>(P, r2, r, ir, el, dl);
        elj = fmaf(0.5f, el, elj);
      }
    }
    const bool ang = act && r2 < P.rcA2;
    if (__any_sync(0xffffffffu, ang)) {
      __syncwarp();
      const float ar = ang ? r : 1.f;
      const float ux = ang ? dx * ir : 1.f, uy = ang ? dy * ir : 0.f, uz = ang ? dz * ir : 0.f;
      float g[S::NA];
      radial_channels<S>(P, ar, ang, g);
      // SOLID: the components chunk by chunk (fewer live registers than 24 values)
      const Solid<S::NLM> H(ux, uy, uz);
      float Y[S::NLM];
      if constexpr (!SOLID) harmonics<S::NLM>(ux, uy, uz, Y);
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        float sv[S::NA][W];
        tm_load<S>(trow, k, sv);
        float2 y01, y23;
        if constexpr (SOLID) {
          H.chunk(k, y01, y23);
        } else {
          y01 = pr(Y[W * k], Y[W * k + 1]);
          y23 = pr(Y[W * k + 2], Y[W * k + 3]);
        }
#pragma unroll
        for (int a = 0; a < S::NA; ++a) {
          const float2 g2 = bc2(g[a]);
          const float2 lo = fma2(g2, y01, pr(sv[a][0], sv[a][1]));
          const float2 hi = fma2(g2, y23, pr(sv[a][2], sv[a][3]));
          sv[a][0] = lo.x; sv[a][1] = lo.y; sv[a][2] = hi.x; sv[a][3] = hi.y;
        }
        tm_store<S>(trow, k, sv);
      }
      tmem_wait_st();
      if (!REC && ang) ++nang;
    }
  }
  if constexpr (REC) {
    nang = (int)((oa - off) / BLOCK);
    nact = nrad = nang + (int)((last - oo) / BLOCK);
  }
  pipe.finish();
  cheb_sums(Q, QR);
}

// Descriptors from the radial basis sums and the sums s_nlm (q_nl = sum_m s_nlm^2, 4-body from the
// l = 2 sums), as descriptors_of.
// SOLID: sums over the solid harmonics (accumulate_atom_tm), scaled by solid_norm here.
template <class S, bool SOLID = false>
__device__ __forceinline__ void descriptors_tm(const Model<S> &P, uint32_t trow, const float (&QR)[S::KR],
                                               float (&q)[S::NDES], FourBody<S> &T) {
  constexpr int W = TMEM_W;
#pragma unroll
  for (int a = 0; a < S::NR; ++a) {
    float t = 0.f;
#pragma unroll
    for (int b = 0; b < S::KR; ++b) t = fmaf(P.cR[a][b], QR[b], t);
    q[a] = t;
  }
#pragma unroll
  for (int v = S::NR; v < S::NR + S::NA * S::LMAX; ++v) q[v] = 0.f;
  float s2[S::NA][5];
#pragma unroll
  for (int k = 0; k < S::NLM / W; ++k) {
    float sv[S::NA][W];
    tm_load<S>(trow, k, sv);
#pragma unroll
    for (int a = 0; a < S::NA; ++a)
#pragma unroll
      for (int cc = 0; cc < W; ++cc) {
        const int lm = W * k + cc;
        if constexpr (SOLID) sv[a][cc] *= solid_norm(S::NLM, lm);
        float &ql = q[S::NR + a * S::LMAX + (SOLID ? solid_l(S::NLM, lm) : lm_l(lm)) - 1];
        ql = fmaf(sv[a][cc], sv[a][cc], ql);
        const int m2 = SOLID ? solid_quadrupole(S::NLM, lm) : (lm >= 3 && lm < 8 ? lm - 3 : -1);
        if (m2 >= 0) s2[a][m2 < 0 ? 0 : m2] = sv[a][cc];
      }
  }
  fourbody_tensors<S>(s2, T, q);
}

// 4-body adjoint factors g4[a] = 3 (T_a^2) : dT_a/ds_m of every channel, with the tensors T_a rebuilt
// from the l = 2 sums (chunks 0 and 1, and the zonal component of chunk 5 with SOLID), so that T need not
// stay live across the network.
template <class S, bool SOLID = false>
__device__ __forceinline__ void fourbody_adjoint_tm(uint32_t trow, float (&g4)[S::NA][5]) {
  static_assert(S::FOURBODY && S::NLM == 24, "teacher shape");
  float s2[S::NA][5];
#pragma unroll
  for (int k = 0; k < S::NLM / TMEM_W; ++k) {
    if (!(k < 2 || (SOLID && k == 5))) continue;
    float sv[S::NA][TMEM_W];
    tm_load<S>(trow, k, sv);
#pragma unroll
    for (int cc = 0; cc < TMEM_W; ++cc) {
      const int lm = TMEM_W * k + cc;
      const int m2 = SOLID ? solid_quadrupole(S::NLM, lm) : (lm >= 3 && lm < 8 ? lm - 3 : -1);
      if (m2 >= 0) {
#pragma unroll
        for (int a = 0; a < S::NA; ++a) s2[a][m2 < 0 ? 0 : m2] = SOLID ? solid_norm(S::NLM, lm) * sv[a][cc] : sv[a][cc];
      }
    }
  }
  FourBody<S> T;
  float q[S::NDES];
  fourbody_tensors<S>(s2, T, q);
#pragma unroll
  for (int a = 0; a < S::NA; ++a) fourbody_adjoint<S>(a, T, g4[a]);
}

// The adjoint of components c..c+3 of channel a, gl = 2 Fp_{a,l} s + (4-body terms for l = 2), as
// adjoint_channel; g4 = fourbody_adjoint of channel a.
// SOLID: sv holds s' (sums over the solid harmonics) and the row is G' = norm G, the weights of the solid
// harmonics: G' = 2 norm^2 Fp s' + norm f4 g4.
template <class S, bool SOLID = false>
__device__ __forceinline__ void adjoint_chunk(int a, int c, const float (&sv)[TMEM_W], const float (&g4)[5],
                                              const float (&Fp)[S::NDES], float (&gl)[TMEM_W]) {
#pragma unroll
  for (int cc = 0; cc < TMEM_W; ++cc) {
    const int lm = c + cc;
    const float h = SOLID ? solid_norm(S::NLM, lm) : 1.f;
    gl[cc] = (2.f * h * h) * Fp[S::NR + a * S::LMAX + (SOLID ? solid_l(S::NLM, lm) : lm_l(lm)) - 1] * sv[cc];
    const int m2 = SOLID ? solid_quadrupole(S::NLM, lm) : (lm >= 3 && lm < 8 ? lm - 3 : -1);
    if (S::FOURBODY && m2 >= 0)
      gl[cc] = fmaf(h * Fp[S::NR + S::NA * S::LMAX + a], g4[m2 < 0 ? 0 : m2], gl[cc]);
  }
}

// ---------------------------------------------------------------------------------------------------
// The network with W0 staged in shared memory: rows of S::NDES weights padded to NDP (a multiple of 4)
// so that each is read with 16-byte broadcast loads (all lanes read the same address), and the forward
// and backward products of a neuron run in float2 pairs over the descriptors.  Same result as network()
// up to the order of the additions.
template <class S>
struct NetSmem {
  static constexpr int NDP = (S::NDES + 3) / 4 * 4;
  float W0[S::NNEU][NDP];
};
template <class MT, class S>
__device__ __forceinline__ void stage_network(const Model<S> &P, NetSmem<S> &N) {
  for (int t = threadIdx.x; t < S::NNEU * NetSmem<S>::NDP; t += blockDim.x) {
    const int mu = t / NetSmem<S>::NDP, v = t % NetSmem<S>::NDP;
    N.W0[mu][v] = v < S::NDES ? round_to<MT>(P.W0[mu][v]) : 0.f;
  }
}
template <class MT, class S>
__device__ __forceinline__ float network_smem(const Model<S> &P, const NetSmem<S> &N, const float (&q)[S::NDES],
                                              bool flagged, float (&Fp)[S::NDES]) {
  constexpr int NDP = NetSmem<S>::NDP, NP = NDP / 2;
  float2 qt[NP], dq[NP];
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    const int v0 = 2 * p, v1 = 2 * p + 1;
    qt[p] = pr(v0 < S::NDES ? round_to<MT>(q[v0 < S::NDES ? v0 : 0] * P.qs[v0 < S::NDES ? v0 : 0]) : 0.f,
               v1 < S::NDES ? round_to<MT>(q[v1 < S::NDES ? v1 : 0] * P.qs[v1 < S::NDES ? v1 : 0]) : 0.f);
    dq[p] = bc2(0.f);
  }
  float U = -P.b1;
#pragma unroll 1
  for (int mu = 0; mu < S::NNEU; ++mu) {
    // the row is read twice (forward, then backward) rather than held in registers
    const float4 *row = reinterpret_cast<const float4 *>(N.W0[mu]);
    float2 z2 = pr(-P.b0[mu], 0.f);
#pragma unroll
    for (int p = 0; p < NDP / 4; ++p) {
      const float4 t = row[p];
      z2 = fma2(pr(t.x, t.y), qt[2 * p], z2);
      z2 = fma2(pr(t.z, t.w), qt[2 * p + 1], z2);
    }
    // mixed: error 2^-11, below that of z (16-bit inputs)
    const float h = std::is_same<MT, float>::value ? tanhf(hsum(z2)) : tanh_sfu(hsum(z2));
    U = fmaf(P.w1[mu], h, U);
    const float2 t2 = bc2(round_to<MT>(P.w1[mu] * (1.f - h * h)));
#pragma unroll
    for (int p = 0; p < NDP / 4; ++p) {
      const float4 t = row[p];
      dq[2 * p] = fma2(t2, pr(t.x, t.y), dq[2 * p]);
      dq[2 * p + 1] = fma2(t2, pr(t.z, t.w), dq[2 * p + 1]);
    }
  }
#pragma unroll
  for (int v = 0; v < S::NDES; ++v) {
    const float d = (v & 1) ? dq[v / 2].y : dq[v / 2].x;
    Fp[v] = flagged ? 0.f : d * P.qs[v];
  }
  return U;
}

}  // namespace nep
