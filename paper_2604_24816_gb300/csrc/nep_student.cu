// nep_student.cu -- training kernels of the student NEP (radial n_max 3, angular n_max 3, l_max 2, no
// 4-body term, 16 neurons), declared in nep_student.h.
//
// The student's descriptors are linear (radial) or quadratic (angular) in per-atom basis sums that
// depend on positions only:
//   q_n  = sum_k cR_nk Q_k,                 Q_k   = sum_j f^R_k(r_ij)
//   q_nl = sum_{m in l} s_nlm^2,  s_nlm = sum_k cA_nk S_klm,   S_klm = sum_j f^A_k(r_ij) Y_lm(u_ij)
// (the radial and angular descriptor definitions of Section III.B).  Q and S are computed once per
// training set; each training step then runs: st_forward (per atom) -> st_energy (per cell) ->
// st_force (pair gather) for the loss, and st_jvp (pair pass) -> st_grad (per atom + fixed-order
// reduction) for its gradient.
//
// Gradient of the force loss.  With v = dL/dF, sum_i v_i . F_i = -sum_i Fp_i . dq_i where
// dq_i = sum_k v_k . dq_i/dr_k is the directional derivative of the descriptors along v, so its
// parameter gradient is -d/dtheta sum_i Fp_i(theta) . dq_i(theta).  dq depends on theta through the
// expansion coefficients only: dq_n = sum_k cR_nk dQ_k, dq_nl = 2 sum_m s_nlm ds_nlm with
// ds_nlm = sum_k cA_nk dS_klm, where dQ, dS are the directional derivatives of the basis sums (st_jvp).
// For the one-hidden-layer network, J = Fp . dq = sum_mu w1_mu (1 - h_mu^2) zdot_mu with
// zdot_mu = sum_nu W0_mu,nu s_nu dq_nu, whose derivatives are written out in st_grad.
#include <cuda_runtime.h>

#include <algorithm>

#include "nep_common.cuh"
#include "nep_student.h"

namespace nep {
namespace {

using SS = StudentShape;
constexpr int KB = SS::KR;                   // basis functions (radial and angular: 8)
constexpr int NLM = SS::NLM;                 // 8 harmonics (l = 1, 2)
constexpr int NSB = SS::KA * NLM;            // 64 angular basis sums
constexpr int NR = SS::NR, NA = SS::NA, ND = SS::NDES, NN = SS::NNEU;
constexpr int OFF_CR = 0, OFF_CA = OFF_CR + NR * KB, OFF_W0 = OFF_CA + NA * KB, OFF_B0 = OFF_W0 + NN * ND,
              OFF_W1 = OFF_B0 + NN, OFF_B1 = OFF_W1 + NN, NPAR = OFF_B1 + 1;
static_assert(NPAR == ST_NPAR && ND == ST_NDES && SS::GS == ST_GS, "header constants out of date");
static_assert(SS::KR == SS::KA, "one basis size for both cutoffs");

constexpr int BLOCK = 128;
constexpr int GRAD_ATOMS = 64;               // atoms per row of partial gradients, at least (st_grad_scratch)
constexpr int GRAD_SERIAL = 32;              // atoms that one lane's float32 sums run over, at most

// The per-step kernels give each atom a group of eight lanes.  One thread per atom left a mini-batch of 40 cells
// (21,000 atoms, 165 blocks of 128 threads) at about one block per SM, each thread walking its row alone, and
// entered the angular branch for nearly every entry of the unsorted rows (some lane always has one) although two
// in five are angular.
constexpr int G = 8;
static_assert(G == KB && G == NLM, "a lane per basis function, or per harmonic component");
constexpr unsigned FULL = 0xffffffffu;

struct Cut {
  float rcR2, rcA2, inv_rcR, inv_rcA;
};
Cut cut_of(st_cutoffs rc) { return Cut{rc.rc_R * rc.rc_R, rc.rc_A * rc.rc_A, 1.f / rc.rc_R, 1.f / rc.rc_A}; }

__device__ __forceinline__ int l_of(int lm) { return lm < 3 ? 1 : 2; }

// A group's sum of v, in every lane.
__device__ __forceinline__ float group_sum(float v) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
  return v;
}
// The group's sums of 8 (4) values: lane gl gets the sum of value gl (gl & 3).
__device__ __forceinline__ float group_scatter8(const float (&v)[8], int gl) {
  float a[4], b[2];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float keep = gl & 4 ? v[4 + k] : v[k], give = gl & 4 ? v[k] : v[4 + k];
    a[k] = keep + __shfl_xor_sync(FULL, give, 4);
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const float keep = gl & 2 ? a[2 + k] : a[k], give = gl & 2 ? a[k] : a[2 + k];
    b[k] = keep + __shfl_xor_sync(FULL, give, 2);
  }
  const float keep = gl & 1 ? b[1] : b[0], give = gl & 1 ? b[0] : b[1];
  return keep + __shfl_xor_sync(FULL, give, 1);
}
__device__ __forceinline__ float group_scatter4(const float (&v)[4], int gl) {
  float b[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const float keep = gl & 2 ? v[2 + k] : v[k], give = gl & 2 ? v[k] : v[2 + k];
    b[k] = keep + __shfl_xor_sync(FULL, give, 2);
  }
  const float keep = gl & 1 ? b[1] : b[0], give = gl & 1 ? b[0] : b[1];
  const float c = keep + __shfl_xor_sync(FULL, give, 1);
  return c + __shfl_xor_sync(FULL, c, 4);
}
__device__ __forceinline__ float from_lane(float v, int src) { return __shfl_sync(FULL, v, src, G); }

// Radial functions of a set of channels as cubics (cheb_to_cubics), in shared memory.
struct Cubics {
  float inv_rcA;
  float2 gE[2][4], gO[2][4], gL[4];
};
static_assert(NR == 4 && NA == 4, "two channel pairs");
// Threads 0..3 fill R from theta's c_R, threads 4..7 A from c_A (a block barrier must follow).
__device__ __forceinline__ void stage_cubics(const float *th, Cut C, Cubics *R, Cubics *A) {
  const int t = threadIdx.x;
  if (t >= 8) return;
  Cubics &Q = t < 4 ? *R : *A;
  const int n = t & 3;
  float c[8], e[4], o[4];
#pragma unroll
  for (int k = 0; k < 8; ++k) c[k] = th[(t < 4 ? OFF_CR : OFF_CA) + n * KB + k];
  cheb_to_cubics(c, e, o);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    (&Q.gE[n >> 1][i].x)[n & 1] = e[i];
    (&Q.gO[n >> 1][i].x)[n & 1] = o[i];
  }
  if (n == 0) Q.inv_rcA = t < 4 ? C.inv_rcR : C.inv_rcA;
}

// Four consecutive floats; V4: p is 16-byte aligned.
template <bool V4>
__device__ __forceinline__ float4 load4(const float *__restrict__ p) {
  if constexpr (V4) return *reinterpret_cast<const float4 *>(p);
  else return make_float4(p[0], p[1], p[2], p[3]);
}

// A row is walked in segments of SEG entries; the angular ones of a segment are listed per atom in shared memory
// and evaluated G at a time.
constexpr int SEG = 64;
static_assert(SEG <= 256, "the lists hold bytes");

// theta (and q_scale) staged in shared memory once per block.
__device__ __forceinline__ void stage_theta(float *sth, const float *theta, float *sqs, const float *qs) {
  for (int p = threadIdx.x; p < NPAR; p += blockDim.x) sth[p] = theta[p];
  if (sqs != nullptr)
    for (int p = threadIdx.x; p < ND; p += blockDim.x) sqs[p] = qs[p];
}

// ---------------------------------------------------------------------------------------------------
__global__ void k_st_pairs(int n, const float4 *__restrict__ pos, const int *__restrict__ start,
                           const float *__restrict__ boxes, float rc2, int cap, int *__restrict__ nbr,
                           float4 *__restrict__ dvec, int *__restrict__ nnum, int *__restrict__ status) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float4 pi = pos[i];
  const int s = __float_as_int(pi.w);
  const float bx = boxes[3 * s], by = boxes[3 * s + 1], bz = boxes[3 * s + 2];
  const float ibx = 1.f / bx, iby = 1.f / by, ibz = 1.f / bz;
  const int j0 = start[s], j1 = start[s + 1];
  int c = 0;
  for (int j = j0; j < j1; ++j) {
    if (j == i) continue;
    const float4 pj = pos[j];
    float dx = pj.x - pi.x, dy = pj.y - pi.y, dz = pj.z - pi.z;
    dx -= bx * rintf(dx * ibx);
    dy -= by * rintf(dy * iby);
    dz -= bz * rintf(dz * ibz);
    if (dx * dx + dy * dy + dz * dz < rc2) {
      if (c < cap) {
        nbr[(size_t)c * n + i] = j;
        dvec[(size_t)c * n + i] = make_float4(dx, dy, dz, 0.f);
      }
      ++c;
    }
  }
  nnum[i] = min(c, cap);
  if (c > cap) atomicOr(status, ST_OVERFLOW);
}

// ---------------------------------------------------------------------------------------------------
__global__ void k_st_basis(int a0, int a1, int n, const int *__restrict__ nnum, const float4 *__restrict__ dvec,
                           Cut C, float *__restrict__ Q, float *__restrict__ S) {
  const int a = a0 + blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= a1) return;
  float q[KB], s[KB][NLM];
#pragma unroll
  for (int k = 0; k < KB; ++k) {
    q[k] = 0.f;
#pragma unroll
    for (int c = 0; c < NLM; ++c) s[k][c] = 0.f;
  }
  const int cnt = nnum[a];
  for (int e = 0; e < cnt; ++e) {
    const float4 d = dvec[(size_t)e * n + a];
    const float r2 = d.x * d.x + d.y * d.y + d.z * d.z;
    const float ir = rsqrtf(r2), r = r2 * ir;
    if (r2 < C.rcR2) {
      float f[KB];
      cheb_basis<KB>(r, C.inv_rcR, f);
#pragma unroll
      for (int k = 0; k < KB; ++k) q[k] += f[k];
    }
    if (r2 < C.rcA2) {
      float f[KB], Y[NLM];
      cheb_basis<KB>(r, C.inv_rcA, f);
      harmonics<NLM>(d.x * ir, d.y * ir, d.z * ir, Y);
#pragma unroll
      for (int k = 0; k < KB; ++k)
#pragma unroll
        for (int c = 0; c < NLM; ++c) s[k][c] = fmaf(f[k], Y[c], s[k][c]);
    }
  }
#pragma unroll
  for (int k = 0; k < KB; ++k) Q[(size_t)a * KB + k] = q[k];
#pragma unroll
  for (int k = 0; k < KB; ++k)
#pragma unroll
    for (int c = 0; c < NLM; ++c) S[(size_t)a * NSB + k * NLM + c] = s[k][c];
}

// An atom's forward pass over its eight lanes (shared by st_forward and st_grad).  Lane gl holds harmonic
// component gl of the sums, the angular descriptor (n, l) = (gl & 3, gl / 4 + 1) and the radial descriptor gl & 3,
// neurons gl and gl + 8.
struct LaneNet {
  float Sk[KB];         // S_k,gl
  float s[NA];          // s_n,gl
  float qr, qa;         // own radial and angular descriptor (unscaled)
  float qt[ND];         // all scaled descriptors
  float h[2], d1h[2];   // own neurons: tanh and 1 - tanh^2
  float U;              // site energy, without the -b1 of the sum: added (every lane)
};
__device__ __forceinline__ int own_v(int gl) { return NR + 2 * (gl & 3) + (gl >> 2); }   // index of the own angular descriptor

// Contractions with the expansion coefficients: s_n = sum_k cA_nk S_k (own component) and the own radial
// descriptor sum_k cR_nk Q_k (n = gl & 3).
__device__ __forceinline__ void contract(const float *th, const float (&Sk)[KB], float (&s)[NA]) {
#pragma unroll
  for (int n = 0; n < NA; ++n) {
    float t = 0.f;
#pragma unroll
    for (int k = 0; k < KB; ++k) t = fmaf(th[OFF_CA + n * KB + k], Sk[k], t);
    s[n] = t;
  }
}
__device__ __forceinline__ float radial_descriptor(const float *th, float Qgl, int gl) {
  float t = 0.f;
#pragma unroll
  for (int k = 0; k < KB; ++k) t = fmaf(th[OFF_CR + (gl & 3) * KB + k], from_lane(Qgl, k), t);
  return t;
}
// All ND values from the lanes' own radial and angular ones.
__device__ __forceinline__ void gather_des(float r, float a, float (&v)[ND]) {
#pragma unroll
  for (int n = 0; n < NR; ++n) v[n] = from_lane(r, n);
#pragma unroll
  for (int g = 0; g < 8; ++g) v[NR + 2 * (g & 3) + (g >> 2)] = from_lane(a, g);
}
// sum_c x_n(c) over the components of each degree: lane gl gets (n, l) = (gl & 3, gl / 4 + 1).
__device__ __forceinline__ float degree_sums(const float (&x)[NA], int gl) {
  float v[8];
#pragma unroll
  for (int n = 0; n < NA; ++n) { v[n] = gl < 3 ? x[n] : 0.f; v[4 + n] = gl < 3 ? 0.f : x[n]; }
  return group_scatter8(v, gl);
}
// sum_mu w_mu W0_mu,v over all neurons (w: the own two): the own radial and angular v, not yet scaled.
__device__ __forceinline__ void back_product(const float *th, const float (&w)[2], int gl, float &r, float &a) {
  float vr[4], va[8];
#pragma unroll
  for (int v = 0; v < ND; ++v) {
    const float t = fmaf(w[1], th[OFF_W0 + (gl + 8) * ND + v], w[0] * th[OFF_W0 + gl * ND + v]);
    if (v < NR) vr[v < NR ? v : 0] = t;
    else va[v < NR ? 0 : ((v - NR) & 1) * 4 + (v - NR) / 2] = t;
  }
  r = group_scatter4(vr, gl);
  a = group_scatter8(va, gl);
}
// One neuron's product with ND values.
__device__ __forceinline__ float neuron(const float *th, int mu, const float (&v)[ND], float z0) {
  float z = z0;
#pragma unroll
  for (int i = 0; i < ND; ++i) z = fmaf(th[OFF_W0 + mu * ND + i], v[i], z);
  return z;
}

__device__ __forceinline__ void lane_net(const float *th, const float *qs, const float *__restrict__ Q,
                                         const float *__restrict__ S, int a, int gl, LaneNet &A) {
  const float Qgl = Q[(size_t)a * KB + gl];
#pragma unroll
  for (int k = 0; k < KB; ++k) A.Sk[k] = S[(size_t)a * NSB + k * NLM + gl];
  contract(th, A.Sk, A.s);
  A.qr = radial_descriptor(th, Qgl, gl);
  float sq[NA];
#pragma unroll
  for (int n = 0; n < NA; ++n) sq[n] = A.s[n] * A.s[n];
  A.qa = degree_sums(sq, gl);
  gather_des(qs[gl & 3] * A.qr, qs[own_v(gl)] * A.qa, A.qt);
  float u = 0.f;
#pragma unroll
  for (int m = 0; m < 2; ++m) {
    const int mu = gl + 8 * m;
    const float h = tanhf(neuron(th, mu, A.qt, -th[OFF_B0 + mu]));
    A.h[m] = h;
    A.d1h[m] = 1.f - h * h;
    u = fmaf(th[OFF_W1 + mu], h, u);
  }
  A.U = group_sum(u) - th[OFF_B1];
}

__global__ void __launch_bounds__(BLOCK)
k_st_forward(int a0, int a1, const float *__restrict__ theta, const float *__restrict__ qscale,
             const float *__restrict__ Q, const float *__restrict__ S, float *__restrict__ Uo,
             float *__restrict__ Gr, float *__restrict__ qout) {
  __shared__ float th[NPAR], qs[ND];
  stage_theta(th, theta, qs, qscale);
  __syncthreads();
  const int gl = threadIdx.x % G;
  const int at = a0 + (int)((blockIdx.x * BLOCK + threadIdx.x) / G);
  const bool live = at < a1;
  const int a = live ? at : a1 - 1;                    // lanes past the last atom repeat it and store nothing
  LaneNet A;
  lane_net(th, qs, Q, S, a, gl, A);
  const float t[2] = {th[OFF_W1 + gl] * A.d1h[0], th[OFF_W1 + gl + 8] * A.d1h[1]};
  float fr, fa;
  back_product(th, t, gl, fr, fa);
  fr *= qs[gl & 3];
  fa *= qs[own_v(gl)];
  float Fp[NA];                                        // dU/dq of (n, l(gl))
#pragma unroll
  for (int n = 0; n < NA; ++n) Fp[n] = from_lane(fa, (l_of(gl) - 1) * 4 + n);
  if (!live) return;
  if (gl == 0) Uo[a] = A.U;
  float *g = Gr + (size_t)a * SS::GS;
#pragma unroll
  for (int n = 0; n < NA; ++n) g[n * NLM + gl] = 2.f * Fp[n] * A.s[n];
  g[NA * NLM + gl] = gl < NR ? fr : 0.f;
  if (qout != nullptr) {
    if (gl < NR) qout[(size_t)a * ND + gl] = A.qr;
    qout[(size_t)a * ND + own_v(gl)] = A.qa;
  }
}

// One warp per cell: lanes stride over its atoms, float64 sums combined by a fixed shuffle tree.
__global__ void k_st_energy(int s0, int s1, const int *__restrict__ start, const float *__restrict__ U,
                            double *__restrict__ E) {
  const int s = s0 + (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (s >= s1) return;
  double t = 0.0;
  for (int a = start[s] + lane; a < start[s + 1]; a += 32) t += (double)U[a];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
  if (lane == 0) E[s] = t;
}

// ---------------------------------------------------------------------------------------------------
// F_i = sum_j D_ij, D_ij = dU_i/dd_ij - dU_j/dd_ji: radial part (Fp_i + Fp_j) . g'(r) u, angular part
// with H_nlm = G^i_nlm + (-1)^l G^j_nlm contracted with grad_d [g^A_n(r) Y_lm(d/r)].
// Angular pairs are prepared one per lane (channel functions and direction, staged in shared memory) and evaluated
// by the whole group, lane gl taking component gl: it keeps its four values of the own row, reads the neighbour's as
// one coalesced 32-byte sector per channel, and forms its share of the force, which is linear in the components.
// Y_c = m.u (l = 1) or u.M u (l = 2), so with the lane's constants K u + k = grad Y_c, and u . grad Y_c = l Y_c.
// The kernel waits on its gathers (long scoreboard 9 of 14 cycles per issue, issue slots 31 % busy before): entries
// are loaded a step ahead, neighbours' rows four pairs at a time.  103,000 atoms: 104 us (157 with one thread per
// atom, 144 with whole pairs per lane, which gathered 128-byte rows from 32 places at once, 134 before the loads were
// moved ahead); 21,000 atoms: 24 us (55).  Six resident blocks; five to eight differ by 5 %, and a loop of resident
// blocks over the atoms measured 3 % slower.
constexpr int ATOMS = BLOCK / G;

template <bool V4>
__global__ void __launch_bounds__(BLOCK, 6)
k_st_force(int a0, int a1, int n, const int *__restrict__ nbr, const float4 *__restrict__ dvec,
           const int *__restrict__ nnum, Cut C, const float *__restrict__ theta,
           const float *__restrict__ Gr, float *__restrict__ F) {
  constexpr int ROW = 20, GRP = G * ROW + 8;           // {g[4] | g'[4] | u, 1/r | j}; groups eight banks apart
  __shared__ Cubics R, A;
  __shared__ uint8_t list[ATOMS][SEG];
  __shared__ __align__(16) float stage[ATOMS * GRP];
  stage_cubics(theta, C, &R, &A);
  __syncthreads();
  const int lane = threadIdx.x & 31, gl = lane % G, grp = lane / G;
  const int at = a0 + (int)((blockIdx.x * BLOCK + threadIdx.x) / G);
  const bool live = at < a1;
  const int a = live ? at : a1 - 1;
  const int cnt = live ? nnum[a] : 0;
  const float *Ga = Gr + (size_t)a * SS::GS;
  uint8_t *L = list[threadIdx.x / G];
  float *sg = stage + (threadIdx.x / G) * GRP;
  const float4 fi = load4<V4>(Ga + NA * NLM);
  float gi[NA];
#pragma unroll
  for (int nn = 0; nn < NA; ++nn) gi[nn] = Ga[nn * NLM + gl];
  // grad Y of the own component: (kx + xx ux + xy uy + xz uz, ...), symmetric; sgn = (-1)^l, il = 1 / l
  const float s3 = 1.7320508075688772f;
  const float kx = gl == 2 ? 1.f : 0.f, ky = gl == 0 ? 1.f : 0.f, kz = gl == 1 ? 1.f : 0.f;
  const float xx = gl == 5 ? -1.f : (gl == 7 ? s3 : 0.f), yy = gl == 5 ? -1.f : (gl == 7 ? -s3 : 0.f);
  const float zz = gl == 5 ? 2.f : 0.f, xy = gl == 3 ? s3 : 0.f, yz = gl == 4 ? s3 : 0.f, xz = gl == 6 ? s3 : 0.f;
  const float sgn = gl < 3 ? -1.f : 1.f, il = gl < 3 ? 1.f : 0.5f;
  float fx = 0.f, fy = 0.f, fz = 0.f;
  const int most = __reduce_max_sync(FULL, cnt);
  const float4 none = make_float4(1e15f, 0.f, 0.f, 0.f);         // past the row: outside every cutoff
  for (int seg = 0; seg < most; seg += SEG) {
    int na = 0;
    // entries one step ahead, the neighbour's radial adjoint requested before its distance is known
    float4 d = seg + gl < cnt ? dvec[(size_t)(seg + gl) * n + a] : none;
    int j = seg + gl < cnt ? nbr[(size_t)(seg + gl) * n + a] : a;
    for (int it = 0; it < SEG && seg + it < most; it += G) {
      const int e1 = seg + it + G + gl;
      const bool more = it + G < SEG && e1 < cnt;
      const float4 fj = load4<V4>(Gr + (size_t)j * SS::GS + NA * NLM);
      const float4 d1 = more ? dvec[(size_t)e1 * n + a] : none;
      const int j1 = more ? nbr[(size_t)e1 * n + a] : a;
      const float r2 = d.x * d.x + d.y * d.y + d.z * d.z;
      if (r2 < C.rcR2) {
        const float ir = rsqrtf(r2), r = r2 * ir;
        float g[NR], dg[NR];
        radial_channels_d<SS>(R, r, g, dg);
        const float2 c2 = fma2(add2(pr(fi.x, fi.y), pr(fj.x, fj.y)), pr(dg[0], dg[1]),
                               mul2(add2(pr(fi.z, fi.w), pr(fj.z, fj.w)), pr(dg[2], dg[3])));
        const float coef = hsum(c2) * ir;
        fx = fmaf(coef, d.x, fx); fy = fmaf(coef, d.y, fy); fz = fmaf(coef, d.z, fz);
      }
      const bool ang = r2 < C.rcA2;
      const unsigned m = (__ballot_sync(FULL, ang) >> (grp * G)) & 0xffu;
      if (ang) L[na + __popc(m & ((1u << gl) - 1u))] = (uint8_t)(it + gl);
      na += __popc(m);
      d = d1; j = j1;
    }
    __syncwarp();
    const int chunks = __reduce_max_sync(FULL, (na + G - 1) / G);
    for (int ch = 0; ch < chunks; ++ch) {
      const int p = ch * G + gl;
      // one pair per lane; a row without a pair is zero and points at the atom itself
      float4 *mine = reinterpret_cast<float4 *>(sg + gl * ROW);
      int jp = a;
      if (p < na) {
        const int e = seg + L[p];
        const float4 dp = dvec[(size_t)e * n + a];
        jp = nbr[(size_t)e * n + a];
        const float r2 = dp.x * dp.x + dp.y * dp.y + dp.z * dp.z;
        const float ir = rsqrtf(r2), r = r2 * ir;
        float g[NA], dg[NA];
        radial_channels_d<SS>(A, r, g, dg);
        mine[0] = make_float4(g[0], g[1], g[2], g[3]);
        mine[1] = make_float4(dg[0], dg[1], dg[2], dg[3]);
        mine[2] = make_float4(dp.x * ir, dp.y * ir, dp.z * ir, ir);
      } else {
        mine[0] = mine[1] = mine[2] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
      sg[gl * ROW + 12] = __int_as_float(jp);
      __syncwarp();
      const int m = __reduce_max_sync(FULL, min(G, na - ch * G));
      // four pairs at a time: sixteen loads of neighbours' rows in flight per lane
      for (int i0 = 0; i0 < m; i0 += 4) {
#pragma unroll
        for (int i = i0; i < i0 + 4; ++i) {
          const float4 *row = reinterpret_cast<const float4 *>(sg + i * ROW);
          const float *Gj = Gr + (size_t)__float_as_int(sg[i * ROW + 12]) * SS::GS + gl;
          const float4 g = row[0], dg = row[1], u = row[2];
          const float h0 = fmaf(sgn, Gj[0], gi[0]), h1 = fmaf(sgn, Gj[NLM], gi[1]);
          const float h2 = fmaf(sgn, Gj[2 * NLM], gi[2]), h3 = fmaf(sgn, Gj[3 * NLM], gi[3]);
          const float av = fmaf(h0, dg.x, fmaf(h1, dg.y, fmaf(h2, dg.z, h3 * dg.w)));
          const float bv = u.w * fmaf(h0, g.x, fmaf(h1, g.y, fmaf(h2, g.z, h3 * g.w)));      // B / r
          const float gx = fmaf(xx, u.x, fmaf(xy, u.y, fmaf(xz, u.z, kx)));
          const float gy = fmaf(xy, u.x, fmaf(yy, u.y, fmaf(yz, u.z, ky)));
          const float gz = fmaf(xz, u.x, fmaf(yz, u.y, fmaf(zz, u.z, kz)));
          const float ug = fmaf(u.x, gx, fmaf(u.y, gy, u.z * gz));                           // l Y
          const float w = ug * fmaf(av, il, -bv);
          fx = fmaf(w, u.x, fmaf(bv, gx, fx));
          fy = fmaf(w, u.y, fmaf(bv, gy, fy));
          fz = fmaf(w, u.z, fmaf(bv, gz, fz));
        }
      }
      __syncwarp();                                    // read before the next pairs (and lists) replace them
    }
  }
  fx = group_sum(fx); fy = group_sum(fy); fz = group_sum(fz);
  if (live && gl < 3) F[3 * (size_t)a + gl] = gl == 0 ? fx : (gl == 1 ? fy : fz);
}

// ---------------------------------------------------------------------------------------------------
// dQ_k = sum_j f^R_k'(r) (u . w),  dS_klm = sum_j [f^A_k'(r) Y_lm (u . w) + f^A_k(r) (grad P_lm(u) . w
// - l Y_lm (u . w)) / r],  w = v_j - v_i: the change of the basis sums when every atom moves along v.
// Angular pairs are evaluated one per lane and staged in shared memory (f_k, f_k', and the two factors per
// component); lane gl then adds them for its component.
__global__ void __launch_bounds__(BLOCK)
k_st_jvp(int a0, int a1, int n, const int *__restrict__ nbr, const float4 *__restrict__ dvec,
         const int *__restrict__ nnum, Cut C, const float *__restrict__ v, float *__restrict__ dQ,
         float *__restrict__ dS) {
  constexpr int ROW = 4 * KB + 4, GRP = G * ROW + 8;   // 16-byte rows; groups eight banks apart
  __shared__ uint8_t list[ATOMS][SEG];
  __shared__ __align__(16) float stage[ATOMS * GRP];
  const int lane = threadIdx.x & 31, gl = lane % G, grp = lane / G;
  const int at = a0 + (int)((blockIdx.x * BLOCK + threadIdx.x) / G);
  const bool live = at < a1;
  const int a = live ? at : a1 - 1;
  const int cnt = live ? nnum[a] : 0;
  uint8_t *L = list[threadIdx.x / G];
  float *sg = stage + (threadIdx.x / G) * GRP;
  const float vax = v[3 * (size_t)a], vay = v[3 * (size_t)a + 1], vaz = v[3 * (size_t)a + 2];
  float2 q[4], s[4];
  float qa = 0.f;                                      // the T_k-independent part of every dQ_k
#pragma unroll
  for (int k = 0; k < 4; ++k) { q[k] = bc2(0.f); s[k] = bc2(0.f); }
  const int most = __reduce_max_sync(FULL, cnt);
  for (int seg = 0; seg < most; seg += SEG) {
    int na = 0;
    for (int it = 0; it < SEG && seg + it < most; it += G) {
      const int e = seg + it + gl;
      const bool ok = e < cnt;
      float r2 = 1e30f;
      if (ok) {
        const float4 d = dvec[(size_t)e * n + a];
        r2 = d.x * d.x + d.y * d.y + d.z * d.z;
        if (r2 < C.rcR2) {
          const size_t j = 3 * (size_t)nbr[(size_t)e * n + a];
          const float wx = v[j] - vax, wy = v[j + 1] - vay, wz = v[j + 2] - vaz;
          const float ir = rsqrtf(r2), r = r2 * ir;
          const float uw = (d.x * wx + d.y * wy + d.z * wz) * ir;
          // f_k' = dh + T_k dh + T_k' dxh; the pairs (T_2m, T_2m+1) and their derivatives by the step-two recurrence
          float h, dh, dxh, x, y;
          cheb_args_d(r, C.inv_rcR, h, dh, dxh, x, y);
          const float2 y2 = bc2(y + y), x8 = bc2(8.f * x), ta = bc2(uw * dh), tb = bc2(uw * dxh);
          const float2 t01 = pr(1.f, x), t23 = pr(y, fmaf(y2.x, x, -x));
          const float2 t45 = fma2(y2, t23, pr(-t01.x, -t01.y)), t67 = fma2(y2, t45, pr(-t23.x, -t23.y));
          const float2 d01 = pr(0.f, 1.f), d23 = pr(4.f * x, fmaf(6.f, y, 3.f));
          const float2 d45 = fma2(y2, d23, fma2(x8, t23, pr(0.f, -1.f)));
          const float2 d67 = fma2(y2, d45, fma2(x8, t45, pr(-d23.x, -d23.y)));
          qa += ta.x;
          q[0] = fma2(ta, t01, fma2(tb, d01, q[0]));
          q[1] = fma2(ta, t23, fma2(tb, d23, q[1]));
          q[2] = fma2(ta, t45, fma2(tb, d45, q[2]));
          q[3] = fma2(ta, t67, fma2(tb, d67, q[3]));
        }
      }
      const bool ang = ok && r2 < C.rcA2;
      const unsigned m = (__ballot_sync(FULL, ang) >> (grp * G)) & 0xffu;
      if (ang) L[na + __popc(m & ((1u << gl) - 1u))] = (uint8_t)(it + gl);
      na += __popc(m);
    }
    __syncwarp();
    const int chunks = __reduce_max_sync(FULL, (na + G - 1) / G);
    for (int ch = 0; ch < chunks; ++ch) {
      const int p = ch * G + gl;
      if (p < na) {
        const int e = seg + L[p];
        const float4 d = dvec[(size_t)e * n + a];
        const size_t j = 3 * (size_t)nbr[(size_t)e * n + a];
        const float wx = v[j] - vax, wy = v[j + 1] - vay, wz = v[j + 2] - vaz;
        const float r2 = d.x * d.x + d.y * d.y + d.z * d.z;
        const float ir = rsqrtf(r2), r = r2 * ir;
        const float ux = d.x * ir, uy = d.y * ir, uz = d.z * ir;
        const float uw = ux * wx + uy * wy + uz * wz;
        float f[KB], df[KB], Y[NLM], t1[NLM], t2[NLM];
        cheb_basis_d<KB>(r, C.inv_rcA, f, df);
        harmonics<NLM>(ux, uy, uz, Y);
#pragma unroll
        for (int c = 0; c < NLM; ++c) {
          float gx = 0.f, gy = 0.f, gz = 0.f;
          harmonic_grad_acc(c, ux, uy, uz, 1.f, gx, gy, gz);
          t1[c] = Y[c] * uw;
          t2[c] = (gx * wx + gy * wy + gz * wz - (float)(c < 3 ? 1 : 2) * t1[c]) * ir;
        }
        float4 *row = reinterpret_cast<float4 *>(sg + gl * ROW);
        row[0] = make_float4(f[0], f[1], f[2], f[3]);
        row[1] = make_float4(f[4], f[5], f[6], f[7]);
        row[2] = make_float4(df[0], df[1], df[2], df[3]);
        row[3] = make_float4(df[4], df[5], df[6], df[7]);
        row[4] = make_float4(t1[0], t1[1], t1[2], t1[3]);
        row[5] = make_float4(t1[4], t1[5], t1[6], t1[7]);
        row[6] = make_float4(t2[0], t2[1], t2[2], t2[3]);
        row[7] = make_float4(t2[4], t2[5], t2[6], t2[7]);
      }
      __syncwarp();
      const int m = min(G, na - ch * G);               // group-uniform
      for (int i = 0; i < m; ++i) {
        const float4 *row = reinterpret_cast<const float4 *>(sg + i * ROW);
        const float4 f0 = row[0], f1 = row[1], e0 = row[2], e1 = row[3];
        const float2 t1 = bc2(sg[i * ROW + 2 * KB + gl]), t2 = bc2(sg[i * ROW + 3 * KB + gl]);
        s[0] = fma2(pr(e0.x, e0.y), t1, fma2(pr(f0.x, f0.y), t2, s[0]));
        s[1] = fma2(pr(e0.z, e0.w), t1, fma2(pr(f0.z, f0.w), t2, s[1]));
        s[2] = fma2(pr(e1.x, e1.y), t1, fma2(pr(f1.x, f1.y), t2, s[2]));
        s[3] = fma2(pr(e1.z, e1.w), t1, fma2(pr(f1.z, f1.w), t2, s[3]));
      }
      __syncwarp();                                    // read before the next pairs replace them
    }
  }
  float qv[8];
#pragma unroll
  for (int k = 0; k < 4; ++k) { qv[2 * k] = q[k].x + qa; qv[2 * k + 1] = q[k].y + qa; }
  const float mine = group_scatter8(qv, gl);
  if (!live) return;
  dQ[(size_t)a * KB + gl] = mine;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    dS[(size_t)a * NSB + (2 * k) * NLM + gl] = s[k].x;
    dS[(size_t)a * NSB + (2 * k + 1) * NLM + gl] = s[k].y;
  }
}

// ---------------------------------------------------------------------------------------------------
// Parameter gradient.  Per atom (U = network output, J = Fp . dq, both functions of theta):
//   dL/dtheta += gE dU/dtheta - dJ/dtheta.
// With qt = s (.) q, u = s (.) dq, zdot = W0 u, h = tanh(z), Fp = s (.) W0^T (w1 (.) (1 - h^2)),
// R = dJ/dq (at fixed dq) = s (.) W0^T (-2 w1 (.) zdot (.) h (.) (1 - h^2)):
//   W0_mu,nu : alpha_mu qt_nu + beta_mu u_nu,   alpha = w1 (1-h^2)(gE + 2 h zdot),  beta = -w1 (1-h^2)
//   b0_mu    : -alpha_mu
//   w1_mu    : gE h_mu - (1 - h_mu^2) zdot_mu
//   b1       : -gE
//   cR_nk    : rho_n Q_k + sigma_n dQ_k,        rho = gE Fp - R (radial), sigma = -Fp (radial)
//   cA_nk    : sum_lm kappa_nlm S_klm + lambda_nlm dS_klm,
//              kappa = 2 (gE Fp_nl - R_nl) s_nlm - 2 Fp_nl ds_nlm,  lambda = -2 Fp_nl s_nlm.
// Eight lanes hold these factors of an atom: lane gl its harmonic component of S, dS, kappa and lambda, neurons gl
// and gl + 8, and k = gl of Q and dQ.  So every lane adds its own 65 products (32 of cA's from its component, 24 of
// W0, 4 of cR, 2 of b0 and of w1, b1) in registers over the atoms of its group, and only the block's totals go
// through shared memory, in a fixed order.  (Records of 289 floats per atom in shared memory, read back for every
// product, held 6 warps per SM and took 34 us for 21,000 atoms.)  Block rows are summed by k_st_grad_reduce in
// float64 in a fixed order, and there are enough of them that no float32 sum runs over more than
// GRAD_SERIAL atoms: equal atoms are off by 1.8e-7 for 21,000 and 5.6e-7 for a million or twelve (9.7e-7 with one record
// per atom and rows of 64; 9.1e-6 for twelve million with never more than four rows per SM).
constexpr int GRAD_BLOCK = 256;
constexpr int GRAD_WARPS = GRAD_BLOCK / 32;

__global__ void __launch_bounds__(GRAD_BLOCK)
k_st_grad(int a0, int a1, const float *__restrict__ theta, const float *__restrict__ qscale,
          const float4 *__restrict__ pos, const float *__restrict__ Q, const float *__restrict__ S,
          const float *__restrict__ dQ, const float *__restrict__ dS, const double *__restrict__ gE,
          float *__restrict__ part) {
  __shared__ float th[NPAR], qs[ND];
  __shared__ float tot[GRAD_WARPS][NPAR];
  stage_theta(th, theta, qs, qscale);
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, gl = lane % G;
  float2 cA[NA][KB / 2], w0[2][ND / 2];
  float cR[NR] = {0.f, 0.f, 0.f, 0.f}, b0[2] = {0.f, 0.f}, w1[2] = {0.f, 0.f}, b1 = 0.f;
#pragma unroll
  for (int i = 0; i < NA; ++i)
#pragma unroll
    for (int k = 0; k < KB / 2; ++k) cA[i][k] = bc2(0.f);
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int k = 0; k < ND / 2; ++k) w0[i][k] = bc2(0.f);
  const int first = (int)((blockIdx.x * GRAD_BLOCK + threadIdx.x) / G), per_pass = (int)(gridDim.x * GRAD_BLOCK / G);
  const int m = a1 - a0, trips = (m + per_pass - 1) / per_pass;   // grid-uniform: every lane takes part in the shuffles
  for (int it = 0; it < trips; ++it) {
    const int i = first + it * per_pass;
    const bool live = i < m;
    const int a = live ? a0 + i : a1 - 1;
    LaneNet A;
    lane_net(th, qs, Q, S, a, gl, A);
    const float ge = live ? (float)gE[__float_as_int(pos[a].w)] : 0.f;
    const float on = live ? 1.f : 0.f;                 // lanes past the last atom add zeros
    // directional derivatives of the descriptors
    float dSk[KB], ds[NA], x[NA], u[ND];
    const float Qk = Q[(size_t)a * KB + gl], dQk = dQ[(size_t)a * KB + gl];
#pragma unroll
    for (int k = 0; k < KB; ++k) dSk[k] = dS[(size_t)a * NSB + k * NLM + gl];
    contract(th, dSk, ds);
#pragma unroll
    for (int n = 0; n < NA; ++n) x[n] = 2.f * A.s[n] * ds[n];
    gather_des(qs[gl & 3] * radial_descriptor(th, dQk, gl), qs[own_v(gl)] * degree_sums(x, gl), u);
    // neurons: t = w1 (1 - h^2) gives Fp; c = gE t + 2 w1 zd h (1 - h^2) gives rho = gE Fp - R and alpha
    float t[2], c[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int mu = gl + 8 * k;
      const float zd = neuron(th, mu, u, 0.f);
      t[k] = th[OFF_W1 + mu] * A.d1h[k] * on;
      c[k] = t[k] * (ge + 2.f * A.h[k] * zd);
      b0[k] -= c[k];
      w1[k] += on * (ge * A.h[k] - A.d1h[k] * zd);
#pragma unroll
      for (int v = 0; v < ND / 2; ++v)
        w0[k][v] = fma2(bc2(c[k]), pr(A.qt[2 * v], A.qt[2 * v + 1]),
                        fma2(bc2(-t[k]), pr(u[2 * v], u[2 * v + 1]), w0[k][v]));
    }
    b1 -= ge;
    float fr, fa, rr, ra;
    back_product(th, t, gl, fr, fa);
    back_product(th, c, gl, rr, ra);
    fr *= qs[gl & 3]; rr *= qs[gl & 3];
    fa *= qs[own_v(gl)]; ra *= qs[own_v(gl)];
#pragma unroll
    for (int n = 0; n < NR; ++n) cR[n] = fmaf(from_lane(rr, n), Qk, fmaf(-from_lane(fr, n), dQk, cR[n]));
#pragma unroll
    for (int n = 0; n < NA; ++n) {
      const int src = (l_of(gl) - 1) * 4 + n;
      const float Fp = from_lane(fa, src), rho = from_lane(ra, src);
      const float kap = 2.f * rho * A.s[n] - 2.f * Fp * ds[n], lam = -2.f * Fp * A.s[n];
#pragma unroll
      for (int k = 0; k < KB / 2; ++k)
        cA[n][k] = fma2(bc2(kap), pr(A.Sk[2 * k], A.Sk[2 * k + 1]),
                        fma2(bc2(lam), pr(dSk[2 * k], dSk[2 * k + 1]), cA[n][k]));
    }
  }
  // the warp's totals: over its four groups, and for cA over the eight components too
  auto groups = [](float v) {
    v += __shfl_xor_sync(FULL, v, 8);
    return v + __shfl_xor_sync(FULL, v, 16);
  };
  float *T = tot[warp];
#pragma unroll
  for (int n = 0; n < NA; ++n) {
    float v[8];
#pragma unroll
    for (int k = 0; k < KB / 2; ++k) { v[2 * k] = cA[n][k].x; v[2 * k + 1] = cA[n][k].y; }
    const float r = groups(group_scatter8(v, gl));     // k = gl
    const float q = groups(cR[n]);
    if (lane < G) {
      T[OFF_CA + n * KB + gl] = r;
      T[OFF_CR + n * KB + gl] = q;
    }
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int mu = gl + 8 * k;
#pragma unroll
    for (int v = 0; v < ND; ++v) {
      const float r = groups(v & 1 ? w0[k][v / 2].y : w0[k][v / 2].x);
      if (lane < G) T[OFF_W0 + mu * ND + v] = r;
    }
    const float rb = groups(b0[k]), rw = groups(w1[k]);
    if (lane < G) {
      T[OFF_B0 + mu] = rb;
      T[OFF_W1 + mu] = rw;
    }
  }
  b1 = groups(b1);
  if (lane == 0) T[OFF_B1] = b1;
  __syncthreads();
  for (int p = threadIdx.x; p < NPAR; p += GRAD_BLOCK) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < GRAD_WARPS; ++w) s += tot[w][p];
    part[(size_t)blockIdx.x * NPAR + p] = s;
  }
}

// One warp per parameter: the lanes stride over the block rows in float64, then a fixed shuffle tree.  (One thread
// per parameter took 30 us for 330 rows.)
__global__ void k_st_grad_reduce(int nblk, const float *__restrict__ part, float *__restrict__ grad) {
  const int p = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (p >= NPAR) return;
  double t = 0.0;
  for (int b = lane; b < nblk; b += 32) t += (double)part[(size_t)b * NPAR + p];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(FULL, t, o);
  if (lane == 0) grad[p] = (float)t;
}

// Loss w_E mean_s ((E_s - E*_s) / n_s)^2 + w_F mean (F - F*)^2 over force components: block sums in float64 (weights
// and means applied), then one block adds them.  Differences of forces in float32, squares and sums in float64.
// keep (or nullptr): what the gradient is formed from later, whatever becomes of the labels, {(E - E*) / n^2 [nc] |
// 1 / n^2 [nc] | F - F* [nf]} (st_loss_keep).
constexpr int LOSS_BLOCK = 256, LOSS_BLOCKS = 128;
template <int NT>
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double w[NT / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(FULL, v, o);
  if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int k = 0; k < NT / 32; ++k) t += w[k];
  return t;
}
__global__ void __launch_bounds__(LOSS_BLOCK)
k_st_loss(int nc, int nf, const double *__restrict__ E, const double *__restrict__ Er, const double *__restrict__ na,
          const float *__restrict__ F, const float *__restrict__ Fr, double wE, double wF, double *__restrict__ keep,
          double *__restrict__ part) {
  const int t = blockIdx.x * LOSS_BLOCK + threadIdx.x, stride = gridDim.x * LOSS_BLOCK;
  double e = 0.0, f = 0.0;
  for (int s = t; s < nc; s += stride) {
    const double d = (E[s] - Er[s]) / na[s];
    if (keep != nullptr) {
      keep[s] = d / na[s];
      keep[nc + s] = 1.0 / (na[s] * na[s]);
    }
    e = fma(d, d, e);
  }
  for (int k = t; k < nf; k += stride) {
    const double d = (double)(F[k] - Fr[k]);
    if (keep != nullptr) keep[2 * (size_t)nc + k] = d;
    f = fma(d, d, f);
  }
  const double v = block_sum<LOSS_BLOCK>(e * (wE / nc) + f * (wF / nf));
  if (threadIdx.x == 0) part[blockIdx.x] = v;
}
__global__ void __launch_bounds__(LOSS_BLOCKS)
k_st_loss_sum(int nb, const double *__restrict__ part, double *__restrict__ loss) {
  const double v = block_sum<LOSS_BLOCKS>((int)threadIdx.x < nb ? part[threadIdx.x] : 0.0);
  if (threadIdx.x == 0) *loss = v;
}
// Its gradients times the upstream derivative *g, from what k_st_loss kept or (keep nullptr) from E, F and the labels.
__global__ void __launch_bounds__(LOSS_BLOCK)
k_st_loss_grad(int nc, int nf, const double *__restrict__ keep, const double *__restrict__ E, const double *__restrict__ Er,
               const double *__restrict__ na, const float *__restrict__ F, const float *__restrict__ Fr, double wE,
               double wF, const double *__restrict__ g, double *__restrict__ gE, float *__restrict__ gF) {
  const int t = blockIdx.x * LOSS_BLOCK + threadIdx.x, stride = gridDim.x * LOSS_BLOCK;
  const double up = *g, ce = 2.0 * up * wE / nc, cf = 2.0 * up * wF / nf;
  for (int s = t; s < nc; s += stride) gE[s] = ce * (keep != nullptr ? keep[s] : (E[s] - Er[s]) / na[s] / na[s]);
  for (int k = t; k < nf; k += stride)
    gF[k] = (float)(cf * (keep != nullptr ? keep[2 * (size_t)nc + k] : (double)(F[k] - Fr[k])));
}

__global__ void k_st_adam(int npar, float *__restrict__ theta, const float *__restrict__ grad, float *__restrict__ m,
                          float *__restrict__ v, float lr, float b1, float b2, float eps, float c1, float c2) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= npar) return;
  const float g = grad[p];
  const float mp = b1 * m[p] + (1.f - b1) * g;
  const float vp = b2 * v[p] + (1.f - b2) * g * g;
  m[p] = mp;
  v[p] = vp;
  theta[p] -= lr * (mp / c1) / (sqrtf(vp / c2) + eps);
}

int blocks_of(int n, int b) { return (n + b - 1) / b; }

}  // namespace
}  // namespace nep

using namespace nep;

extern "C" {

int st_pairs(int n, const float *pos, const int *start, const float *boxes, st_cutoffs rc, int cap, int *nbr,
             float *dvec, int *nnum, int *status, void *stream) {
  if (n <= 0) return 0;
  k_st_pairs<<<blocks_of(n, BLOCK), BLOCK, 0, (cudaStream_t)stream>>>(
      n, reinterpret_cast<const float4 *>(pos), start, boxes, rc.rc_R * rc.rc_R, cap, nbr,
      reinterpret_cast<float4 *>(dvec), nnum, status);
  return (int)cudaGetLastError();
}

int st_basis(int a0, int a1, int n, int cap, const int *nbr, const float *dvec, const int *nnum, st_cutoffs rc,
             float *Q, float *S, void *stream) {
  (void)cap; (void)nbr;
  if (a1 <= a0) return 0;
  k_st_basis<<<blocks_of(a1 - a0, BLOCK), BLOCK, 0, (cudaStream_t)stream>>>(
      a0, a1, n, nnum, reinterpret_cast<const float4 *>(dvec), cut_of(rc), Q, S);
  return (int)cudaGetLastError();
}

int st_forward(int a0, int a1, const float *theta, const float *q_scale, const float *Q, const float *S, float *U,
               float *G, float *q_out, void *stream) {
  if (a1 <= a0) return 0;
  k_st_forward<<<blocks_of(a1 - a0, ATOMS), BLOCK, 0, (cudaStream_t)stream>>>(a0, a1, theta, q_scale, Q, S, U, G,
                                                                              q_out);
  return (int)cudaGetLastError();
}

int st_energy(int s0, int s1, const int *start, const float *U, double *E, void *stream) {
  if (s1 <= s0) return 0;
  const int warps = s1 - s0;
  k_st_energy<<<blocks_of(warps * 32, BLOCK), BLOCK, 0, (cudaStream_t)stream>>>(s0, s1, start, U, E);
  return (int)cudaGetLastError();
}

int st_force(int a0, int a1, int n, int cap, const int *nbr, const float *dvec, const int *nnum, st_cutoffs rc,
             const float *theta, const float *G, float *F, void *stream) {
  (void)cap;
  if (a1 <= a0) return 0;
  // rows of 160 bytes: 16-byte loads when the array starts on a 16-byte boundary
  auto kernel = (reinterpret_cast<uintptr_t>(G) & 15) == 0 ? k_st_force<true> : k_st_force<false>;
  kernel<<<blocks_of(a1 - a0, ATOMS), BLOCK, 0, (cudaStream_t)stream>>>(
      a0, a1, n, nbr, reinterpret_cast<const float4 *>(dvec), nnum, cut_of(rc), theta, G, F);
  return (int)cudaGetLastError();
}

int st_jvp(int a0, int a1, int n, int cap, const int *nbr, const float *dvec, const int *nnum, st_cutoffs rc,
           const float *v, float *dQ, float *dS, void *stream) {
  (void)cap;
  if (a1 <= a0) return 0;
  k_st_jvp<<<blocks_of(a1 - a0, ATOMS), BLOCK, 0, (cudaStream_t)stream>>>(
      a0, a1, n, nbr, reinterpret_cast<const float4 *>(dvec), nnum, cut_of(rc), v, dQ, dS);
  return (int)cudaGetLastError();
}

int64_t st_grad_scratch(int a0, int a1) {
  return a1 > a0 ? (int64_t)blocks_of(a1 - a0, GRAD_ATOMS) * NPAR : 0;
}

int st_grad(int a0, int a1, const float *theta, const float *q_scale, const float *pos, const float *Q,
            const float *S, const float *dQ, const float *dS, const double *gE, float *scratch, float *grad,
            void *stream) {
  cudaStream_t st = (cudaStream_t)stream;
  if (a1 <= a0) return (int)cudaMemsetAsync(grad, 0, NPAR * sizeof(float), st);
  // as many rows of partial sums as the scratch holds (GRAD_ATOMS atoms each, two per group), up to four blocks per SM;
  // above 1,024 atoms for each of those, as many as keep the float32 sums at GRAD_SERIAL atoms
  const int m = a1 - a0;
  const int nblk = std::max(std::min(blocks_of(m, GRAD_ATOMS), 4 * sm_count()), blocks_of(m, GRAD_BLOCK / G * GRAD_SERIAL));
  k_st_grad<<<nblk, GRAD_BLOCK, 0, st>>>(a0, a1, theta, q_scale, reinterpret_cast<const float4 *>(pos), Q, S, dQ, dS,
                                         gE, scratch);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return (int)e;
  k_st_grad_reduce<<<blocks_of(NPAR * 32, BLOCK), BLOCK, 0, st>>>(nblk, scratch, grad);
  return (int)cudaGetLastError();
}

int64_t st_loss_scratch(void) { return LOSS_BLOCKS; }

int64_t st_loss_kept(int n_cells, int n_comp) { return 2 * (int64_t)n_cells + n_comp; }

int st_loss_keep(int n_cells, int n_comp, const double *E, const double *E_ref, const double *natoms, const float *F,
                 const float *F_ref, double w_E, double w_F, double *kept, double *scratch, double *loss, void *stream) {
  if (n_cells <= 0 || n_comp <= 0) return (int)cudaErrorInvalidValue;
  cudaStream_t st = (cudaStream_t)stream;
  const int nb = std::min(LOSS_BLOCKS, blocks_of(std::max(n_cells, n_comp), LOSS_BLOCK));
  k_st_loss<<<nb, LOSS_BLOCK, 0, st>>>(n_cells, n_comp, E, E_ref, natoms, F, F_ref, w_E, w_F, kept, scratch);
  k_st_loss_sum<<<1, LOSS_BLOCKS, 0, st>>>(nb, scratch, loss);
  return (int)cudaGetLastError();
}

int st_loss(int n_cells, int n_comp, const double *E, const double *E_ref, const double *natoms, const float *F,
            const float *F_ref, double w_E, double w_F, double *scratch, double *loss, void *stream) {
  return st_loss_keep(n_cells, n_comp, E, E_ref, natoms, F, F_ref, w_E, w_F, nullptr, scratch, loss, stream);
}

static int loss_grad(int n_cells, int n_comp, const double *kept, const double *E, const double *E_ref,
                     const double *natoms, const float *F, const float *F_ref, double w_E, double w_F, const double *g,
                     double *gE, float *gF, void *stream) {
  if (n_cells <= 0 || n_comp <= 0) return (int)cudaErrorInvalidValue;
  k_st_loss_grad<<<std::min(8 * sm_count(), blocks_of(std::max(n_cells, n_comp), LOSS_BLOCK)), LOSS_BLOCK, 0,
                   (cudaStream_t)stream>>>(n_cells, n_comp, kept, E, E_ref, natoms, F, F_ref, w_E, w_F, g, gE, gF);
  return (int)cudaGetLastError();
}

int st_loss_grad(int n_cells, int n_comp, const double *E, const double *E_ref, const double *natoms, const float *F,
                 const float *F_ref, double w_E, double w_F, const double *g, double *gE, float *gF, void *stream) {
  return loss_grad(n_cells, n_comp, nullptr, E, E_ref, natoms, F, F_ref, w_E, w_F, g, gE, gF, stream);
}

int st_loss_kept_grad(int n_cells, int n_comp, const double *kept, double w_E, double w_F, const double *g, double *gE,
                      float *gF, void *stream) {
  return loss_grad(n_cells, n_comp, kept, nullptr, nullptr, nullptr, nullptr, nullptr, w_E, w_F, g, gE, gF, stream);
}

int st_adam(int npar, float *theta, const float *grad, float *m, float *v, float lr, float beta1, float beta2,
            float eps, int t, void *stream) {
  if (npar <= 0 || t < 1) return (int)cudaErrorInvalidValue;
  const float c1 = 1.f - powf(beta1, (float)t), c2 = 1.f - powf(beta2, (float)t);
  k_st_adam<<<blocks_of(npar, BLOCK), BLOCK, 0, (cudaStream_t)stream>>>(npar, theta, grad, m, v, lr, beta1, beta2,
                                                                       eps, c1, c2);
  return (int)cudaGetLastError();
}

}  // extern "C"
