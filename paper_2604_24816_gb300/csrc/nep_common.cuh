// nep_common.cuh -- device-side building blocks shared by the NEP kernels (sm_103a).
//
// Layout conventions (all per-atom arrays in cell-sorted order):
//   pos[i]   float4: position relative to the origin of the atom's cell at the last rebuild (x, y, z)
//            and the packed cell coordinates (w, as int bits: cx | cy << 10 | cz << 20).
//   nbr      int32 [cap][N] (neighbour-major, so a thread per atom reads coalesced rows); entry =
//            j | shift << 27, shift = (dx+1) + 3 (dy+1) + 9 (dz+1) the cell offset of j's image.
//            Row i = [pairs owned by i | the others], each part grouped by distance band; nown[i]
//            is the length of the owned part.
//   Ffix     int64 [3][N]: forces in fixed point (2^-32 eV/Angstrom units), accumulated with
//            integer atomics, so the sum does not depend on the order of the additions.
//   G        float or half [N][S::GS]: per-atom adjoint dU_i/ds_nlm (NA * NLM values, index n * NLM + lm)
//            followed by the radial adjoint in basis space dU_i/dQ_k = sum_n dU_i/dq_n cR_nk (KR <= 8
//            values, Q_k = sum_j f_k(r_ij) the radial basis sums) and padding
//            (teacher shape: 5 x 24 + 8 = 128 per row; student shape: 4 x 8 + 8 = 40).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace nep {

// SMs of the current device (152 if that cannot be read).
inline int sm_count() {
  int d = 0, sms = 0;
  if (cudaGetDevice(&d) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, d) != cudaSuccess ||
      sms <= 0) {
    cudaGetLastError();
    sms = 152;
  }
  return sms;
}

constexpr int J_BITS = 27;
constexpr uint32_t J_MASK = (1u << J_BITS) - 1u;
constexpr float FIX_SCALE = 4294967296.0f;        // 2^32 fixed-point units per eV/Angstrom
constexpr double FIX_INV = 1.0 / 4294967296.0;

// Status bits of the device status word.
enum : int {
  ST_OVERFLOW = 1,   // neighbour list capacity exceeded
  ST_NAN = 2,        // non-finite value seen
  ST_FB_OVERFLOW = 8, // more atoms flagged for the fallback model than its list holds
  ST_SLOT = 16        // a block found no free pair-record slot on its SM (not expected: see PairCache)
};

// The far band of a neighbour-list row starts at rc_R + FAR_EDGE * skin.  For fcc Cu at rc_R = 5 A and
// a 1 A skin this edge (5.4 A) lies between the 5.11 A and 5.72 A shells, so every atom's far band is
// the same shell and the walked rows stay aligned across the lanes of a warp; an edge inside a shell's
// thermal spread gives neighbouring atoms walked counts that differ by one or two, which misaligns the
// lanes' bands and costs more than the skipped entries save.
constexpr float FAR_EDGE = 0.4f;

// Device-side control block (one per handle).
struct Control {
  int status;           // OR of ST_* bits
  int moved;            // some atom moved more than skin/2 since the last rebuild
  int do_rebuild;       // decision of the current step
  int steps_since;      // MD steps since the last rebuild
  int rebuild_every;    // 0 = displacement-triggered only
  long long rebuilds;   // neighbour builds done
  long long steps;      // MD steps done
  int nb_next;          // next group of atoms for the neighbour scan (reset by each rebuild)
  float dmax2;          // largest squared displacement of an atom since the last rebuild (Angstrom^2)
  float far_dmax2;      // below this, no list entry of the far band can be inside the largest cutoff
  int skip_far;         // decision for the current evaluation: row walks may skip the far band
  int changed;          // an upload into the kept cell order changed some atom's float32 position
  int pending;          // the last MD step's closing half kick is still owed (applied by the next step's
                        // opening kick, or by the kick that ends md_verlet_step)
  int fb_count;         // atoms the last evaluation handed to the fallback model
};

// Arguments of the rebuild chain (cell sort + neighbour list).
struct RebuildArgs {
  int n, ncell;               // ncell: slices of cells (see slice_shift in nep_neighbor.cu)
  int ssh;
  double L[3], l[3];
  int nc[3];
  double *x, *y, *z, *vx, *vy, *vz, *xb, *yb, *zb, *vxb, *vyb, *vzb;
  int *id, *idb, *cell_of, *count, *cursor, *start, *tile_sums;   // count: zero between builds
  int2 *perm;
  float4 *pos, *pos_ref;
  int32_t *nbr, *nnum, *nang, *nown, *nband0, *nfar;
  int cap;
  float rl2, ra2, ba2, br2;   // (rc_R+skin)^2, (rc_A+skin)^2, rc_A^2, rc_R^2
  float fs2;                  // (rc_R + FAR_EDGE skin)^2: where the far band starts
  Control *ctrl;
};

// Compile-time model shape: NR radial functions, NA angular channels, KR/KA basis functions, 3-body
// harmonics l = 1..LMAX (NLM = LMAX (LMAX + 2) components), optional 4-body term (built from l = 2),
// NNEU hidden neurons.  GS = elements per adjoint row (NA * NLM, then an 8-element tail).
template <int NR_, int NA_, int KR_, int KA_, int LMAX_, bool FOURBODY_, int NNEU_>
struct Shape {
  static constexpr int NR = NR_, NA = NA_, KR = KR_, KA = KA_, LMAX = LMAX_, NNEU = NNEU_;
  static constexpr bool FOURBODY = FOURBODY_;
  static constexpr int NLM = LMAX * (LMAX + 2);
  static constexpr int NDES = NR + NA * LMAX + (FOURBODY ? NA : 0);
  static constexpr int GS = NA * NLM + 8;
  static_assert(NLM % 8 == 0, "rows are read in 16-byte vectors of up to 8 values: LMAX must be 2 or 4");
  static_assert(NR <= 8, "radial adjoint lives in the 8-element row tail");
  static_assert(!FOURBODY || LMAX >= 2, "the 4-body term is built from the l = 2 sums");
};

// The teacher NEP of the workload (n_max 4/4, basis 8/8, l_max 4, 4-body, 30 neurons) and the
// distilled student (n_max 3/3, basis 8/8, l_max 2, no 4-body, 16 neurons).
using CuShape = Shape<5, 5, 8, 8, 4, true, 30>;
using StudentShape = Shape<4, 4, 8, 8, 2, false, 16>;

// Model parameters, passed by value as a __grid_constant__ kernel argument so that every uniform
// access compiles to a constant-bank operand.
template <class S>
struct Model {
  float cR[S::NR][S::KR];
  float cA[S::NA][S::KA];
  float W0[S::NNEU][S::NDES];
  float b0[S::NNEU];
  float w1[S::NNEU];
  float qs[S::NDES];
  float b1;
  float rcR, rcA, rcR2, rcA2, inv_rcR, inv_rcA;
  float lj_on, lj_c12, lj_c6, lj_rc2, lj_e_rc, lj_de_rc, lj_rc;  // shifted-force LJ
  float lj_e0, lj_m12, lj_p6;   // rc E'(rc) - E(rc), -12 c12, 6 c6 (the factored forms of lj_pair)
  float rmax2;   // max(rcR, lj_rc)^2
  // g_n(r) = h(r) [E_n(y) + x O_n(y)], h = fc / 2, y = 2 x^2 - 1 (cheb_to_cubics of cA_n): coefficients of
  // y^0..y^3, channels 2p and 2p + 1 side by side; gL: the last channel's (E, O) when NA is odd.
  float2 gE[S::NA / 2][4], gO[S::NA / 2][4], gL[4];
};

// sum_k c_k (T_k(x) + 1), k = 0..7, as E(y) + x O(y) with y = T_2(x) = 2 x^2 - 1 and cubics E, O: the even
// orders are T_2j(x) = T_j(y), the odd ones x times 1, 2y - 1, 4y^2 - 2y - 1, 8y^3 - 4y^2 - 4y + 1.  The
// coefficients stay below 8, so a Horner evaluation on |y| <= 1 rounds like the three-term recurrence, with
// half its dependent steps and no basis values.  The fused kernels are bound by issue slots (67 % busy) and by
// the walk's dependent chains: with the cubics and the step-two recurrence of cheb_accumulate the teacher's
// takes 1.114 ms instead of 1.145 at 1,048,576 atoms, the student's 60.4 us instead of 61.8 at 56,000; forces
// against 64 bits are as far off as before (2.9e-6 relative on 862 atoms, both).
template <class T>
__host__ __device__ __forceinline__ void cheb_to_cubics(const T (&c)[8], T (&e)[4], T (&o)[4]) {
  const T sum = ((c[0] + c[1]) + (c[2] + c[3])) + ((c[4] + c[5]) + (c[6] + c[7]));
  e[0] = c[0] - c[4] + sum;
  e[1] = c[2] - 3 * c[6];
  e[2] = 2 * c[4];
  e[3] = 4 * c[6];
  o[0] = (c[1] - c[3]) - (c[5] - c[7]);
  o[1] = 2 * (c[3] - c[5]) - 4 * c[7];
  o[2] = 4 * (c[5] - c[7]);
  o[3] = 8 * c[7];
}

// The derived members of a model (host): the radial polynomials of its angular channels.
template <class S>
void fill_radial_polynomials(Model<S> &M) {
  static_assert(S::KA == 8, "eight basis functions");
  for (int a = 0; a < S::NA; ++a) {
    double c[8], e[4], o[4];
    for (int k = 0; k < 8; ++k) c[k] = M.cA[a][k];
    cheb_to_cubics(c, e, o);
    for (int i = 0; i < 4; ++i) {
      if (S::NA % 2 == 1 && a == S::NA - 1) {
        M.gL[i] = make_float2((float)e[i], (float)o[i]);
      } else {
        float *pe = a % 2 ? &M.gE[a / 2][i].y : &M.gE[a / 2][i].x;
        float *po = a % 2 ? &M.gO[a / 2][i].y : &M.gO[a / 2][i].x;
        *pe = (float)e[i];
        *po = (float)o[i];
      }
    }
  }
}

// Pair records of the fused kernels: the descriptor walk stores every active pair's displacement and
// neighbour index, and the force pass reads them back instead of walking the neighbour list again.
// Each resident block owns one region [pmax][BLOCK] float4 of `rec`, chosen by the SM it runs on and a
// free slot among that SM's `slots` (one bit each in slot_mask[sm]).  The teacher's fused kernels use
// PC_SLOTS: at most that many of their blocks fit on an SM (each holds 512 / PC_SLOTS of the SM's
// tensor-memory columns); the student's register-resident fused kernel uses PC_SLOTS_REG, checked on
// the host against its occupancy.  So a slot is always free for a starting block.  Regions are reused
// block after block, so their lines stay in L2.
constexpr int PC_SLOTS = 4;
constexpr int PC_SLOTS_REG = 8;
struct PairCache {
  float4 *rec;           // [nsm * slots][pmax][BLOCK]
  unsigned *slot_mask;   // [nsm], zero-initialised; bit b: slot b of that SM is held
  int nsm;               // bound on the SM index (%nsmid)
  int pmax;              // records per atom: >= the neighbour-list capacity
  int slots;             // regions per SM index
};

__device__ __forceinline__ unsigned sm_index() {
  unsigned r;
  asm volatile("mov.u32 %0, %%smid;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned sm_index_bound() {
  unsigned r;
  asm volatile("mov.u32 %0, %%nsmid;" : "=r"(r));
  return r;
}

// A free pair-record region of this SM for the calling block (one thread calls it): sm * slots + b, or
// -1 after 64 rounds over the SM's slots (the caller reports that; it cannot happen while no more than
// `slots` blocks of the kernel are resident on an SM).
__device__ __forceinline__ int acquire_record_slot(const PairCache &pc) {
  const unsigned sm = sm_index();
  int slot = -1;
  if ((int)sm < pc.nsm) {
    for (int it = 0; it < 64 && slot < 0; ++it)
      for (int b = 0; b < pc.slots && slot < 0; ++b)
        if ((atomicOr(pc.slot_mask + sm, 1u << b) & (1u << b)) == 0u) slot = (int)sm * pc.slots + b;
  }
  return slot;
}

// Cell geometry of the current neighbour list.
struct Geom {
  float lx, ly, lz;      // cell edge lengths (float)
  int ncx, ncy, ncz;
};

__device__ __forceinline__ int cell_x(float w) { return __float_as_int(w) & 1023; }
__device__ __forceinline__ int cell_y(float w) { return (__float_as_int(w) >> 10) & 1023; }
__device__ __forceinline__ int cell_z(float w) { return (__float_as_int(w) >> 20) & 1023; }

// Offsets of the 27 neighbouring cell images: shift s = (dx+1) + 3(dy+1) + 9(dz+1).
__device__ __forceinline__ void fill_shift_table(float4 *tab, const Geom &g) {
  for (int s = threadIdx.x; s < 27; s += blockDim.x) {
    int dx = s % 3 - 1, dy = (s / 3) % 3 - 1, dz = s / 9 - 1;
    tab[s] = make_float4(dx * g.lx, dy * g.ly, dz * g.lz, 0.f);
  }
}

// Packed float2 arithmetic: two FP32 operations per instruction on the sm_100 family (FFMA2, FADD2,
// FMUL2), each rounded as its scalar counterpart.  The hot loops pair independent operations so that
// they issue half as many FP32 instructions.
// (The host forms serve the host-side checks.)
__host__ __device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
#ifdef __CUDA_ARCH__
  return __ffma2_rn(a, b, c);
#else
  return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y));
#endif
}
__host__ __device__ __forceinline__ float2 add2(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
  return __fadd2_rn(a, b);
#else
  return make_float2(a.x + b.x, a.y + b.y);
#endif
}
__host__ __device__ __forceinline__ float2 mul2(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
  return __fmul2_rn(a, b);
#else
  return make_float2(a.x * b.x, a.y * b.y);
#endif
}
__host__ __device__ __forceinline__ float2 bc2(float a) { return make_float2(a, a); }
__host__ __device__ __forceinline__ float2 pr(float a, float b) { return make_float2(a, b); }
__host__ __device__ __forceinline__ float hsum(float2 a) { return a.x + a.y; }

// sum_k c[k] f[k] (K even) as K/2 paired multiply-adds (even and odd k accumulated apart) and one add.
template <int K>
__device__ __forceinline__ float dot_pairs(const float (&c)[K], const float (&f)[K]) {
  static_assert(K % 2 == 0, "even length");
  float2 t = mul2(pr(c[0], c[1]), pr(f[0], f[1]));
#pragma unroll
  for (int k = 2; k < K; k += 2) t = fma2(pr(c[k], c[k + 1]), pr(f[k], f[k + 1]), t);
  return hsum(t);
}
// Two dot products with the same coefficients: sum_k c[k] f[k] and sum_k c[k] d[k].
template <int K>
__device__ __forceinline__ void dot_pairs2(const float (&c)[K], const float (&f)[K], const float (&d)[K], float &tf,
                                           float &td) {
  static_assert(K % 2 == 0, "even length");
  const float2 c0 = pr(c[0], c[1]);
  float2 a = mul2(c0, pr(f[0], f[1])), b = mul2(c0, pr(d[0], d[1]));
#pragma unroll
  for (int k = 2; k < K; k += 2) {
    const float2 ck = pr(c[k], c[k + 1]);
    a = fma2(ck, pr(f[k], f[k + 1]), a);
    b = fma2(ck, pr(d[k], d[k + 1]), b);
  }
  tf = hsum(a);
  td = hsum(b);
}

// Chebyshev basis f_k(r) = (T_k(x) + 1)/2 * fc(r), x = 2 (r/rc - 1)^2 - 1, fc = (1 + cos(pi r/rc))/2,
// evaluated as f_k = h T_k + h with h = fc / 2 (T_k by the three-term recurrence, the f_k in pairs).
// The cutoff uses the hardware sine/cosine (absolute error below 2^-21.4 for arguments in [-pi, pi];
// here pi r / rc lies in [0, pi]), a few instructions instead of the range-reduced library call.
template <int K>
__device__ __forceinline__ void cheb_basis(float r, float inv_rc, float (&f)[K]) {
  static_assert(K % 2 == 0 && K >= 2, "even basis size");
  float s, c;
  const float t = r * inv_rc;
  __sincosf(3.14159265358979f * t, &s, &c);
  const float h = fmaf(0.25f, c, 0.25f);         // fc / 2 (= (c + 1) / 4, one rounding)
  const float u = t - 1.f;
  const float x = fmaf(2.f * u, u, -1.f);
  const float x2 = x + x;
  float T[K];
  T[0] = 1.f; T[1] = x;
#pragma unroll
  for (int k = 2; k < K; ++k) T[k] = fmaf(x2, T[k - 1], -T[k - 2]);
  const float2 h2 = bc2(h);
#pragma unroll
  for (int k = 0; k < K; k += 2) {
    const float2 v = fma2(h2, pr(T[k], T[k + 1]), h2);
    f[k] = v.x; f[k + 1] = v.y;
  }
}

// Basis and radial derivative: f_k' = (T_k + 1) h' + T_k'(x) x'(r) h, with h = fc / 2, h' = fc' / 2,
// T_k' by the differentiated recurrence T_k' = 2 T_{k-1} + 2 x T_{k-1}' - T_{k-2}'.
template <int K>
__device__ __forceinline__ void cheb_basis_d(float r, float inv_rc, float (&f)[K], float (&df)[K]) {
  static_assert(K % 2 == 0 && K >= 2, "even basis size");
  float s, c;
  const float t = r * inv_rc;
  __sincosf(3.14159265358979f * t, &s, &c);
  const float h = fmaf(0.25f, c, 0.25f);                           // fc / 2
  const float dh = (-0.25f * 3.14159265358979f * inv_rc) * s;      // fc' / 2
  const float u = t - 1.f;
  const float x = fmaf(2.f * u, u, -1.f);
  const float x2 = x + x;
  const float dxh = (4.f * inv_rc) * u * h;                        // x'(r) h
  float T[K], D[K];
  T[0] = 1.f; T[1] = x;
  D[0] = 0.f; D[1] = 1.f;
#pragma unroll
  for (int k = 2; k < K; ++k) {
    T[k] = fmaf(x2, T[k - 1], -T[k - 2]);
    D[k] = fmaf(x2, D[k - 1], fmaf(2.f, T[k - 1], -D[k - 2]));
  }
  const float2 h2 = bc2(h), dh2 = bc2(dh), dxh2 = bc2(dxh);
#pragma unroll
  for (int k = 0; k < K; k += 2) {
    const float2 tk = pr(T[k], T[k + 1]);
    const float2 v = fma2(h2, tk, h2);
    const float2 d = fma2(pr(D[k], D[k + 1]), dxh2, fma2(tk, dh2, dh2));
    f[k] = v.x; f[k + 1] = v.y;
    df[k] = d.x; df[k + 1] = d.y;
  }
}

// The same cutoff and argument for the forms that never build the f_k: h = fc / 2, x and y = 2 x^2 - 1
// (cheb_args), with dh = fc' / 2 and dxh = x'(r) h (cheb_args_d).
__device__ __forceinline__ void cheb_args(float r, float inv_rc, float &h, float &x, float &y) {
  const float t = r * inv_rc;
  h = fmaf(0.25f, __cosf(3.14159265358979f * t), 0.25f);
  const float u = t - 1.f;
  x = fmaf(2.f * u, u, -1.f);
  y = fmaf(2.f * x, x, -1.f);
}
__device__ __forceinline__ void cheb_args_d(float r, float inv_rc, float &h, float &dh, float &dxh, float &x, float &y) {
  float s, c;
  const float t = r * inv_rc;
  __sincosf(3.14159265358979f * t, &s, &c);
  h = fmaf(0.25f, c, 0.25f);
  dh = (-0.25f * 3.14159265358979f * inv_rc) * s;
  const float u = t - 1.f;
  x = fmaf(2.f * u, u, -1.f);
  y = fmaf(2.f * x, x, -1.f);
  dxh = (4.f * inv_rc) * u * h;
}

// Adds h T_k(x), k = 0..7, of one pair to the sums Q (pairs (T_0, T_1), (T_2, T_3), ...), the last two pairs
// with the opposite sign.  Step-two recurrence T_(k+2) = 2 y T_k - T_(k-2) on the pairs: three dependent steps
// for the eight orders (the three-term recurrence takes six, each on one order), and the alternating sign
// needs no negated operand.
__device__ __forceinline__ void cheb_accumulate(float r, float inv_rc, float2 (&Q)[4]) {
  float h, x, y;
  cheb_args(r, inv_rc, h, x, y);
  const float y2 = y + y;
  const float2 h2 = bc2(h);
  const float2 t01 = pr(1.f, x), t23 = pr(y, fmaf(y2, x, -x));
  const float2 n45 = fma2(bc2(-y2), t23, t01);      // -(T_4, T_5)
  const float2 n67 = fma2(bc2(y2), n45, t23);       // -(T_6, T_7)
  Q[0] = fma2(h2, t01, Q[0]);
  Q[1] = fma2(h2, t23, Q[1]);
  Q[2] = fma2(h2, n45, Q[2]);
  Q[3] = fma2(h2, n67, Q[3]);
}
// The radial basis sums from the accumulated Q: sum f_k = sum h T_k + sum h (T_0 = 1: Q[0].x is sum h).
__device__ __forceinline__ void cheb_sums(const float2 (&Q)[4], float (&QR)[8]) {
  const float sh = Q[0].x;
  QR[0] = Q[0].x + sh; QR[1] = Q[0].y + sh;
  QR[2] = Q[1].x + sh; QR[3] = Q[1].y + sh;
  QR[4] = sh - Q[2].x; QR[5] = sh - Q[2].y;
  QR[6] = sh - Q[3].x; QR[7] = sh - Q[3].y;
}

// The angular channels' radial functions g_n(r) = h [E_n(y) + x O_n(y)] (Model::gE, gO, gL), two channels per
// instruction; on: g = 0 when false.
template <class S>
__device__ __forceinline__ void radial_channels(const Model<S> &P, float r, bool on, float (&g)[S::NA]) {
  float h, x, y;
  cheb_args(r, P.inv_rcA, h, x, y);
  h = on ? h : 0.f;
  const float2 yy = bc2(y), xx = bc2(x), hh = bc2(h);
#pragma unroll
  for (int p = 0; p < S::NA / 2; ++p) {
    float2 e = P.gE[p][3], o = P.gO[p][3];
#pragma unroll
    for (int i = 2; i >= 0; --i) { e = fma2(e, yy, P.gE[p][i]); o = fma2(o, yy, P.gO[p][i]); }
    const float2 v = mul2(fma2(xx, o, e), hh);
    g[2 * p] = v.x; g[2 * p + 1] = v.y;
  }
  if constexpr (S::NA % 2 == 1) {
    float2 v = P.gL[3];
#pragma unroll
    for (int i = 2; i >= 0; --i) v = fma2(v, yy, P.gL[i]);
    g[S::NA - 1] = fmaf(x, v.y, v.x) * h;
  }
}
// g_n and g_n': with p = E + x O, dp/dx = 4 x (E' + x O') + O, g' = p dh + dp/dx dxh.
// (M: a Model, or any holder of inv_rcA, gE, gO, gL.)
template <class S, class M>
__device__ __forceinline__ void radial_channels_d(const M &P, float r, float (&g)[S::NA], float (&dg)[S::NA]) {
  float h, dh, dxh, x, y;
  cheb_args_d(r, P.inv_rcA, h, dh, dxh, x, y);
  const float x4 = 4.f * x;
  const float2 yy = bc2(y), xx = bc2(x), xx4 = bc2(x4), hh = bc2(h), dhh = bc2(dh), dxx = bc2(dxh);
#pragma unroll
  for (int p = 0; p < S::NA / 2; ++p) {
    float2 de = P.gE[p][3], dd = P.gO[p][3];
    float2 e = fma2(de, yy, P.gE[p][2]), o = fma2(dd, yy, P.gO[p][2]);
#pragma unroll
    for (int i = 1; i >= 0; --i) {
      de = fma2(de, yy, e); dd = fma2(dd, yy, o);
      e = fma2(e, yy, P.gE[p][i]); o = fma2(o, yy, P.gO[p][i]);
    }
    const float2 v = fma2(xx, o, e);
    const float2 dv = fma2(xx4, fma2(xx, dd, de), o);
    const float2 a = mul2(v, hh), b = fma2(v, dhh, mul2(dv, dxx));
    g[2 * p] = a.x; g[2 * p + 1] = a.y;
    dg[2 * p] = b.x; dg[2 * p + 1] = b.y;
  }
  if constexpr (S::NA % 2 == 1) {
    float2 d = P.gL[3];
    float2 v = fma2(d, yy, P.gL[2]);
#pragma unroll
    for (int i = 1; i >= 0; --i) { d = fma2(d, yy, v); v = fma2(v, yy, P.gL[i]); }
    const float q = fmaf(x, v.y, v.x), dq = fmaf(x4, fmaf(x, d.y, d.x), v.y);
    g[S::NA - 1] = q * h;
    dg[S::NA - 1] = fmaf(q, dh, dq * dxh);
  }
}

// sum_k t_k f_k'(r) for a radial adjoint t held as cubics (cheb_to_cubics; c0 = (e0, o0, e1, o1), c1 = (e2, o2,
// e3, o3)): p dh + dp/dx dxh as in radial_channels_d; the second form evaluates two pairs at once.
__device__ __forceinline__ float cubics_deriv(float4 c0, float4 c1, float r, float inv_rc) {
  float h, dh, dxh, x, y;
  cheb_args_d(r, inv_rc, h, dh, dxh, x, y);
  const float2 yy = bc2(y);
  float2 d = pr(c1.z, c1.w);
  float2 v = fma2(d, yy, pr(c1.x, c1.y));
  d = fma2(d, yy, v);
  v = fma2(v, yy, pr(c0.z, c0.w));
  d = fma2(d, yy, v);
  v = fma2(v, yy, pr(c0.x, c0.y));
  return fmaf(fmaf(x, v.y, v.x), dh, fmaf(4.f * x, fmaf(x, d.y, d.x), v.y) * dxh);
}
__device__ __forceinline__ float2 cubics_deriv_x2(float4 c0, float4 c1, float2 r, float inv_rc) {
  float2 s, cs;
  const float2 t = mul2(r, bc2(inv_rc));
  __sincosf(3.14159265358979f * t.x, &s.x, &cs.x);
  __sincosf(3.14159265358979f * t.y, &s.y, &cs.y);
  const float2 h = fma2(bc2(0.25f), cs, bc2(0.25f));
  const float2 dh = mul2(bc2(-0.25f * 3.14159265358979f * inv_rc), s);
  const float2 u = add2(t, bc2(-1.f));
  const float2 x = fma2(add2(u, u), u, bc2(-1.f));
  const float2 y = fma2(add2(x, x), x, bc2(-1.f));
  const float2 dxh = mul2(mul2(bc2(4.f * inv_rc), u), h);
  float2 de = bc2(c1.z), dd = bc2(c1.w);
  float2 e = fma2(de, y, bc2(c1.x)), o = fma2(dd, y, bc2(c1.y));
  de = fma2(de, y, e); dd = fma2(dd, y, o);
  e = fma2(e, y, bc2(c0.z)); o = fma2(o, y, bc2(c0.w));
  de = fma2(de, y, e); dd = fma2(dd, y, o);
  e = fma2(e, y, bc2(c0.x)); o = fma2(o, y, bc2(c0.y));
  const float2 v = fma2(x, o, e);
  const float2 dv = fma2(mul2(bc2(4.f), x), fma2(x, dd, de), o);
  return fma2(v, dh, mul2(dv, dxh));
}

// Normalised real harmonics Yh_lm(u) = sqrt(4 pi / (2l+1)) Y_lm(u), l = 1..4 (24 values, m = -l..l),
// so that sum_m Yh_lm(u) Yh_lm(v) = P_l(u . v).  Written as solid-harmonic polynomials of a unit vector.
// NLM = 8 computes l = 1, 2 only.
template <int NLM>
__host__ __device__ __forceinline__ void harmonics(float x, float y, float z, float (&Y)[NLM]) {
  static_assert(NLM == 8 || NLM == 24, "l_max 2 or 4");
  const float x2 = x * x, y2 = y * y, z2 = z * z;
  const float s3 = 1.7320508075688772f, s5 = 2.2360679774997896f, s6 = 2.449489742783178f;
  const float s10 = 3.1622776601683795f, s15 = 3.872983346207417f, s35 = 5.916079783099616f;
  const float s70 = 8.366600265340756f;
  // l = 1
  Y[0] = y; Y[1] = z; Y[2] = x;
  // l = 2
  Y[3] = s3 * x * y;
  Y[4] = s3 * y * z;
  Y[5] = z2 - 0.5f * (x2 + y2);
  Y[6] = s3 * x * z;
  Y[7] = 0.5f * s3 * (x2 - y2);
  if constexpr (NLM > 8) {
  // l = 3
  const float a3 = 4.f * z2 - x2 - y2;
  Y[8] = 0.25f * s10 * y * (3.f * x2 - y2);
  Y[9] = s15 * x * y * z;
  Y[10] = 0.25f * s6 * y * a3;
  Y[11] = z * (z2 - 1.5f * (x2 + y2));
  Y[12] = 0.25f * s6 * x * a3;
  Y[13] = 0.5f * s15 * z * (x2 - y2);
  Y[14] = 0.25f * s10 * x * (x2 - 3.f * y2);
  // l = 4
  const float rr = x2 + y2 + z2;
  const float b4 = 7.f * z2 - rr, c4 = 7.f * z2 - 3.f * rr;
  Y[15] = 0.5f * s35 * x * y * (x2 - y2);
  Y[16] = 0.25f * s70 * y * z * (3.f * x2 - y2);
  Y[17] = 0.5f * s5 * x * y * b4;
  Y[18] = 0.25f * s10 * y * z * c4;
  Y[19] = 0.125f * (35.f * z2 * z2 - 30.f * z2 * rr + 3.f * rr * rr);
  Y[20] = 0.25f * s10 * x * z * c4;
  Y[21] = 0.25f * s5 * (x2 - y2) * b4;
  Y[22] = 0.25f * s70 * x * z * (x2 - 3.f * y2);
  Y[23] = 0.125f * s35 * (x2 * x2 - 6.f * x2 * y2 + y2 * y2);
  }
}

// Gradient (ax, ay, az) of the solid-harmonic polynomial of component lm at (x, y, z).  lm is a
// compile-time constant after unrolling; harmonic_grad_mask(lm) has bit d set when component d can be
// non-zero, so callers skip the multiply-adds of the identically zero ones.
__host__ __device__ __forceinline__ void harmonic_grad(int lm, float x, float y, float z, float (&a)[3]) {
  const float x2 = x * x, y2 = y * y, z2 = z * z;
  const float s3 = 1.7320508075688772f, s5 = 2.2360679774997896f, s6 = 2.449489742783178f;
  const float s10 = 3.1622776601683795f, s15 = 3.872983346207417f, s35 = 5.916079783099616f;
  const float s70 = 8.366600265340756f;
  float ax = 0.f, ay = 0.f, az = 0.f;
  switch (lm) {
    case 0: ay = 1.f; break;
    case 1: az = 1.f; break;
    case 2: ax = 1.f; break;
    case 3: ax = s3 * y; ay = s3 * x; break;
    case 4: ay = s3 * z; az = s3 * y; break;
    case 5: ax = -x; ay = -y; az = 2.f * z; break;
    case 6: ax = s3 * z; az = s3 * x; break;
    case 7: ax = s3 * x; ay = -s3 * y; break;
    case 8: ax = 1.5f * s10 * x * y; ay = 0.75f * s10 * (x2 - y2); break;
    case 9: ax = s15 * y * z; ay = s15 * x * z; az = s15 * x * y; break;
    case 10: ax = -0.5f * s6 * x * y; ay = -0.25f * s6 * (x2 + 3.f * y2 - 4.f * z2); az = 2.f * s6 * y * z; break;
    case 11: ax = -3.f * x * z; ay = -3.f * y * z; az = -1.5f * (x2 + y2 - 2.f * z2); break;
    case 12: ax = -0.25f * s6 * (3.f * x2 + y2 - 4.f * z2); ay = -0.5f * s6 * x * y; az = 2.f * s6 * x * z; break;
    case 13: ax = s15 * x * z; ay = -s15 * y * z; az = 0.5f * s15 * (x2 - y2); break;
    case 14: ax = 0.75f * s10 * (x2 - y2); ay = -1.5f * s10 * x * y; break;
    case 15: ax = 0.5f * s35 * y * (3.f * x2 - y2); ay = 0.5f * s35 * x * (x2 - 3.f * y2); break;
    case 16: ax = 1.5f * s70 * x * y * z; ay = 0.75f * s70 * z * (x2 - y2); az = 0.25f * s70 * y * (3.f * x2 - y2); break;
    case 17: ax = -0.5f * s5 * y * (3.f * x2 + y2 - 6.f * z2); ay = -0.5f * s5 * x * (x2 + 3.f * y2 - 6.f * z2);
             az = 6.f * s5 * x * y * z; break;
    case 18: ax = -1.5f * s10 * x * y * z; ay = -0.25f * s10 * z * (3.f * x2 + 9.f * y2 - 4.f * z2);
             az = -0.75f * s10 * y * (x2 + y2 - 4.f * z2); break;
    case 19: ax = 1.5f * x * (x2 + y2 - 4.f * z2); ay = 1.5f * y * (x2 + y2 - 4.f * z2);
             az = -2.f * z * (3.f * x2 + 3.f * y2 - 2.f * z2); break;
    case 20: ax = -0.25f * s10 * z * (9.f * x2 + 3.f * y2 - 4.f * z2); ay = -1.5f * s10 * x * y * z;
             az = -0.75f * s10 * x * (x2 + y2 - 4.f * z2); break;
    case 21: ax = -s5 * x * (x2 - 3.f * z2); ay = s5 * y * (y2 - 3.f * z2); az = 3.f * s5 * z * (x2 - y2); break;
    case 22: ax = 0.75f * s70 * z * (x2 - y2); ay = -1.5f * s70 * x * y * z; az = 0.25f * s70 * x * (x2 - 3.f * y2); break;
    case 23: ax = 0.5f * s35 * x * (x2 - 3.f * y2); ay = -0.5f * s35 * y * (3.f * x2 - y2); break;
    default: break;
  }
  a[0] = ax; a[1] = ay; a[2] = az;
}
__host__ __device__ constexpr int harmonic_grad_mask(int lm) {
  return lm == 0 ? 2 : lm == 1 ? 4 : lm == 2 ? 1 : lm == 3 ? 3 : lm == 4 ? 6 : lm == 6 ? 5 :
         (lm == 7 || lm == 8 || lm == 14 || lm == 15 || lm == 23) ? 3 : 7;
}

// Gradient of the solid-harmonic polynomial of component lm, evaluated at (x, y, z), accumulated
// with weight b into (gx, gy, gz).
__device__ __forceinline__ void harmonic_grad_acc(int lm, float x, float y, float z, float b, float &gx,
                                                  float &gy, float &gz) {
  float a[3];
  harmonic_grad(lm, x, y, z, a);
  const int m = harmonic_grad_mask(lm);
  if (m & 1) gx = fmaf(b, a[0], gx);
  if (m & 2) gy = fmaf(b, a[1], gy);
  if (m & 4) gz = fmaf(b, a[2], gz);
}

// The same for the two components lm0, lm0 + 1 with weights b = (b_lm0, b_lm0+1), accumulated into the
// component pairs g[d] (even and odd lm apart): paired multiply-adds where both are non-zero.
__device__ __forceinline__ void harmonic_grad_acc2(int lm0, float x, float y, float z, float2 b, float2 (&g)[3]) {
  float a0[3], a1[3];
  harmonic_grad(lm0, x, y, z, a0);
  harmonic_grad(lm0 + 1, x, y, z, a1);
  const int m0 = harmonic_grad_mask(lm0), m1 = harmonic_grad_mask(lm0 + 1);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const bool n0 = (m0 >> d) & 1, n1 = (m1 >> d) & 1;
    if (n0 && n1) g[d] = fma2(b, pr(a0[d], a1[d]), g[d]);
    else if (n0) g[d].x = fmaf(b.x, a0[d], g[d].x);
    else if (n1) g[d].y = fmaf(b.y, a1[d], g[d].y);
  }
}

__host__ __device__ constexpr int lm_l(int lm) { return lm < 3 ? 1 : (lm < 8 ? 2 : (lm < 15 ? 3 : 4)); }

// Shifted-force LJ pair energy E(r) and dE/dr, from r^2, r and ir = 1/r (reciprocal square root).
// No division: 1/r^2 = ir^2 refined by one Newton step (error about 1 ulp, which the twelfth power
// would otherwise amplify from the reciprocal square root's 2 ulp), 1/r = ir.
template <class S>
__device__ __forceinline__ void lj_pair(const Model<S> &P, float r2, float r, float ir, float &e, float &de) {
  float ir2 = ir * ir;
  ir2 = fmaf(ir2, fmaf(-r2, ir2, 1.f), ir2);
  const float ir6 = ir2 * ir2 * ir2;
  // E = c12 r^-12 - c6 r^-6 - E(rc) - (r - rc) E'(rc) = r^-6 (c12 r^-6 - c6) + (rc E'(rc) - E(rc)) - r E'(rc)
  e = fmaf(ir6, fmaf(P.lj_c12, ir6, -P.lj_c6), fmaf(-P.lj_de_rc, r, P.lj_e0));
  // dE/dr = r^-6 (-12 c12 r^-6 + 6 c6) / r - E'(rc)
  de = fmaf(ir6 * fmaf(P.lj_m12, ir6, P.lj_p6), ir, -P.lj_de_rc);
}

// lj_pair for two pairs at once.
template <class S>
__device__ __forceinline__ void lj_pair_x2(const Model<S> &P, float2 r2, float2 r, float2 ir, float2 &e, float2 &de) {
  float2 ir2 = mul2(ir, ir);
  ir2 = fma2(ir2, fma2(make_float2(-r2.x, -r2.y), ir2, bc2(1.f)), ir2);
  const float2 ir6 = mul2(mul2(ir2, ir2), ir2);
  e = fma2(ir6, fma2(bc2(P.lj_c12), ir6, bc2(-P.lj_c6)), fma2(bc2(-P.lj_de_rc), r, bc2(P.lj_e0)));
  de = fma2(mul2(ir6, fma2(bc2(P.lj_m12), ir6, bc2(P.lj_p6))), ir, bc2(-P.lj_de_rc));
}

// Exact conversion of a float to 64-bit fixed point with 32 fractional bits, without a 64-bit
// conversion instruction (those run on the narrow FP64 pipe).
// |v| < 2^12 (every force, energy and virial term of a physical configuration): v * 2^32 is split as
// h * 2^22 + l with h = rint(v * 2^10) and |l| <= 2^21.  Both parts are exact in float32 (l is the
// rounding remainder of v * 2^10, scaled by a power of two), and each is turned into an integer by
// adding 1.5 * 2^23, which places the rounded integer in the low mantissa bits: full-rate FP32 and
// integer instructions only, rounding to nearest (ties to even).
// Larger magnitudes, infinities and NaN take an integer bit-manipulation path (round half away from
// zero; valid for |v| < 2^30).  Either way the result is a fixed function of v, so fixed-point sums
// do not depend on the order of their terms.
__device__ __forceinline__ long long to_fix32(float v) {
  constexpr float SHIFT = 12582912.0f;          // 1.5 * 2^23
  if (fabsf(v) < 4096.f) {
    const float hm = fmaf(v, 1024.f, SHIFT);     // SHIFT + rint(v * 2^10)
    const float h = hm - SHIFT;
    const float l = fmaf(v, 4294967296.f, -h * 4194304.f);
    const int hi = __float_as_int(hm) - 0x4B400000;
    const int lo = __float_as_int(l + SHIFT) - 0x4B400000;
    return ((long long)hi << 22) + lo;
  }
  const uint32_t b = __float_as_uint(v);
  const int ex = (int)((b >> 23) & 0xffu);
  const long long man = (long long)((b & 0x7fffffu) | 0x800000u);
  const int sh = ex - 118;                      // v * 2^32 = man * 2^(ex - 127 - 23 + 32)
  long long r;
  if (sh >= 0) r = man << min(sh, 39);
  else r = (man + (1ll << (-sh - 1))) >> (-sh);
  return (b >> 31) ? -r : r;
}

// to_fix32 of three values with one range test and the float parts of x and y in float2 pairs (the
// same results as three to_fix32 calls).
__device__ __forceinline__ void to_fix32x3(float x, float y, float z, long long &a, long long &b, long long &cz) {
  constexpr float SHIFT = 12582912.0f;
  const float m = fmaxf(fmaxf(fabsf(x), fabsf(y)), fabsf(z));
  if (m < 4096.f) {
    const float2 xy = make_float2(x, y);
    const float2 hm = __ffma2_rn(xy, make_float2(1024.f, 1024.f), make_float2(SHIFT, SHIFT));
    const float hmz = fmaf(z, 1024.f, SHIFT);
    const float2 h = __fadd2_rn(hm, make_float2(-SHIFT, -SHIFT));
    const float hz = hmz - SHIFT;
    const float2 l = __ffma2_rn(xy, make_float2(4294967296.f, 4294967296.f), __fmul2_rn(h, make_float2(-4194304.f, -4194304.f)));
    const float lz = fmaf(z, 4294967296.f, hz * -4194304.f);
    const float2 lm = __fadd2_rn(l, make_float2(SHIFT, SHIFT));
    const float lmz = lz + SHIFT;
    a = ((long long)(__float_as_int(hm.x) - 0x4B400000) << 22) + (__float_as_int(lm.x) - 0x4B400000);
    b = ((long long)(__float_as_int(hm.y) - 0x4B400000) << 22) + (__float_as_int(lm.y) - 0x4B400000);
    cz = ((long long)(__float_as_int(hmz) - 0x4B400000) << 22) + (__float_as_int(lmz) - 0x4B400000);
  } else {
    a = to_fix32(x); b = to_fix32(y); cz = to_fix32(z);
  }
}

// 64-bit integer add to global memory whose result nobody reads (the fixed-point force scatter, the running
// sums): a reduction, which returns nothing, so no register waits for the memory system (atomicAdd on a
// generic pointer becomes a value-returning atomic).  Integer addition is associative, so the sums do
// not depend on the order in which the additions arrive.
__device__ __forceinline__ void red_add(unsigned long long *p, long long v) {
  asm volatile("red.global.add.u64 [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "l"(v));
}

// Energy, virial and counters of an evaluation.  Every block adds its integer (fixed-point) sums to the running
// totals acc, and the last block of the evaluation's last kernel turns them into sums and counters and clears
// acc: no array of per-block rows and no reduction kernel (which took 2.4 us per step up to 16,384 atoms, 6.4 at
// 1,048,576 and 36 at 8,388,608; 18 reductions per block disappear beside the block's own work).  Integer sums:
// the result does not depend on the order of the blocks.
// Index v: 0 E, 1..9 W, 10 kinetic energy, 11..14 {radial pairs, angular pairs, list entries, active pairs} of the
// descriptor walk, 15..18 {list entries, active, radial, angular pairs} of the force pass.
// counters[v - 11] += total for v >= 11, counters[8] += 1 per evaluation.
constexpr int N_SUMS = 19;
struct EvalSums {
  long long *acc;        // [N_SUMS] running totals (zero between evaluations); nullptr: nothing is summed
  unsigned *done;        // blocks of the publishing kernel that have added theirs (zero between kernels)
  double *sums;
  long long *counters;
  int publish;           // this kernel is the evaluation's last
};
// The totals of index v, published by one thread.
__device__ __forceinline__ void publish_sum(const EvalSums &E, int v) {
  const long long tot = (long long)atomicExch(reinterpret_cast<unsigned long long *>(E.acc + v), 0ull);
  E.sums[v] = v <= 10 ? (double)tot * FIX_INV : (double)tot;       // energies/virial are fixed point
  if (v >= 11) E.counters[v - 11] += tot;
  if (v == 0) E.counters[8] += 1;
}
// Whether the calling warp's block is the last of the grid to get here (after its additions); resets the count.
__device__ __forceinline__ bool last_block(unsigned *done) {
  __threadfence();
  __syncwarp();
  unsigned k = 0;
  if ((threadIdx.x & 31) == 0) k = atomicAdd(done, 1u);
  const bool last = __shfl_sync(0xffffffffu, k, 0) == gridDim.x - 1;
  if (last) {
    __threadfence();
    if ((threadIdx.x & 31) == 0) *done = 0u;
  }
  return last;
}

// The warp's sums of NV int64 values, written by lane 0 to dst[0..NV-1].
template <int NV>
__device__ __forceinline__ void warp_sum_stage(long long (&v)[NV], long long *dst) {
#pragma unroll
  for (int k = 0; k < NV; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
  }
  if ((threadIdx.x & 31) == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) dst[k] = v[k];
  }
}
// After a block barrier that follows warp_sum_stage: the block's staged sums of NW warps, d = {E, radial pairs,
// angular pairs, list entries, active pairs} and f = {W[9], list entries, active, radial, angular pairs} (either may
// be nullptr), added to the running totals.
template <int NW>
__device__ __forceinline__ void eval_add(const EvalSums &E, const long long (*d)[5], const long long (*f)[13]) {
  const int t = threadIdx.x;
  if (t >= 32 || E.acc == nullptr) return;
  long long v = 0;
  int idx = 0;
  if (t < 5) {
    idx = t == 0 ? 0 : 10 + t;
    if (d != nullptr)
      for (int w = 0; w < NW; ++w) v += d[w][t];
  } else if (t < 18) {
    const int k = t - 5;
    idx = k < 9 ? 1 + k : 6 + k;
    if (f != nullptr)
      for (int w = 0; w < NW; ++w) v += f[w][k];
  }
  if (v != 0) red_add(reinterpret_cast<unsigned long long *>(E.acc + idx), v);
  if (E.publish && last_block(E.done) && t < 18) publish_sum(E, idx);
}
// Stages and adds one of the two groups at the end of a kernel (block barrier inside).
template <int NW>
__device__ __forceinline__ void eval_add_d(const EvalSums &E, long long (&v)[5]) {
  __shared__ long long w[NW][5];
  warp_sum_stage<5>(v, w[threadIdx.x >> 5]);
  __syncthreads();
  eval_add<NW>(E, w, nullptr);
}
template <int NW>
__device__ __forceinline__ void eval_add_f(const EvalSums &E, long long (&v)[13]) {
  __shared__ long long w[NW][13];
  warp_sum_stage<13>(v, w[threadIdx.x >> 5]);
  __syncthreads();
  eval_add<NW>(E, nullptr, w);
}

// ---------------------------------------------------------------------------------------------------
// Asynchronous per-thread neighbour pipeline (cp.async into shared memory).  The walk over an atom's
// list is a chain of dependent loads (list entry -> neighbour position); the pipeline keeps list
// entries DE ahead and neighbour positions DP ahead in shared-memory rings, so the loads of later
// entries are in flight while the current one is computed, without holding registers.
// Layout: ring_e[DE][BLOCK] uint32 and ring_p[DP][BLOCK] float4 (bank-conflict-free per thread).
__device__ __forceinline__ void cp_async4(void *smem, const void *gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem) : "memory");
}
// 16 bytes, cached in L2 only (records that are read once)
__device__ __forceinline__ void cp_async16_cg(void *smem, const void *gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// The entries of a row that a walk visits: c entries, the first c1 at list slots 0..c1-1, the rest
// after a gap of `gap` slots (the owned part's far band, skipped together with the other part's).
struct RowSpan {
  int c, c1, gap;
};
// Whole row [owned | not owned], each part ending with its far band (counts packed in nfar: owned in
// the low 16 bits).  skip: leave both far bands out.
__device__ __forceinline__ RowSpan full_row(int nnum, int nown, int nfar, bool skip) {
  if (!skip) return RowSpan{nnum, nnum, 0};
  const int of = nfar & 0xffff, nf = nfar >> 16;
  return RowSpan{nnum - of - nf, nown - of, of};
}
// The owned part only (each unordered pair once).
__device__ __forceinline__ RowSpan owned_row(int nown, int nfar, bool skip) {
  const int c = skip ? nown - (nfar & 0xffff) : nown;
  return RowSpan{c, c, 0};
}

// The per-atom extents of the neighbour list that the row walks read, and the control block whose
// skip_far says whether this evaluation leaves the far bands out (nullptr: never).
struct RowExt {
  const int32_t *nnum, *nown, *nband0, *nfar;
  const Control *ctrl;
};
__device__ __forceinline__ bool skip_far(const RowExt &X) { return X.ctrl != nullptr && X.ctrl->skip_far != 0; }
__device__ __forceinline__ RowSpan full_row(const RowExt &X, int i, bool skip) {
  return skip ? full_row(X.nnum[i], X.nown[i], X.nfar[i], true) : RowSpan{X.nnum[i], X.nnum[i], 0};
}
__device__ __forceinline__ RowSpan owned_row(const RowExt &X, int i, bool skip) {
  return skip ? owned_row(X.nown[i], X.nfar[i], true) : RowSpan{X.nown[i], X.nown[i], 0};
}

template <int DE, int DP, int BLOCK>
struct NbrPipe {
  static_assert(DE >= 2 * DP && DP >= 1, "entries must run at least twice as far ahead as positions");
  uint32_t *re;            // this thread's column of ring_e
  float4 *rp;              // this thread's column of ring_p
  const int32_t *row;      // &nbr[0 * n + i]
  size_t n;
  const float4 *pos;
  int cnt, c1, gap;        // the walked entries (RowSpan)

  // list slot of the k-th walked entry
  __device__ __forceinline__ size_t slot(int k) const { return (size_t)(k < c1 ? k : k + gap); }

  __device__ __forceinline__ void start(uint32_t *ring_e, float4 *ring_p, const int32_t *row_, size_t n_,
                                        const float4 *pos_, RowSpan sp) {
    re = ring_e + threadIdx.x; rp = ring_p + threadIdx.x; row = row_; n = n_; pos = pos_;
    cnt = sp.c; c1 = sp.c1; gap = sp.gap;
#pragma unroll
    for (int k = 0; k < DE; ++k)
      if (k < cnt) cp_async4(re + k * BLOCK, row + slot(k) * n);
    cp_async_commit();
    cp_async_wait<0>();
#pragma unroll
    for (int k = 0; k < DP; ++k) {
      if (k < cnt) cp_async16(rp + k * BLOCK, pos + (re[k * BLOCK] & J_MASK));
      cp_async_commit();
    }
  }
  __device__ __forceinline__ void start(uint32_t *ring_e, float4 *ring_p, const int32_t *row_, size_t n_,
                                        const float4 *pos_, int cnt_) {
    start(ring_e, ring_p, row_, n_, pos_, RowSpan{cnt_, cnt_, 0});
  }

  // Entry k (0 <= k < cnt, called for k = 0, 1, 2, ... in order): its packed list entry and the
  // neighbour's position; issues the copies for entries k + DE and k + DP.
  __device__ __forceinline__ void get(int k, uint32_t &e, float4 &p) {
    cp_async_wait<DP - 1>();
    e = re[(k % DE) * BLOCK];
    p = rp[(k % DP) * BLOCK];
    if (k + DE < cnt) cp_async4(re + ((k + DE) % DE) * BLOCK, row + slot(k + DE) * n);
    if (k + DP < cnt) cp_async16(rp + ((k + DP) % DP) * BLOCK, pos + (re[((k + DP) % DE) * BLOCK] & J_MASK));
    cp_async_commit();
  }

  __device__ __forceinline__ void finish() { cp_async_wait<0>(); }
};

// cp.async ring of pair records (16 bytes each, L2 only): record k of this thread is src[k * stride];
// DQ records in flight, as NbrPipe's positions.
template <int DQ, int BLOCK, int STRIDE>
struct RecPipe {
  float4 *rg;
  const float4 *base;   // the record array (a kernel parameter)
  unsigned off;         // element offset of record 0 of this thread
  int cnt;
  __device__ __forceinline__ void start(float4 *ring, const float4 *base_, unsigned off_, int cnt_) {
    rg = ring + threadIdx.x; base = base_; off = off_; cnt = cnt_;
#pragma unroll
    for (int k = 0; k < DQ; ++k) {
      if (k < cnt) cp_async16_cg(rg + k * BLOCK, base + (off + k * STRIDE));
      cp_async_commit();
    }
  }
  __device__ __forceinline__ float4 get(int k) {
    cp_async_wait<DQ - 1>();
    const float4 v = rg[(k % DQ) * BLOCK];
    if (k + DQ < cnt) cp_async16_cg(rg + ((k + DQ) % DQ) * BLOCK, base + (off + (k + DQ) * STRIDE));
    cp_async_commit();
    return v;
  }
  __device__ __forceinline__ void finish() { cp_async_wait<0>(); }
};

}  // namespace nep
