// nep_wide.cu -- descriptors, network and forces with G lanes per atom (sm_103a).
//
// The fused kernels of nep_force.cu give each atom one thread, which walks its row alone: 45 us from one block
// to one block per SM, whatever the atom count, since a warp then issues one instruction every three cycles.
// Systems that leave the chip empty that way (and the few atoms that a student's fallback hands to the
// teacher) take k_nep_wide: a group of G = 4, 8, 16 or 32 lanes shares an atom.
//   walk      the lanes stride over the neighbour row; entries inside the cutoff are compacted by ballot into
//             the group's shared memory (angular pairs from the front, the others from the back), radial
//             basis sums and LJ energy in registers, combined by shuffles;
//   sums      G angular pairs at a time: each lane writes one pair's channel functions g_n and solid harmonics
//             to shared memory, then owns NLM / G components and adds all channels over the staged pairs;
//   network   descriptors, neurons and their backward products distributed over the lanes (W0 in shared
//             memory, rows padded to an odd length so that both rows and columns are read without conflicts);
//   forces    the lanes stride over the compacted entries again, each evaluating whole pairs with the adjoint
//             row read from shared memory, and scatter d_ij as the fused kernels do.
// Everything of an atom stays inside its warp, so no block barrier is needed after the tables are staged.  The
// sums of a row are taken in a fixed order (lane, then shuffle tree), so results are reproducible bit for bit.
// MT = __nv_bfloat16 / __half rounds the network's operands (scaled descriptors, W0, backward factors) to that
// type before the float32 products, as the tensor-core form does with its GEMM operands, and takes its tanh from
// the special-function unit as well.
#include <algorithm>
#include <type_traits>

#include "nep_pair.cuh"

namespace nep {
namespace {

constexpr int WIDE_BLOCK = 128;
constexpr int WIDE_WARPS = WIDE_BLOCK / 32;
constexpr int WIDE_CAP = 128;          // entries per atom: the largest list capacity

// The model tables the lanes index (read from shared memory; the constant bank serves one address at a time).
// W0 by rows and by columns, zero-padded to whole 16-byte vectors: a product reads a lane's row and the atom's
// values four at a time, eight lanes' rows without bank conflicts.
template <class S>
struct __align__(16) WideNet {
  static constexpr int NV = (S::NDES + 3) / 4, NM = (S::NNEU + 3) / 4;      // vectors per row, per column
  static constexpr int LD = S::NDES > 16 ? 4 * NV + 4 : 4 * NV, LDT = 4 * NM + 4;
  float W0[S::NNEU * LD], W0t[S::NDES * LDT];
  float cR[S::NR * S::KR];
  float qs[S::NDES], b0[S::NNEU], w1[S::NNEU], norm[S::NLM];
};

// One atom's workspace.
template <class S>
struct __align__(16) WideAtom {
  uint32_t ent[WIDE_CAP];              // active list entries: angular from the front, others from the back
  float q[32], t[32];                  // scaled descriptors then dU/dq; backward factors (zero past the last)
  float Q[8];                          // radial sums, then the radial adjoint
  float g4[S::FOURBODY ? S::NA : 1][5];
};

// sum of w[k] v[k] over 4 N values, both on 16-byte boundaries.
template <int N>
__device__ __forceinline__ float dot4(const float *w, const float *v, float z0) {
  float2 a = pr(z0, 0.f), b = bc2(0.f);
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const float4 x = reinterpret_cast<const float4 *>(w)[k], y = reinterpret_cast<const float4 *>(v)[k];
    a = fma2(pr(x.x, x.y), pr(y.x, y.y), a);
    b = fma2(pr(x.z, x.w), pr(y.z, y.w), b);
  }
  return hsum(add2(a, b));
}

template <class S>
struct RowShared {
  const float *g;
  __device__ __forceinline__ void load(int k, float (&h)[S::NA][4]) const {
#pragma unroll
    for (int a = 0; a < S::NA; ++a) {
      const float4 v = *reinterpret_cast<const float4 *>(g + a * S::NLM + 4 * k);
      h[a][0] = v.x; h[a][1] = v.y; h[a][2] = v.z; h[a][3] = v.w;
    }
  }
};

template <int G>
__device__ __forceinline__ float group_sum(float v) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sums of the 8 values over the group, to dst[0..7] (lane gl holds value gl / (G / 8), or values 2 gl and 2 gl + 1).
template <int G>
__device__ __forceinline__ void group_sum8(const float (&v)[8], int gl, float *dst) {
  float a[4], b[2];
  const bool h0 = (gl & (G / 2)) != 0, h1 = (gl & (G / 4)) != 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float keep = h0 ? v[4 + k] : v[k], give = h0 ? v[k] : v[4 + k];
    a[k] = keep + __shfl_xor_sync(0xffffffffu, give, G / 2);
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const float keep = h1 ? a[2 + k] : a[k], give = h1 ? a[k] : a[2 + k];
    b[k] = keep + __shfl_xor_sync(0xffffffffu, give, G / 4);
  }
  if constexpr (G >= 8) {
    const bool h2 = (gl & (G / 8)) != 0;
    const float keep = h2 ? b[1] : b[0], give = h2 ? b[0] : b[1];
    float c = keep + __shfl_xor_sync(0xffffffffu, give, G / 8);
#pragma unroll
    for (int o = G / 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if ((gl & (G / 8 - 1)) == 0) dst[gl / (G / 8)] = c;
  } else {
    dst[2 * gl] = b[0];
    dst[2 * gl + 1] = b[1];
  }
}

template <class S, int G>
struct __align__(16) WideShared {
  float4 shift[27];
  WideAtom<S> ws[WIDE_WARPS * (32 / G)];
  WideNet<S> net;
  // one staged pair per lane; with rows of an odd length the lanes write their own rows, and the lanes of a
  // group read consecutive values of one row, G rows apart from the next group's, without bank conflicts
  // (when all pairs are summed, the groups' rows take the same memory: s', then the adjoint row, 16-byte vectors)
  static constexpr int STP = (S::NA + S::NLM) | 1, ROW = S::NA * S::NLM;
  static constexpr int STAGE = 32 * STP > 32 / G * ROW ? 32 * STP : 32 / G * ROW;
  static_assert(STAGE % 4 == 0 && ROW % 4 == 0, "16-byte rows");
  __align__(16) float stage[WIDE_WARPS][STAGE];
};

template <class S, class MT, int G, bool LIST>
__device__ __forceinline__ void wide_body(WideShared<S, G> &M, const Model<S> &P, const Geom &geom, const int n,
                                          const int m, const int32_t *__restrict__ list, const float4 *__restrict__ pos,
                                          const int32_t *__restrict__ nbr, const RowExt &X, float *__restrict__ usite,
                                          float *__restrict__ qout, unsigned long long *__restrict__ Ffix,
                                          const EvalSums &sums, int *__restrict__ status, const Fallback &fb) {
  constexpr bool MIX = !std::is_same<MT, float>::value;
  constexpr int NG = 32 / G;                           // atoms per warp
  constexpr int LD = WideNet<S>::LD, LDT = WideNet<S>::LDT, NV = WideNet<S>::NV, NM = WideNet<S>::NM;
  constexpr int STP = WideShared<S, G>::STP;
  constexpr int CPL = (S::NLM + G - 1) / G;            // components per lane
  constexpr int NP2 = 2 * solid_pairs(S::NLM);
  float4 *shift = M.shift;
  WideNet<S> &net = M.net;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gl = lane % G, grp = lane / G;
  int base = ((int)blockIdx.x * WIDE_WARPS + warp) * NG;
  const bool skip = skip_far(X);
  // an atom's row extent, first two entries per lane and first neighbour: loaded before the tables are staged
  // and at the end of the previous atom, so that the chain extent -> entry -> position starts early
  bool live;
  int i;
  RowSpan sp;
  float4 pi, pj;
  uint32_t e, e1;
  auto entry = [&](int k) -> uint32_t {                // the k-th walked entry of atom i
    return k < sp.c ? (uint32_t)nbr[(size_t)(k < sp.c1 ? k : k + sp.gap) * n + i] : 0u;
  };
  auto load_atom = [&]() {
    live = base + grp < m;
    i = live ? (LIST ? list[base + grp] : base + grp) : 0;
    sp = live ? full_row(X, i, skip) : RowSpan{0, 0, 0};
    pi = pos[i];
    e = entry(gl);
    e1 = entry(gl + G);
    pj = pos[e & J_MASK];
  };
  __shared__ long long wsum_d[WIDE_WARPS][5], wsum_f[WIDE_WARPS][13];
  if ((int)blockIdx.x * WIDE_WARPS * NG >= m) {        // a block without atoms only takes part in the closing count
    if (threadIdx.x < 32) eval_add<WIDE_WARPS>(sums, nullptr, nullptr);
    return;
  }
  load_atom();
  fill_shift_table(shift, geom);
  for (int t = threadIdx.x; t < 4 * NM * 4 * NV; t += WIDE_BLOCK) {
    const int mu = t / (4 * NV), v = t % (4 * NV);
    const float w = mu < S::NNEU && v < S::NDES ? round_to<MT>(P.W0[mu < S::NNEU ? mu : 0][v < S::NDES ? v : 0]) : 0.f;
    if (mu < S::NNEU) net.W0[mu * LD + v] = w;
    if (v < S::NDES) net.W0t[v * LDT + mu] = w;
  }
  for (int t = threadIdx.x; t < S::NR * S::KR; t += WIDE_BLOCK) net.cR[t] = P.cR[t / S::KR][t % S::KR];
  for (int t = threadIdx.x; t < S::NDES; t += WIDE_BLOCK) net.qs[t] = P.qs[t];
  for (int t = threadIdx.x; t < S::NNEU; t += WIDE_BLOCK) { net.b0[t] = P.b0[t]; net.w1[t] = P.w1[t]; }
  for (int t = threadIdx.x; t < S::NLM; t += WIDE_BLOCK) {
    float v = 0.f;
#pragma unroll
    for (int c = 0; c < S::NLM; ++c)
      if (t == c) v = solid_norm(S::NLM, c);
    net.norm[t] = v;
  }
  __syncthreads();
  const unsigned gmask = (G == 32 ? 0xffffffffu : ((1u << G) - 1u)), below = (1u << gl) - 1u;
  WideAtom<S> &A = M.ws[warp * NG + grp];
  float *st = M.stage[warp] + lane * STP;              // this lane's staged pair
  float *row = M.stage[warp] + grp * WideShared<S, G>::ROW;   // the atom's row
  for (int k = gl; k < 32; k += G) {
    if (k >= S::NDES) A.q[k] = 0.f;
    if (k >= S::NNEU) A.t[k] = 0.f;
  }
  const float *sg = M.stage[warp] + grp * G * STP;     // the group's
  long long acc_d[5] = {0, 0, 0, 0, 0}, acc_f[13] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
  const int per_pass = (int)gridDim.x * WIDE_WARPS * NG;
  for (; base < m; base += per_pass) {                 // warp-uniform
    auto offset_of = [&](uint32_t e, float4 pj, float &dx, float &dy, float &dz) {
      const float4 o = shift[e >> J_BITS];
      dx = pj.x - pi.x + o.x; dy = pj.y - pi.y + o.y; dz = pj.z - pi.z + o.z;
      return dx * dx + dy * dy + dz * dz;
    };

    // walk: entries one step further ahead than positions
    float2 Q[4] = {bc2(0.f), bc2(0.f), bc2(0.f), bc2(0.f)};
    float elj = 0.f;
    int na = 0, no = 0, nrad = 0;
    const int trip = __reduce_max_sync(0xffffffffu, (sp.c + G - 1) / G);
    for (int it = 0; it < trip; ++it) {
      const int k = it * G + gl;
      const uint32_t e2 = entry(k + 2 * G);
      const float4 p1 = pos[e1 & J_MASK];
      float dx, dy, dz;
      const float r2 = offset_of(e, pj, dx, dy, dz);
      const bool act = k < sp.c && r2 < P.rmax2, ang = act && r2 < P.rcA2;
      const unsigned ba = (__ballot_sync(0xffffffffu, ang) >> (grp * G)) & gmask;
      const unsigned bo = (__ballot_sync(0xffffffffu, act && !ang) >> (grp * G)) & gmask;
      if (act) A.ent[ang ? na + __popc(ba & below) : WIDE_CAP - 1 - (no + __popc(bo & below))] = e;
      na += __popc(ba);
      no += __popc(bo);
      if (act) {
        const float ir = rsqrtf(r2), r = r2 * ir;
        if (r2 < P.rcR2) {
          cheb_accumulate(r, P.inv_rcR, Q);
          ++nrad;
        }
        if (!LIST && P.lj_on != 0.f && r2 < P.lj_rc2) {
          float el, dl;
          lj_pair<S>(P, r2, r, ir, el, dl);
          elj = fmaf(0.5f, el, elj);
        }
      }
      e = e1; e1 = e2; pj = p1;
    }
    {
      float v[8];
      cheb_sums(Q, v);                                 // linear: the lanes' sums add up to the atom's
      group_sum8<G>(v, gl, A.Q);
    }
    elj = group_sum<G>(elj);
    __syncwarp();

    // angular sums, G pairs at a time
    float s[S::NA][CPL];
#pragma unroll
    for (int a = 0; a < S::NA; ++a)
#pragma unroll
      for (int c = 0; c < CPL; ++c) s[a][c] = 0.f;
    const int chunks = __reduce_max_sync(0xffffffffu, (na + G - 1) / G);
    for (int ch = 0; ch < chunks; ++ch) {
      const int p = ch * G + gl;
      const bool has = p < na;
      float r = 1.f, ux = 1.f, uy = 0.f, uz = 0.f;
      if (has) {
        const uint32_t ep = A.ent[p];
        float dx, dy, dz;
        const float r2 = offset_of(ep, pos[ep & J_MASK], dx, dy, dz);
        const float ir = rsqrtf(r2);
        r = r2 * ir; ux = dx * ir; uy = dy * ir; uz = dz * ir;
      }
      float g[S::NA];
      radial_channels<S>(P, r, has, g);                // zero without a pair
      const Solid<S::NLM> H(ux, uy, uz);
#pragma unroll
      for (int a = 0; a < S::NA; ++a) st[a] = g[a];
#pragma unroll
      for (int k = 0; k < S::NLM / 4; ++k) {
        float2 y01, y23;
        H.chunk(k, y01, y23);
        st[S::NA + 4 * k] = y01.x; st[S::NA + 4 * k + 1] = y01.y;
        st[S::NA + 4 * k + 2] = y23.x; st[S::NA + 4 * k + 3] = y23.y;
      }
      __syncwarp();
      const int cnt = __reduce_max_sync(0xffffffffu, min(G, na - ch * G));
#pragma unroll 2
      for (int q = 0; q < cnt; ++q) {
        const float *sq = sg + q * STP;
        float y[CPL];
#pragma unroll
        for (int c = 0; c < CPL; ++c) y[c] = gl + c * G < S::NLM ? sq[S::NA + gl + c * G] : 0.f;
#pragma unroll
        for (int a = 0; a < S::NA; ++a) {
          const float ga = sq[a];
#pragma unroll
          for (int c = 0; c < CPL; ++c) s[a][c] = fmaf(ga, y[c], s[a][c]);
        }
      }
      __syncwarp();                                    // read before the next chunk's pairs replace them
    }
#pragma unroll
    for (int c = 0; c < CPL; ++c)
      if (gl + c * G < S::NLM) {
#pragma unroll
        for (int a = 0; a < S::NA; ++a) row[a * S::NLM + gl + c * G] = s[a][c];
      }
    __syncwarp();

    // descriptors [q_n | q_nl | q4_n], one per lane and turn
    bool out = false;
    for (int d = gl; d < S::NDES; d += G) {
      float q;
      if (d < S::NR) {
        q = 0.f;
#pragma unroll
        for (int k = 0; k < S::KR; ++k) q = fmaf(net.cR[d * S::KR + k], A.Q[k], q);
      } else if (d < S::NR + S::NA * S::LMAX) {
        const int a = (d - S::NR) / S::LMAX, l = (d - S::NR) % S::LMAX + 1;
        const float z = net.norm[NP2 + l - 1] * row[a * S::NLM + NP2 + l - 1];
        q = z * z;
        for (int c = l * (l - 1); c < l * (l + 1); ++c) {
          const float v = net.norm[c] * row[a * S::NLM + c];
          q = fmaf(v, v, q);
        }
      } else {
        q = 0.f;
        if constexpr (S::FOURBODY) {
          // one channel's tensor: fourbody_tensors / fourbody_adjoint of a one-channel shape
          using One = Shape<1, 1, 8, 8, 4, true, 1>;
          const int a = d - S::NR - S::NA * S::LMAX;
          float s2[1][5], q1[One::NDES], g1[5];
#pragma unroll
          for (int p = 0; p < S::NLM; ++p) {
            const int m2 = solid_quadrupole(S::NLM, p);
            if (m2 >= 0) s2[0][m2 < 0 ? 0 : m2] = solid_norm(S::NLM, p) * row[a * S::NLM + p];
          }
          FourBody<One> T;
          fourbody_tensors<One>(s2, T, q1);
          q = q1[One::NR + One::NA * One::LMAX];
          fourbody_adjoint<One>(0, T, g1);
#pragma unroll
          for (int k = 0; k < 5; ++k) A.g4[a][k] = g1[k];
        }
      }
      if (!LIST && live && qout != nullptr) qout[(size_t)i * S::NDES + d] = q;
      const float qt = q * net.qs[d];
      if constexpr (S::NDES <= 16) {
        if (!LIST && fb.on) out |= (qt < fb.lo[d]) | (qt > fb.hi[d]);
      }
      A.q[d] = round_to<MT>(qt);
    }
    bool flagged = false;
    if constexpr (!LIST && S::NDES <= 16) {
      const unsigned any = __ballot_sync(0xffffffffu, out);   // by every lane, also those past the last atom
      flagged = live && fb.on && ((any >> (grp * G)) & gmask) != 0u;
      if (flagged && gl == 0) flag_atom(fb, i, status);
    }
    __syncwarp();

    // network: neurons, then their backward products
    float U = 0.f;
    for (int mu = gl; mu < S::NNEU; mu += G) {
      const float z = dot4<NV>(net.W0 + mu * LD, A.q, -net.b0[mu]);
      const float h = MIX && S::NLM > 8 ? tanh_sfu(z) : tanhf(z);   // as the forms of one thread per atom
      U = fmaf(net.w1[mu], h, U);
      A.t[mu] = round_to<MT>(net.w1[mu] * (1.f - h * h));
    }
    U = group_sum<G>(U) - P.b1;
    __syncwarp();                                      // t is complete, q has been read
    for (int v = gl; v < S::NDES; v += G) {
      const float d = dot4<NM>(net.W0t + v * LDT, A.t, 0.f);
      A.q[v] = flagged ? 0.f : d * net.qs[v];          // dU/dq
    }
    __syncwarp();

    // adjoint row G' = 2 norm^2 Fp s' + norm f4 g4 over the sums, radial adjoint over the radial sums
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
      const int p = gl + c * G;
      if (p < S::NLM) {
        const int l = p < NP2 ? (p < 2 ? 1 : (p < 6 ? 2 : (p < 12 ? 3 : 4))) : p - NP2 + 1;
        const float h = net.norm[p], hh = 2.f * h * h;
        int m2 = -1;
#pragma unroll
        for (int u = 0; u < S::NLM; ++u)
          if (u == p) m2 = solid_quadrupole(S::NLM, u);
#pragma unroll
        for (int a = 0; a < S::NA; ++a) {
          float gl_ = hh * A.q[S::NR + a * S::LMAX + l - 1] * s[a][c];
          if constexpr (S::FOURBODY) {
            if (m2 >= 0) gl_ = fmaf(h * A.q[S::NR + S::NA * S::LMAX + a], A.g4[a][m2], gl_);
          }
          row[a * S::NLM + p] = gl_;
        }
      }
    }
    for (int k = gl; k < 8; k += G) {
      float t = 0.f;
#pragma unroll
      for (int a = 0; a < S::NR; ++a) t = fmaf(A.q[a], net.cR[a * S::KR + k], t);
      A.Q[k] = t;
    }
    __syncwarp();
    float4 c0, c1;
    {
      float tail[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) tail[k] = A.Q[k];
      radial_tail_cubics(tail, c0, c1);
    }
    if (live && gl == 0) {
      const float ui = LIST ? U : (flagged ? elj : U + elj);
      if (LIST) usite[i] += U;                         // the student's kernel left the LJ energy there
      else usite[i] = ui;
      if (!isfinite(ui)) atomicOr(status, ST_NAN);
      acc_d[0] += to_fix32(ui);
      acc_d[2] += na;
      acc_d[3] += sp.c;
      acc_d[4] += na + no;
    }
    acc_d[1] += nrad;

    // forces: the compacted entries, angular ones first
    const RowShared<S> adjoint{row};
    float fx = 0.f, fy = 0.f, fz = 0.f;
    float wxx = 0.f, wxy = 0.f, wxz = 0.f, wyy = 0.f, wyz = 0.f, wzz = 0.f;
    const int nact = na + no;
    const int ftrip = __reduce_max_sync(0xffffffffu, (nact + G - 1) / G);
    auto active = [&](int p) -> uint32_t {
      return p < nact ? A.ent[p < na ? p : WIDE_CAP - 1 - (p - na)] : 0u;
    };
    e = active(gl);
    pj = pos[e & J_MASK];
    for (int it = 0; it < ftrip; ++it) {
      const int p = it * G + gl;
      const uint32_t en = active(p + G);
      const float4 pn = pos[en & J_MASK];
      const bool valid = p < nact, ang = p < na;
      float dx = 1.f, dy = 0.f, dz = 0.f, r2 = 1.f;
      if (valid) r2 = offset_of(e, pj, dx, dy, dz);
      const float ir = rsqrtf(r2), r = r2 * ir;
      float coef = valid ? radial_lj_coef<S, false, !LIST>(P, c0, c1, r2, r, ir) : 0.f;
      float vx = 0.f, vy = 0.f, vz = 0.f;
      if (ang) {
        float ca;
        angular_pair_solid<S>(P, adjoint, false, r, ir, dx, dy, dz, ca, vx, vy, vz);
        coef += ca;
      }
      if (valid) {
        const int j = (int)(e & J_MASK);
        const float Dx = fmaf(coef, dx, vx), Dy = fmaf(coef, dy, vy), Dz = fmaf(coef, dz, vz);
        fx += Dx; fy += Dy; fz += Dz;
        long long ox, oy, oz;
        to_fix32x3(-Dx, -Dy, -Dz, ox, oy, oz);
        red_add(Ffix + j, ox);
        red_add(Ffix + (size_t)n + j, oy);
        red_add(Ffix + 2 * (size_t)n + j, oz);
        wxx = fmaf(dx, Dx, wxx); wxy = fmaf(dx, Dy, wxy); wxz = fmaf(dx, Dz, wxz);
        wyy = fmaf(dy, Dy, wyy); wyz = fmaf(dy, Dz, wyz); wzz = fmaf(dz, Dz, wzz);
      }
      e = en; pj = pn;
    }
    fx = group_sum<G>(fx); fy = group_sum<G>(fy); fz = group_sum<G>(fz);
    if (live && gl == 0) {
      red_add(Ffix + i, to_fix32(fx));
      red_add(Ffix + (size_t)n + i, to_fix32(fy));
      red_add(Ffix + 2 * (size_t)n + i, to_fix32(fz));
      if (!(isfinite(fx) && isfinite(fy) && isfinite(fz))) atomicOr(status, ST_NAN);
    }
    // W = -sum of r_ij (x) d_ij, upper triangle (symmetric: U_i is rotation invariant)
    acc_f[0] -= to_fix32(wxx); acc_f[1] -= to_fix32(wxy); acc_f[2] -= to_fix32(wxz);
    acc_f[4] -= to_fix32(wyy); acc_f[5] -= to_fix32(wyz); acc_f[8] -= to_fix32(wzz);
    base += per_pass;
    if (base < m) load_atom();                         // warp-uniform
    base -= per_pass;
    __syncwarp();                                      // the workspace is the warp's next atoms'
  }
  acc_f[3] = acc_f[1]; acc_f[6] = acc_f[2]; acc_f[7] = acc_f[5];
  if constexpr (LIST) {
    // the counts are the student's; these atoms only add energy and virial
    acc_d[1] = acc_d[2] = acc_d[3] = acc_d[4] = 0;
  } else {
    // the force pass visits the walk's active pairs
    acc_f[9] = acc_d[3]; acc_f[10] = acc_d[4]; acc_f[11] = acc_d[1]; acc_f[12] = acc_d[2];
  }
  warp_sum_stage<5>(acc_d, wsum_d[warp]);
  warp_sum_stage<13>(acc_f, wsum_f[warp]);
  __syncthreads();
  eval_add<WIDE_WARPS>(sums, wsum_d, wsum_f);
}

// One evaluation of all n atoms.
template <class S, class MT, int G>
__global__ void __launch_bounds__(WIDE_BLOCK, 4)
k_nep_wide(const __grid_constant__ Model<S> P, const Geom geom, const int n, const float4 *__restrict__ pos,
           const int32_t *__restrict__ nbr, const RowExt X, float *__restrict__ usite, float *__restrict__ qout,
           unsigned long long *__restrict__ Ffix, const EvalSums sums, int *__restrict__ status,
           const __grid_constant__ Fallback fb) {
  extern __shared__ __align__(16) unsigned char raw[];
  wide_body<S, MT, G, false>(*reinterpret_cast<WideShared<S, G> *>(raw), P, geom, n, n, nullptr, pos, nbr, X, usite, qout, Ffix, sums, status, fb);
}

// The fallback model on the first min(*count, cap) atoms of list: only its network's part is added to usite, to
// the forces and to the partial sums (the pair term is the student's).  Few flagged atoms take a warp each, many
// a quarter of one: at 131,072 atoms 20 us against 27 for 1,311 flagged ones, 39 against 35 for 6,554, 440 against 272
// for all (eager times, with 6 us of launch).  The two kernels of one thread per flagged
// atom that this replaces took 70 us from one to 16,384 flagged atoms (their serial row walk), 322 for 131,072, 549 for
// 262,400 (this: 544), and less than this only above 450,000: 992 against 1,007 for 500,000, 2,011 against 2,097 for
// 1,048,576.  Not kept for those: eight lanes alone (2,029 there, but 28 us instead of 18 for a few flagged atoms, which
// is what a range is set for), and four lanes above 81,920 flagged ones (1,859, but 56 KB of shared memory per block
// instead of 40, taken from L1: 55 us instead of 46 for 7,805 of 780,448 atoms).
constexpr int LIST_WARP_MAX = 4096;
template <class S>
__global__ void __launch_bounds__(WIDE_BLOCK, 4)
k_nep_wide_list(const __grid_constant__ Model<S> P, const Geom geom, const int n, const int32_t *__restrict__ list,
                const int *__restrict__ count, const int cap, const float4 *__restrict__ pos,
                const int32_t *__restrict__ nbr, const RowExt X, float *__restrict__ usite,
                unsigned long long *__restrict__ Ffix, const EvalSums sums, int *__restrict__ status) {
  __shared__ __align__(16) unsigned char raw[sizeof(WideShared<S, 8>)];
  static_assert(sizeof(WideShared<S, 8>) >= sizeof(WideShared<S, 32>), "one buffer for both splits");
  const int m = min(*count, cap);
  if (blockIdx.x == 0 && threadIdx.x == 0)
    atomicAdd(reinterpret_cast<unsigned long long *>(sums.counters + 9), (unsigned long long)m);
  const Fallback none{};
  if (m <= LIST_WARP_MAX)
    wide_body<S, float, 32, true>(reinterpret_cast<WideShared<S, 32> &>(raw), P, geom, n, m, list, pos, nbr, X, usite,
                                  nullptr, Ffix, sums, status, none);
  else
    wide_body<S, float, 8, true>(reinterpret_cast<WideShared<S, 8> &>(raw), P, geom, n, m, list, pos, nbr, X, usite,
                                 nullptr, Ffix, sums, status, none);
}

// Blocks that fit on the device at once, or fewer for few atoms; the kernels loop.
template <class K>
int wide_grid(K kernel, int atoms, int lanes, size_t smem) {
  int d = 0, sms = 0, per = 0;
  if ((smem > 48 * 1024 && cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) ||
      cudaGetDevice(&d) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, d) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, WIDE_BLOCK, smem) != cudaSuccess || sms * per <= 0) {
    cudaGetLastError();
    sms = 152;
    per = 1;
  }
  const long long need = ((long long)atoms * lanes + WIDE_BLOCK - 1) / WIDE_BLOCK;
  return (int)std::max(1ll, std::min(need, (long long)sms * per));
}

}  // namespace

// Lanes per atom for a system of n atoms, 0: one thread per atom (the fused kernels of nep_force.cu).  The last
// two lines are where all atoms still fit the resident warps at once (608 blocks of 16 and of 32 atoms).  Measured per
// evaluation of the teacher (eager, with the launch's own 7 us), one thread per atom, then 4 / 8 / 16 / 32 lanes:
// 256 atoms 49, 30 / 23 / 19 / 17 us; 2,048 49, 32 / 24 / 21 / 23; 4,000 50, 32 / 26 / 27 / 29; 6,912 50,
// 36 / 30 / 36 / 38; 10,976 51, 42 / 43 / 46 / 50; 16,384 51 (MD step 60.3), 49 (58.0) / 52 (61.3) / 57 / 67; 23,328 64,
// 69 / 62 / 73 / 88; 32,000 66, 81 / 80 / 92 / 113, where the wide forms' extra work is no longer
// hidden.  The student (39 us with one thread per atom up to 16,384 atoms; 19 at 4,000 with 16, 22 at 6,912 with 8,
// 34 at 16,384 with 4) and the mixed forms cross at the same sizes.
int wide_lanes(int n) { return n <= 1024 ? 32 : (n <= 4096 ? 16 : (n <= 9728 ? 8 : (n <= 19456 ? 4 : 0))); }

// One force evaluation with `lanes` (4, 8, 16 or 32) lanes per atom; Ffix must be zero.
template <class S, class MT>
cudaError_t launch_wide(int lanes, const Model<S> &P, const Geom &g, int n, const float4 *pos, const int32_t *nbr,
                        const RowExt &X, float *usite, float *qout, long long *Ffix, const EvalSums &sums,
                        int *status, const Fallback &fb, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  auto run = [&](auto kernel, int g_lanes, size_t smem) {
    kernel<<<wide_grid(kernel, n, g_lanes, smem), WIDE_BLOCK, smem, st>>>(
        P, g, n, pos, nbr, X, usite, qout, reinterpret_cast<unsigned long long *>(Ffix), sums, status, fb);
  };
  if (lanes == 32) run(k_nep_wide<S, MT, 32>, 32, sizeof(WideShared<S, 32>));
  else if (lanes == 16) run(k_nep_wide<S, MT, 16>, 16, sizeof(WideShared<S, 16>));
  else if (lanes == 8) run(k_nep_wide<S, MT, 8>, 8, sizeof(WideShared<S, 8>));
  else run(k_nep_wide<S, MT, 4>, 4, sizeof(WideShared<S, 4>));
  return cudaGetLastError();
}

// The fallback model on the flagged atoms (list, count on the device): its site energies are added to usite and to
// the running energy, its forces to Ffix, its virial to the running virial, the atom count to counters[9].
template <class S>
cudaError_t launch_wide_list(const Model<S> &P, const Geom &g, int n, const float4 *pos, const int32_t *nbr,
                             const RowExt &X, const int *list, const int *count, int cap, float *usite, long long *Ffix,
                             const EvalSums &sums, int *status, cudaStream_t st) {
  if (n <= 0 || cap <= 0) return cudaSuccess;
  k_nep_wide_list<S><<<wide_grid(k_nep_wide_list<S>, cap, 32, 0), WIDE_BLOCK, 0, st>>>(
      P, g, n, list, count, cap, pos, nbr, X, usite, reinterpret_cast<unsigned long long *>(Ffix), sums, status);
  return cudaGetLastError();
}
template cudaError_t launch_wide_list<CuShape>(const Model<CuShape> &, const Geom &, int, const float4 *, const int32_t *,
                                               const RowExt &, const int *, const int *, int, float *, long long *,
                                               const EvalSums &, int *, cudaStream_t);

#define NEP_INSTANTIATE(SH, MT)                                                                                     \
  template cudaError_t launch_wide<SH, MT>(int, const Model<SH> &, const Geom &, int, const float4 *, const int32_t *, \
                                           const RowExt &, float *, float *, long long *, const EvalSums &, int *,    \
                                           const Fallback &, cudaStream_t);
NEP_INSTANTIATE(CuShape, float)
NEP_INSTANTIATE(CuShape, __nv_bfloat16)
NEP_INSTANTIATE(CuShape, __half)
NEP_INSTANTIATE(StudentShape, float)
NEP_INSTANTIATE(StudentShape, __nv_bfloat16)
NEP_INSTANTIATE(StudentShape, __half)
#undef NEP_INSTANTIATE

}  // namespace nep
