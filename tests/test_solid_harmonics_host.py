"""The fused kernels' solid harmonics (csrc/nep_solid.cuh), compiled for the host and run on the CPU.

solid_norm x Solid must be the normalised harmonics of nep_common.cuh (both rows of the same degree span the
same space; here component by component, matched by name), and SolidGrad, which uses the relations between the
degrees instead of gradient polynomials, must give sum_lm b_lm grad R_lm.  Both on seeded unit vectors and on
the axes, for the two compiled degrees; the cubics of cheb_to_cubics against the Chebyshev sum they stand for."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2604_24816_gb300", "csrc")

PROGRAM = r"""
#include "nep_solid.cuh"
#include <cmath>
#include <cstdio>
#include <cstdint>
using namespace nep;
static uint64_t state = 0x9E3779B97F4A7C15ull;
static double uniform() {                      // splitmix64 -> [-1, 1)
  uint64_t z = (state += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return 2.0 * (double)((z ^ (z >> 31)) >> 11) * 0x1.0p-53 - 1.0;
}
// the normalised component of position p: degree l lists m = -l..l from l^2 - 1 on, S_lm at -m, C_lm at +m
template <int NLM>
static int component(int p) {
  const int l = solid_l(NLM, p), m = solid_m(NLM, p);
  const bool sine = m > 0 && p % 2 == 1;
  return l * l - 1 + l + (sine ? -m : m);
}
template <int NLM>
static void check(double *ev, double *eg) {
  for (int t = 0; t < 20006; ++t) {
    double v[3] = {uniform(), uniform(), uniform()};
    if (t < 6) for (int d = 0; d < 3; ++d) v[d] = t % 3 == d ? (t < 3 ? 1.0 : -1.0) : 0.0;
    const double n = sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
    if (n < 1e-3) continue;
    const float x = (float)(v[0] / n), y = (float)(v[1] / n), z = (float)(v[2] / n);
    const Solid<NLM> H(x, y, z);
    float Y[NLM], s[NLM], b[NLM];
    harmonics<NLM>(x, y, z, Y);
    for (int k = 0; k < NLM / 4; ++k) {
      float2 a, c;
      H.chunk(k, a, c);
      s[4 * k] = a.x; s[4 * k + 1] = a.y; s[4 * k + 2] = c.x; s[4 * k + 3] = c.y;
    }
    double g[3] = {0, 0, 0};
    for (int p = 0; p < NLM; ++p) {
      *ev = fmax(*ev, fabs((double)solid_norm(NLM, p) * s[p] - Y[component<NLM>(p)]));
      b[p] = (float)uniform() * solid_norm(NLM, p);   // weights over R: G' = norm G
      float a[3];
      harmonic_grad(component<NLM>(p), x, y, z, a);
      // the normalised polynomials are homogeneous forms of their degree, as R_lm: the same function
      for (int d = 0; d < 3; ++d) g[d] += (double)b[p] / solid_norm(NLM, p) * a[d];
    }
    constexpr int NP = solid_pairs(NLM);
    float2 bp[NP];
    for (int k = 0; k < NP; ++k) bp[k] = make_float2(b[2 * k], b[2 * k + 1]);
    SolidGrad G;
    G.add<1>(H, bp, b[2 * NP]);
    G.add<2>(H, bp + 1, b[2 * NP + 1]);
    if constexpr (NLM == 24) {
      G.add<3>(H, bp + 3, b[2 * NP + 2]);
      G.add<4>(H, bp + 6, b[2 * NP + 3]);
    }
    float q[3];
    G.get(q[0], q[1], q[2]);
    for (int d = 0; d < 3; ++d) *eg = fmax(*eg, fabs(g[d] - q[d]));
  }
}
int main() {
  double v24 = 0, g24 = 0, v8 = 0, g8 = 0, ec = 0;
  check<24>(&v24, &g24);
  check<8>(&v8, &g8);
  for (int t = 0; t < 2000; ++t) {
    double c[8], e[4], o[4], T0 = 1, x = uniform(), T1 = x, want = 0;
    for (int k = 0; k < 8; ++k) {
      c[k] = uniform();
      want += c[k] * (T0 + 1);
      const double T2 = 2 * x * T1 - T0;
      T0 = T1; T1 = T2;
    }
    cheb_to_cubics(c, e, o);
    const double y = 2 * x * x - 1;
    const double got = ((e[3] * y + e[2]) * y + e[1]) * y + e[0] + x * (((o[3] * y + o[2]) * y + o[1]) * y + o[0]);
    ec = fmax(ec, fabs(got - want));
  }
  printf("%.6e %.6e %.6e %.6e %.6e\n", v24, g24, v8, g8, ec);
  return 0;
}
"""


def test_solid_harmonics_and_their_weighted_gradient(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src = tmp_path / "solid_check.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "solid_check"
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "--expt-relaxed-constexpr",
                        "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-o", str(exe), str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    v24, g24, v8, g8, ec = map(float, subprocess.run([str(exe)], capture_output=True, text=True,
                                                     check=True).stdout.split())
    # values below 1: a dozen roundings of 2^-24 with intermediate terms up to 35/8 (l = 4)
    assert v24 < 12 * 2 ** -24 * 35 / 8 and v8 < 12 * 2 ** -24, (v24, v8)
    # gradients: 24 (8) weights up to 1, each |grad Yh_lm| <= l(l+1)/sqrt(2) < 15 (3), some ten roundings each
    assert g24 < 24 * 15 * 10 * 2 ** -24 and g8 < 8 * 3 * 10 * 2 ** -24, (g24, g8)
    assert ec < 1e-13, ec
