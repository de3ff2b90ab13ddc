"""The kernels' harmonic helpers (csrc/nep_common.cuh), compiled by nvcc for the host and run on the CPU.

The normalised harmonics Yh_lm and their gradients (harmonics, harmonic_grad, with the zero pattern harmonic_grad_mask:
the separate force kernels, the training kernels) against an independent form written here: polynomials Ph_lm with
small integer coefficients, Yh_lm = hnorm(lm) Ph_lm, on seeded points on and off the unit sphere (the gradients treat
x, y, z as free variables).  The fused kernels' solid harmonics are compared with the same helpers in
test_solid_harmonics_host.py; the GPU parity tests pin both against the FP64 oracle (descriptors, forces).
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2604_24816_gb300", "csrc")

PROGRAM = r"""
#include "nep_common.cuh"
#include <cmath>
#include <cstdio>
#include <cstdint>
using namespace nep;

// Yh_lm = hnorm(lm) Ph_lm, with Ph_lm a polynomial with small integer coefficients
static constexpr float hnorm(int lm) {
  constexpr float s3 = 1.7320508075688772f, s5 = 2.2360679774997896f, s6 = 2.449489742783178f;
  constexpr float s10 = 3.1622776601683795f, s15 = 3.872983346207417f, s35 = 5.916079783099616f;
  constexpr float s70 = 8.366600265340756f;
  return lm < 3 ? 1.f : lm == 3 || lm == 4 || lm == 6 ? s3 : lm == 5 ? 1.f : lm == 7 ? 0.5f * s3 :
         lm == 8 || lm == 14 ? 0.25f * s10 : lm == 9 ? s15 : lm == 10 || lm == 12 ? 0.25f * s6 :
         lm == 11 ? 1.f : lm == 13 ? 0.5f * s15 : lm == 15 ? 0.5f * s35 : lm == 16 || lm == 22 ? 0.25f * s70 :
         lm == 17 ? 0.5f * s5 : lm == 18 || lm == 20 ? 0.25f * s10 : lm == 19 ? 0.125f :
         lm == 21 ? 0.25f * s5 : 0.125f * s35;
}

template <int NLM>
static void harmonics_p(float x, float y, float z, float (&P)[NLM]) {
  static_assert(NLM == 8 || NLM == 24, "l_max 2 or 4");
  const float x2 = x * x, y2 = y * y, z2 = z * z;
  const float xy = x * y, yz = y * z, xz = x * z, d = x2 - y2, e = x2 + y2;
  P[0] = y; P[1] = z; P[2] = x;
  P[3] = xy;
  P[4] = yz;
  P[5] = fmaf(-0.5f, e, z2);
  P[6] = xz;
  P[7] = d;
  if constexpr (NLM > 8) {
  const float a3 = fmaf(4.f, z2, -e);          // 4 z^2 - x^2 - y^2
  const float p8 = y * fmaf(3.f, x2, -y2);     // y (3 x^2 - y^2)
  const float p14 = x * fmaf(-3.f, y2, x2);    // x (x^2 - 3 y^2)
  P[8] = p8;
  P[9] = xy * z;
  P[10] = y * a3;
  P[11] = z * fmaf(-1.5f, e, z2);
  P[12] = x * a3;
  P[13] = z * d;
  P[14] = p14;
  const float b4 = fmaf(6.f, z2, -e);          // 7 z^2 - r^2
  const float c4 = fmaf(-3.f, e, 4.f * z2);    // 7 z^2 - 3 r^2
  const float rr = e + z2;
  P[15] = xy * d;
  P[16] = z * p8;
  P[17] = xy * b4;
  P[18] = yz * c4;
  P[19] = fmaf(35.f * z2, z2, fmaf(-30.f * z2, rr, 3.f * rr * rr));
  P[20] = xz * c4;
  P[21] = d * b4;
  P[22] = z * p14;
  P[23] = fmaf(x2, x2, fmaf(-6.f * x2, y2, y2 * y2));
  }
}

// Ph_lm alone (lm a compile-time constant after unrolling).
static float harmonic_p(int lm, float x, float y, float z) {
  const float x2 = x * x, y2 = y * y, z2 = z * z;
  const float xy = x * y, d = x2 - y2, e = x2 + y2;
  switch (lm) {
    case 0: return y;
    case 1: return z;
    case 2: return x;
    case 3: return xy;
    case 4: return y * z;
    case 5: return fmaf(-0.5f, e, z2);
    case 6: return x * z;
    case 7: return d;
    case 8: return y * fmaf(3.f, x2, -y2);
    case 9: return xy * z;
    case 10: return y * fmaf(4.f, z2, -e);
    case 11: return z * fmaf(-1.5f, e, z2);
    case 12: return x * fmaf(4.f, z2, -e);
    case 13: return z * d;
    case 14: return x * fmaf(-3.f, y2, x2);
    case 15: return xy * d;
    case 16: return z * (y * fmaf(3.f, x2, -y2));
    case 17: return xy * fmaf(6.f, z2, -e);
    case 18: return (y * z) * fmaf(-3.f, e, 4.f * z2);
    case 19: { const float rr = e + z2; return fmaf(35.f * z2, z2, fmaf(-30.f * z2, rr, 3.f * rr * rr)); }
    case 20: return (x * z) * fmaf(-3.f, e, 4.f * z2);
    case 21: return d * fmaf(6.f, z2, -e);
    case 22: return z * (x * fmaf(-3.f, y2, x2));
    case 23: return fmaf(x2, x2, fmaf(-6.f * x2, y2, y2 * y2));
    default: return 0.f;
  }
}

// Gradient of Ph_lm at (x, y, z) (harmonic_grad / hnorm(lm)); the same zero pattern (harmonic_grad_mask).
static void harmonic_grad_p(int lm, float x, float y, float z, float (&a)[3]) {
  const float x2 = x * x, y2 = y * y, z2 = z * z;
  const float xy = x * y, yz = y * z, xz = x * z, d = x2 - y2, e = x2 + y2;
  float ax = 0.f, ay = 0.f, az = 0.f;
  switch (lm) {
    case 0: ay = 1.f; break;
    case 1: az = 1.f; break;
    case 2: ax = 1.f; break;
    case 3: ax = y; ay = x; break;
    case 4: ay = z; az = y; break;
    case 5: ax = -x; ay = -y; az = 2.f * z; break;
    case 6: ax = z; az = x; break;
    case 7: ax = 2.f * x; ay = -2.f * y; break;
    case 8: ax = 6.f * xy; ay = 3.f * d; break;
    case 9: ax = yz; ay = xz; az = xy; break;
    case 10: ax = -2.f * xy; ay = fmaf(4.f, z2, -fmaf(3.f, y2, x2)); az = 8.f * yz; break;
    case 11: ax = -3.f * xz; ay = -3.f * yz; az = fmaf(-1.5f, e, 3.f * z2); break;
    case 12: ax = fmaf(4.f, z2, -fmaf(3.f, x2, y2)); ay = -2.f * xy; az = 8.f * xz; break;
    case 13: ax = 2.f * xz; ay = -2.f * yz; az = d; break;
    case 14: ax = 3.f * d; ay = -6.f * xy; break;
    case 15: ax = y * fmaf(3.f, x2, -y2); ay = x * fmaf(-3.f, y2, x2); break;
    case 16: ax = 6.f * xy * z; ay = 3.f * z * d; az = y * fmaf(3.f, x2, -y2); break;
    case 17: ax = y * fmaf(6.f, z2, -fmaf(3.f, x2, y2)); ay = x * fmaf(6.f, z2, -fmaf(3.f, y2, x2));
             az = 12.f * xy * z; break;
    case 18: ax = -6.f * xy * z; ay = z * fmaf(4.f, z2, -fmaf(9.f, y2, 3.f * x2));
             az = 3.f * y * fmaf(4.f, z2, -e); break;
    case 19: { const float w = fmaf(-4.f, z2, e);   // x^2 + y^2 - 4 z^2
               ax = 12.f * x * w; ay = 12.f * y * w; az = -16.f * z * fmaf(3.f, e, -2.f * z2); break; }
    case 20: ax = z * fmaf(4.f, z2, -fmaf(9.f, x2, 3.f * y2)); ay = -6.f * xy * z;
             az = 3.f * x * fmaf(4.f, z2, -e); break;
    case 21: ax = -4.f * x * fmaf(-3.f, z2, x2); ay = 4.f * y * fmaf(-3.f, z2, y2); az = 12.f * z * d; break;
    case 22: ax = 3.f * z * d; ay = -6.f * xy * z; az = x * fmaf(-3.f, y2, x2); break;
    case 23: ax = 4.f * x * fmaf(-3.f, y2, x2); ay = -4.f * y * fmaf(3.f, x2, -y2); break;
    default: break;
  }
  a[0] = ax; a[1] = ay; a[2] = az;
}

static uint64_t state = 0x9E3779B97F4A7C15ull;
static double uniform() {                      // splitmix64 -> [0, 1)
  uint64_t z = (state += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return (double)((z ^ (z >> 31)) >> 11) * 0x1.0p-53;
}

int main() {
  double ey = 0, eg = 0, ep = 0, e8 = 0;
  int mask_bad = 0;
  for (int t = 0; t < 20000; ++t) {
    double v[3], n2 = 0;
    for (int d = 0; d < 3; ++d) { v[d] = 3.0 * uniform() - 1.5; n2 += v[d] * v[d]; }
    const double s = (t & 1) ? 1.0 / sqrt(n2) : 1.0;   // odd points on the unit sphere
    const float x = (float)(v[0] * s), y = (float)(v[1] * s), z = (float)(v[2] * s);
    const double scale = fmax(1.0, pow(sqrt((double)x * x + (double)y * y + (double)z * z), 4));
    float Y[24], P[24], Y8[8], P8[8];
    harmonics<24>(x, y, z, Y);
    harmonics_p<24>(x, y, z, P);
    harmonics<8>(x, y, z, Y8);
    harmonics_p<8>(x, y, z, P8);
    for (int lm = 0; lm < 24; ++lm) {
      ey = fmax(ey, fabs(Y[lm] - (double)hnorm(lm) * P[lm]) / scale);
      ep = fmax(ep, fabs(P[lm] - harmonic_p(lm, x, y, z)) / scale);
      if (lm < 8) e8 = fmax(e8, fabs(Y8[lm] - (double)hnorm(lm) * P8[lm]) / scale);
      float a[3], b[3];
      harmonic_grad(lm, x, y, z, a);
      harmonic_grad_p(lm, x, y, z, b);
      const int m = harmonic_grad_mask(lm);
      for (int d = 0; d < 3; ++d) {
        eg = fmax(eg, fabs(a[d] - (double)hnorm(lm) * b[d]) / scale);
        if (!((m >> d) & 1) && (a[d] != 0.f || b[d] != 0.f)) ++mask_bad;
      }
    }
  }
  printf("%.6e %.6e %.6e %.6e %d\n", ey, eg, ep, e8, mask_bad);
  return 0;
}
"""


def test_unnormalised_harmonics_reproduce_the_normalised_ones(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src = tmp_path / "harmonics_check.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "harmonics_check"
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "--expt-relaxed-constexpr",
                        "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-o", str(exe), str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    ey, eg, ep, e8, mask_bad = float(out[0]), float(out[1]), float(out[2]), float(out[3]), int(out[4])
    # float32 evaluation of degree <= 4 polynomials with |coefficients| <= 35 (times |r|^4 off the
    # sphere): a few units of 2^-24 relative to the largest term
    assert ey < 2e-5 and e8 < 2e-5, (ey, e8)
    assert eg < 5e-5, eg
    assert ep == 0.0, ep              # harmonic_p is the same arithmetic as harmonics_p, component by component
    assert mask_bad == 0
