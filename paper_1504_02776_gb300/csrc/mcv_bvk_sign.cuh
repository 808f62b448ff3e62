// FP32 signs for the FP64 single-crystal kernel's root search, with a proven bound.
//
// An FP64 evaluation of g(Ef) = Ei - Ef - s hw_b(Q(Ef)) costs some 300 FP64 instructions (an
// eigen-solve and six sines), 64 cycles each, and the 33 nodes and 50 bisection steps took 84 of
// them.  The sign of g is that of omega_b against the energy transfer, i.e. how many eigenvalues
// of D lie below lambda* = (Ei - Ef)^2 / (hbar^2 phi/M): the sign changes along the leading
// minors of D - lambda* (Sturm), a few dozen FP32 operations.  BvkSign evaluates them with a
// bound on their FP32 errors and answers +1 or -1 only where all three are beyond it, else 0:
// FP64 decides the nodes and bisection steps left (5 to 10 per event), and a bracketed secant
// iteration takes the place of the remaining steps.  FP64 crystal, 5e4 neutrons: 25.1 -> 6.1 ms.
//
// The header also compiles as plain C++ (a CPU test checks the bound over cells, stiffnesses and
// energies there).
#pragma once

#include "mcv_params.h"

#ifdef __CUDACC__
#define MCV_BVK __device__ __forceinline__
#else
#include <cmath>
#define MCV_BVK inline
#endif

namespace mcv {

#ifdef __CUDACC__
MCV_BVK void bvk_sincos(float x, float* s, float* c) { sincosf(x, s, c); }
#else
void bvk_sincos(float x, float* s, float* c);  // the test's: with errors of its choice
#endif

// the entries of D - lambda* in units of phi/M (xx yy zz xy xz yz), the bound on their errors and
// on their magnitude
struct BvkMinors {
  float d0, d1, d2, e01, e02, e12;
  float m2, m3;  // the second and third leading minors; the first is d0
  float err, size;
};

struct BvkSign {
  float ax, ay, az, bx, by, bz;  // half-cell phases: a - kf b
  float ei, inv_hwu;
  float pa, pb;                  // |ax| + |ay| + |az|, |bx| + |by| + |bz|
  int b, sg;

  MCV_BVK void set_phases(float ax_, float ay_, float az_, float bx_, float by_, float bz_) {
    ax = ax_;
    ay = ay_;
    az = az_;
    bx = bx_;
    by = by_;
    bz = bz_;
    pa = fabsf(ax) + fabsf(ay) + fabsf(az);
    pb = fabsf(bx) + fabsf(by) + fabsf(bz);
  }

  // The errors, with u = 2^-24 (one FP32 rounding; division and square root are rounded
  // correctly, sine and cosine are within 2 units in the last place, 2^-23):
  //   phases:   kf carries 4.5 u, kf b 6.5 u, and a and the difference one u each: before the
  //             cancellation of a - kf b that is 7.5 u (|a| + kf |b|) of each phase, and an entry
  //             moves by at most four times one phase and twice the two others: 30 u = 1.8e-6
  //             of the sum over the three of |a| + kf |b|
  //   entries:  40 u = 2.4e-6 for sines, cosines and their products
  //   lambda*:  t carries 4 u (ei + ef) inv_hwu, so lambda* 9.1 u t (ei + ef) inv_hwu, and its
  //             subtraction one u of it: 6.1e-7 t (ei + ef) inv_hwu
  // The minors of entries that are within err, and at most S = 8 + lambda*, are within
  // (2 S + 4) err and (3 S^2 + 12 S + 36) err, and their own rounding within 3 u S^2 and
  // 6 u S^3: together below 4 S err and 12 S^2 err, since S >= 8 and err > 8e-7 lambda* + 2e-5.
  MCV_BVK BvkMinors minors(float ef, float t) const {
    const float kf = (float)kKPerV * sqrtf(ef / (float)kMeVPerV2);
    float sx, cx, sy, cy, sz, cz;
    bvk_sincos(ax - kf * bx, &sx, &cx);
    bvk_sincos(ay - kf * by, &sy, &cy);
    bvk_sincos(az - kf * bz, &sz, &cz);
    const float lam = t * t;
    BvkMinors m;
    m.d0 = 4.0f - 2.0f * cx * (cy + cz) - lam;
    m.d1 = 4.0f - 2.0f * cy * (cx + cz) - lam;
    m.d2 = 4.0f - 2.0f * cz * (cx + cy) - lam;
    m.e01 = 2.0f * sx * sy;
    m.e02 = 2.0f * sx * sz;
    m.e12 = 2.0f * sy * sz;
    m.m2 = m.d0 * m.d1 - m.e01 * m.e01;
    m.m3 = m.d2 * m.m2 - m.e12 * (m.d0 * m.e12 - m.e01 * m.e02) +
           m.e02 * (m.e01 * m.e12 - m.d1 * m.e02);
    m.err = 2e-6f * (10.0f + pa + kf * pb) + 8e-7f * t * (ei + ef) * inv_hwu;
    m.size = 8.0f + lam;
    return m;
  }

  // The sign of g(Ef), or 0 where FP32 does not decide it (an energy transfer below 0.1 % of
  // Ei + Ef among them).
  MCV_BVK int operator()(double Ef) const {
    const float ef = (float)Ef;
    const float t = (float)sg * (ei - ef) * inv_hwu;
    const BvkMinors m = minors(ef, t);
    if (!(t > 1e-3f * (ei + ef) * inv_hwu && fabsf(m.d0) > m.err &&
          fabsf(m.m2) > 4.0f * m.size * m.err && fabsf(m.m3) > 12.0f * m.size * m.size * m.err))
      return 0;
    const int below = (m.d0 < 0.0f) + ((m.m2 < 0.0f) != (m.d0 < 0.0f)) +
                      ((m.m3 < 0.0f) != (m.m2 < 0.0f));
    const bool lower = below > b;  // omega_b below the energy transfer
    return lower == (sg > 0) ? 1 : -1;
  }
};

}  // namespace mcv
