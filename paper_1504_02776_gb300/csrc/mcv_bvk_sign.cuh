// FP32 signs for the FP64 single-crystal kernel's root search, with a proven bound.
//
// An FP64 evaluation of g(Ef) = Ei - Ef - s hw_b(Q(Ef)) costs some 300 FP64 instructions (an
// eigen-solve and six sines), 64 cycles each, and the 33 nodes and 50 bisection steps took 84 of
// them.  The sign of g is that of omega_b against the energy transfer, i.e. how many eigenvalues
// of D lie below lambda* = (Ei - Ef)^2 / (hbar^2 phi/M): the sign changes along the leading
// minors of D - lambda* (Sturm), a few dozen FP32 operations.  BvkSign evaluates them with a
// bound on their FP32 errors and answers +1 or -1 only where all three are beyond it, else 0:
// FP64 decides those (bracket_root).  The bound follows the entries' and cofactors' values: it
// leaves 0.01 % of the points open where the signs are not (and the node at Ef = Ei), against
// 2.2 % with one from the largest values they can have.  FP64 crystal, 5e4 neutrons: 25.1 ms
// with FP64 throughout, 5.3 ms, and 8.3 ms with the wider bound.
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

// the entries of D - lambda* in units of phi/M (xx yy zz xy xz yz), the second and third leading
// minors (the first is d0), and the bounds on the errors of the entries and of the minors
struct BvkMinors {
  float d0, d1, d2, e01, e02, e12;
  float m2, m3;
  float err, err2, err3;
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
  // The minors of entries that are within err: a minor moves by err times the sum of its
  // cofactors' magnitudes (off-diagonal ones twice), plus 2 err^2 (second) and 2 err^2 times the
  // sum of the entries' magnitudes (third: adj(E) is at most 2 err^2), plus its own rounding, at
  // most 3 u and 5 u of the sum of its products' magnitudes; 1.1 for the rounding of the bounds
  // and the terms err^3.
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
    const float c00 = m.d1 * m.d2 - m.e12 * m.e12, c11 = m.d0 * m.d2 - m.e02 * m.e02;
    const float c01 = m.e02 * m.e12 - m.e01 * m.d2, c02 = m.e01 * m.e12 - m.e02 * m.d1,
                c12 = m.e01 * m.e02 - m.e12 * m.d0;
    m.m2 = m.d0 * m.d1 - m.e01 * m.e01;
    m.m3 = m.d2 * m.m2 + m.e12 * c12 + m.e02 * c02;
    m.err = 2e-6f * (2.0f + pa + kf * pb) + 8e-7f * t * (ei + ef) * inv_hwu;
    const float a0 = fabsf(m.d0), a1 = fabsf(m.d1), a2 = fabsf(m.d2);
    const float b01 = fabsf(m.e01), b02 = fabsf(m.e02), b12 = fabsf(m.e12);
    const float p2 = a0 * a1 + b01 * b01;
    const float p3 = a2 * p2 + b12 * (b12 * a0 + b01 * b02) + b02 * (b01 * b12 + b02 * a1);
    m.err2 = 1.1f * (m.err * (a0 + a1 + 2.0f * (b01 + m.err)) + 1.8e-7f * p2);
    m.err3 = 1.1f * (m.err * (fabsf(c00) + fabsf(c11) + fabsf(m.m2) +
                              2.0f * (fabsf(c01) + fabsf(c02) + fabsf(c12)) +
                              2.0f * m.err * (a0 + a1 + a2 + 2.0f * (b01 + b02 + b12))) +
                     3e-7f * p3);
    return m;
  }

  // The sign of g(Ef), or 0 where FP32 does not decide it (an energy transfer below 0.1 % of
  // Ei + Ef among them).
  MCV_BVK int operator()(double Ef) const {
    const float ef = (float)Ef;
    const float t = (float)sg * (ei - ef) * inv_hwu;
    const BvkMinors m = minors(ef, t);
    if (!(t > 1e-3f * (ei + ef) * inv_hwu && fabsf(m.d0) > m.err && fabsf(m.m2) > m.err2 &&
          fabsf(m.m3) > m.err3))
      return 0;
    const int below = (m.d0 < 0.0f) + ((m.m2 < 0.0f) != (m.d0 < 0.0f)) +
                      ((m.m3 < 0.0f) != (m.m2 < 0.0f));
    const bool lower = below > b;  // omega_b below the energy transfer
    return lower == (sg > 0) ? 1 : -1;
  }
};

}  // namespace mcv
