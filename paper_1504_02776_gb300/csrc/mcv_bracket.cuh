// The root of g in one grid cell of the FP64 single-crystal kernel, from FP32 signs and few FP64
// evaluations.  Also compiles as plain C++ (a CPU test runs it on hard functions).
#pragma once

#include "mcv_soft64.cuh"

namespace mcv {

// The root that 50 bisection steps of the cell [ea, eb] give, where g has opposite signs at the
// ends (pos_a: g > 0 at ea).  sign(x): the sign of g where it is cheap and certain, else 0.
// 2e-16 (ei + x) is the rounding of g(x) = ei - x - ...
//
// 1. Bisection on its own midpoints by the cheap sign, and by g where that is undecided and the
//    bracket wider than 2^-12 of the cell: a cell with several roots so gives the root that plain
//    bisection gives, unless they are within 2^-12 of the cell of each other.
// 2. On that bracket the secant iteration (regula falsi, Illinois variant) until g is its
//    rounding.  Every fourth step is a halving, and from the 24th step on all are: after 60 the
//    bracket is below 2^-52 of the cell whatever the function.  A smooth one takes 4 to 6.
// 3. Where that rounding over the slope is more than 1e-13 of the root (a root near zero, a
//    tangency) bisection and secant differ by it: the remaining steps of the bisection, by g
//    where the midpoint is as near to the secant's root.
//
// The evaluations of g are few and apart from the cheap loops, so that the lanes of a warp make
// them together.
template <class Sign, class G>
MCV_S64 double bracket_root(double ea, double eb, bool pos_a, double ei, const Sign& sign, const G& g) {
  const double wide = 0x1p-12 * (eb - ea), least = 0x1p-52 * (eb - ea);
  double mid = 0.0;
  int it = 0;
  for (;;) {
    int s = 0;
    while (it < 50) {
      mid = 0.5 * (ea + eb);
      s = sign(mid);
      if (s == 0) break;
      if ((s > 0) == pos_a)
        ea = mid;
      else
        eb = mid;
      ++it;
    }
    if (it == 50 || !(eb - ea > wide)) break;
    if (soft64::positive(g(mid)) == pos_a)
      ea = mid;
    else
      eb = mid;
    ++it;
  }
  double xa = ea, xb = eb, ga = g(xa), gb = g(xb), x = 0.5 * (xa + xb), slope = 0.0;
  int side = 0;
  for (int k = 0; k < 60; ++k) {
    const double w = xb - xa;
    mid = 0.5 * (xa + xb);
    x = mid;
    if (!(w > 2.3e-16 * xb && w > least)) break;  // neighbouring doubles
    if ((k & 3) != 3 && k < 24) {
      const double c = xa + w * soft64::div(ga, ga - gb);
      if (c > xa && c < xb) mid = c;
    }
    if (!(mid > xa && mid < xb)) break;
    x = mid;
    const double gm = g(mid);
    const bool left = soft64::positive(gm) == pos_a;
    slope = left ? soft64::div(gm - gb, mid - xb) : soft64::div(gm - ga, mid - xa);
    if (!(::fabs(gm) > 2e-16 * (ei + mid))) break;
    if (left) {
      xa = mid;
      ga = gm;
      if (side == 1) gb *= 0.5;
      side = 1;
    } else {
      xb = mid;
      gb = gm;
      if (side == -1) ga *= 0.5;
      side = -1;
    }
  }
  const double blur = 2e-16 * (ei + x);
  if (!(blur > 1e-13 * x * ::fabs(slope))) return x;
  const double near = 4.0 * soft64::div(blur, ::fabs(slope));
  for (; it < 50; ++it) {
    mid = 0.5 * (ea + eb);
    bool left = mid < x;
    if (!(::fabs(mid - x) > near)) left = soft64::positive(g(mid)) == pos_a;
    if (left)
      ea = mid;
    else
      eb = mid;
  }
  return 0.5 * (ea + eb);
}

}  // namespace mcv
