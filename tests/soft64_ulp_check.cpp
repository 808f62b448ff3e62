// Largest errors of csrc/mcv_soft64.cuh's elementary functions in units in the last place of the
// result, against long double, over the whole range of each and next to the arguments where the
// result is small (quarter turns, 1).  Prints one JSON object.
#include <cstdio>
#include <cstdlib>
#include <random>

#include "mcv_soft64.cuh"

int mcv::soft64::seed_error = 0;
using namespace mcv::soft64;

static double ulps(double r, long double t) {
  if (t == 0) return r == 0 ? 0 : 1e300;
  int e;
  std::frexp(std::fabs(t), &e);
  return (double)(std::fabs((long double)r - t) / std::scalbn(1.0L, e - 53));
}

int main(int argc, char** argv) {
  const long n = argc > 1 ? std::atol(argv[1]) : 1000000;
  std::mt19937_64 r(3);
  double e_sc = 0, e_exp = 0, e_log = 0;
  for (long i = 0; i < n; ++i) {
    seed_error = (int)(i % 5) - 2;
    const double u = std::fma((double)(r() >> 11), 0x1p-53, 0x1p-54);
    const double small = std::ldexp(u, -(int)(r() % 54));
    // uniforms over (0, 1], the smallest of them, and next to every quarter turn
    const double us[] = {u, std::fmax(small, 0x1p-54), 0.25 * (1 + r() % 4) - 0.125 * small,
                         0.25 * (1 + r() % 3) + 0.125 * small, 0.25 * (1 + r() % 4)};
    for (double w : us) {
      const double x = 6.283185307179586 * w;
      const Pair p = sincos2pi(w);
      e_sc = std::fmax(e_sc, ulps(p.x, std::sin((long double)x)));
      e_sc = std::fmax(e_sc, ulps(p.y, std::cos((long double)x)));
    }
    for (double x : {-700.0 * u, -50.0 * u, -small, -700.0 * small})
      e_exp = std::fmax(e_exp, ulps(mcv::soft64::exp(x), std::exp((long double)x)));
    const double far = std::ldexp(0.5 + 0.5 * u, (int)(r() % 122) - 60);
    for (double x : {u, far, 1.0 - small, 1.0 + small})
      if (x > 0x1p-60)
        e_log = std::fmax(e_log, ulps(mcv::soft64::log(x), std::log((long double)x)));
  }
  std::printf("{\"sincos\": %.6g, \"exp\": %.6g, \"log\": %.6g}\n", e_sc, e_exp, e_log);
}
