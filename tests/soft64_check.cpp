// Checks csrc/mcv_soft64.cuh as plain C++: division and square root bit for bit against the
// FPU, the elementary functions against long double references (units in the last place; sin and
// cos also as absolute errors beyond half a unit).  Prints one JSON object.
#include <cstdio>
#include <cstdlib>
#include <random>

#include "mcv_soft64.cuh"

int mcv::soft64::seed_error = 0;
using namespace mcv::soft64;

static double ulps(double r, long double t) {
  const double a = std::fabs((double)t);
  if (a == 0) return r == 0 ? 0 : 1e9;
  int e;
  std::frexp(a, &e);
  return (double)(std::fabs((long double)r - t) / std::scalbn(1.0L, e - 53));
}

static bool same(double a, double b) { return bits(a) == bits(b) || (a != a && b != b); }

int main(int argc, char** argv) {
  const long n = argc > 1 ? std::atol(argv[1]) : 1000000;
  std::mt19937_64 r(1);
  long div_bad = 0, sqrt_bad = 0;
  for (int p = -2; p <= 2; ++p) {
    seed_error = p;
    for (long i = 0; i < n; ++i) {
      uint64_t A = r(), B = r();
      const int mode = i % 5;
      if (mode == 1) {  // quotients near 1
        A = (A & 0x800fffffffffffffull) | 0x3ff0000000000000ull;
        B = (B & 0x800fffffffffffffull) | 0x3ff0000000000000ull;
      } else if (mode == 2) {  // significands next to 1 and to 2
        A = 0x3ff0000000000000ull | (r() % 16) | ((r() % 3) << 50);
        B = 0x3ff0000000000000ull | (r() % 16) | (0xfffffffffff00ull * (r() % 2));
      } else if (mode == 3) {  // quotients next to a double or to the middle of two
        B = (B & 0xfffffffffffffull) | 0x3ff0000000000000ull;
        A = bits(from_bits(B) * from_bits(0x3ff0000000000000ull | (r() & 0xfffffffffffffull)));
      }
      const double a = from_bits(A), b = from_bits(B);
      div_bad += !same(div(a, b), a / b);
      double x = std::fabs(a);
      if (mode == 3) {
        const double t = from_bits(0x3ff0000000000000ull | (r() & 0xfffffffffffffull));
        x = t * t * ((i & 8) ? 2 : 1);
      }
      if (i % 1000 == 7) x = -x;
      sqrt_bad += !same(mcv::soft64::sqrt(x), std::sqrt(x));
    }
  }
  const double special[] = {0.0, -0.0, 1.0, -1.0, INFINITY, -INFINITY, NAN, 5e-324, 2.2250738585072014e-308,
                            1.7976931348623157e308, -5e-324};
  for (double a : special) {
    for (double b : special) div_bad += !same(div(a, b), a / b);
    sqrt_bad += !same(mcv::soft64::sqrt(a), std::sqrt(a));
  }
  seed_error = 1;
  double e_log = 0, e_exp = 0, e_tan = 0, e_sc = 0;
  for (long i = 0; i < n; ++i) {
    double u = std::fma((double)(r() >> 11), 0x1p-53, 0x1p-54);  // the uniforms of the method
    if (i % 7 == 0) u = std::ldexp(u, -(int)(r() % 50));
    if (i % 11 == 0) u = 1.0 - std::ldexp((double)(r() >> 11), -53 - (int)(r() % 52));
    if (!(u > 0 && u < 1)) continue;
    e_log = std::fmax(e_log, ulps(mcv::soft64::log(u), std::log((long double)u)));
    const double big = 1.0 / u > 1e18 ? 2.0 : 1.0 / u;
    e_log = std::fmax(e_log, ulps(mcv::soft64::log(big), std::log((long double)big)));
    double y = -std::ldexp(u, (int)(r() % 20) - 10);
    if (y < -700) y = -u;
    e_exp = std::fmax(e_exp, ulps(mcv::soft64::exp(y), std::exp((long double)y)));
    const double t = u * 0.0624 * ((i & 1) ? 1 : -1);
    e_tan = std::fmax(e_tan, ulps(mcv::soft64::tan(t), std::tan((long double)t)));
    const Pair sc = sincos2pi(u);
    const double x = 2.0 * 3.14159265358979323846 * u;
    const double v[2] = {sc.x, sc.y};
    const long double w[2] = {std::sin((long double)x), std::cos((long double)x)};
    for (int k = 0; k < 2; ++k) {
      const double half = v[k] == 0 ? 0 : std::ldexp(0.5, std::ilogb(std::fabs(v[k])) - 52);
      e_sc = std::fmax(e_sc, (double)std::fabs((long double)v[k] - w[k]) - half);
    }
  }
  // the integer tests and conversions
  long conv_bad = 0;
  for (long i = 0; i < n; ++i) {
    double a = from_bits(r()), b = from_bits(r());
    if (i % 3 == 1) a = std::ldexp((double)(r() >> 11), -50 + (int)(r() % 30)) * ((r() & 1) ? 1 : -1);
    if (i % 3 == 2) a = special[r() % 11];
    if (a != a) a = NAN;
    conv_bad += positive(a) != (a > 0);
    conv_bad += is_zero(a) != (a == 0);
    const double c = std::fabs(a), e = std::fabs(b);
    if (c == c && e == e) conv_bad += lt_nonneg(c, e) != (c < e);
    const int m = 1 + (int)(r() % 2000);
    const double f = std::floor(a);
    conv_bad += index_below(a, m) != ((f >= 0 && f < m) ? (int)f : -1);
    conv_bad += index_clamped(a, m) != (!(f > 0) ? 0 : f >= m ? m - 1 : (int)f);
    uint32_t h = (uint32_t)r(), l = (uint32_t)r();
    if (i % 5 == 0) h >>= r() % 32;
    if (i % 50 == 0) h = 0;
    if (i % 7 == 0) h = ~0u - (uint32_t)(r() % 3);
    const uint64_t k = ((uint64_t)h << 21) | (l >> 11);
    conv_bad += uniform53(h, l) != std::fma((double)k, 0x1p-53, 0x1p-54);
  }
  std::printf("{\"conv_bad\": %ld, \"div_bad\": %ld, \"sqrt_bad\": %ld, \"log\": %.6g, \"exp\": %.6g, \"tan\": %.6g, "
              "\"sincos\": %.6g, \"exp0\": %.17g, \"log1\": %.17g}\n", conv_bad, div_bad, sqrt_bad, e_log, e_exp,
              e_tan, e_sc, mcv::soft64::exp(0.0), mcv::soft64::log(1.0));
}
