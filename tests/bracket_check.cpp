// Runs csrc/mcv_bracket.cuh as plain C++ against 50 plain bisection steps: functions on which a
// secant iteration is slow (kinks, jumps, roots of high and of fractional order), and cells with
// three roots, one of them at the first midpoint, where the cheap sign does not decide.  Prints
// one JSON object: the largest distance between the two roots over 2^-50 of the cell plus two
// neighbouring doubles, the cells where they are different roots, the most evaluations of g,
// and their mean number for a smooth function.
#include <cstdio>
#include <cstdlib>
#include <random>

#include "mcv_bracket.cuh"

int mcv::soft64::seed_error = 0;

template <class G>
static double bisect(double ea, double eb, bool pos_a, const G& g) {
  for (int it = 0; it < 50; ++it) {
    const double mid = 0.5 * (ea + eb);
    if ((g(mid) > 0) == pos_a) ea = mid;
    else eb = mid;
  }
  return 0.5 * (ea + eb);
}

int main(int argc, char** argv) {
  const long n = argc > 1 ? std::atol(argv[1]) : 100000;
  std::mt19937_64 r(5);
  auto uni = [&] { return (double)(r() >> 11) * 0x1p-53; };
  double far = 0;
  long other = 0, most = 0, smooth = 0, n_smooth = 0;
  for (long i = 0; i < n; ++i) {
    const double ea = i % 4 == 0 ? 0.0 : uni(), cell = 0.03 * (0.1 + uni()), eb = ea + cell;
    const double root = ea + cell * uni(), big = 1.0 + uni(), up = r() & 1 ? 1.0 : -1.0;
    const double c1 = ea + cell * 0.25 * uni(), c3 = eb - cell * 0.25 * uni();
    const double c2 = 0.5 * (ea + eb) + cell * 1e-7 * (uni() - 0.5);
    const int kind = (int)(r() % 6);
    const bool cheap = r() % 3;  // else a function whose sign is never cheap
    long calls = 0;
    auto f = [&](double x) {
      const double d = x - root, s = d > 0 ? 1.0 : -1.0;
      switch (kind) {
        case 0: return up * (d + 0.3 * d * d / cell + 0.1 * d * d * d / (cell * cell));  // smooth
        case 1: return up * (d > 0 ? d : 1e-4 * d) * big;             // a kink at the root
        case 2: return up * (d > 0 ? 1.0 : -1e-9) * big;              // a jump
        case 3: return up * s * std::pow(std::fabs(d) / cell, 1.0 / 9.0);
        case 4: return up * s * (std::exp(std::fabs(d) / cell * (d > 0 ? 40.0 : 1.0)) - 1.0);
        default: return up * (x - c1) * (x - c2) * (x - c3) / (cell * cell * cell);
      }
    };
    auto g = [&](double x) { ++calls; return f(x); };
    // undecided within 1e-5 of the cell of a root, always beyond it
    auto sign = [&](double x) {
      const double d = kind == 5 ? std::fmin(std::fabs(x - c1), std::fmin(std::fabs(x - c2), std::fabs(x - c3)))
                                 : std::fabs(x - root);
      if (kind != 5 && !cheap) return 0;
      return d < 1e-5 * cell ? 0 : (f(x) > 0 ? 1 : -1);
    };
    const bool pos_a = f(ea) > 0;
    const double want = bisect(ea, eb, pos_a, f);
    const double got = mcv::bracket_root(ea, eb, pos_a, 1e-3, sign, g);
    if (std::fabs(got - want) > 1e-6 * cell)
      ++other;
    else if (std::fabs(f(got)) > 2e-16 * (1e-3 + got))  // else g counts as zero there
      far = std::fmax(far, std::fabs(got - want) / (0x1p-50 * cell + 4.6e-16 * got));
    most = calls > most ? calls : most;
    if (kind == 0 && cheap) smooth += calls, ++n_smooth;
  }
  std::printf("{\"far\": %.6g, \"other\": %ld, \"most\": %ld, \"smooth\": %.3g}\n", far, other, most,
              (double)smooth / n_smooth);
}
