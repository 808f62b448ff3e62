// Checks csrc/mcv_bvk_sign.cuh as plain C++ against the same matrix in double: the entries of
// D - lambda* against the bound `err`, the minors against theirs, and every sign that is not left
// undecided.  Cells, stiffnesses, masses, energies, directions (near forward
// among them) and modes are drawn; sine and cosine are off by up to two units in the last place.
// Prints one JSON object: the largest error over its bound, the wrong signs, and the share of
// undecided ones.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>

#include "mcv_bvk_sign.cuh"

static std::mt19937_64 g_r(11);
static float nudge(float x) {
  int32_t b;
  std::memcpy(&b, &x, 4);
  b += (int)(g_r() % 5) - 2;
  std::memcpy(&x, &b, 4);
  return x;
}
void mcv::bvk_sincos(float x, float* s, float* c) {
  *s = nudge((float)std::sin((double)x));
  *c = nudge((float)std::cos((double)x));
}

static double uni() { return (double)(g_r() >> 11) * 0x1p-53; }
static double log_uni(double lo, double hi) { return lo * std::pow(hi / lo, uni()); }

int main(int argc, char** argv) {
  const long n = argc > 1 ? std::atol(argv[1]) : 1000000;
  double r_entry = 0, r_m2 = 0, r_m3 = 0;
  long wrong = 0, open = 0;
  for (long i = 0; i < n; ++i) {
    const double a = log_uni(2.0, 60.0), phi = log_uni(1.0, 300.0), mass = log_uni(4.0, 240.0);
    const double Ei = log_uni(3.0, 2000.0);
    // hbar sqrt(phi / M) in meV
    const double hwu = mcv::kHbar * std::sqrt(phi / (mass * 1.66053906660e-27)) / (mcv::kElemCharge * 1e-3);
    double di[3], df[3], norm = 0;
    for (double& d : di) d = 2 * uni() - 1, norm += d * d;
    for (double& d : di) d /= std::sqrt(norm);
    norm = 0;
    // every other event within a small angle of forward
    const double turn = i & 1 ? log_uni(1e-6, 1.0) : 2.0;
    for (int k = 0; k < 3; ++k) {
      df[k] = di[k] * (i & 1 ? 1.0 : 0.0) + turn * (uni() - 0.5);
      norm += df[k] * df[k];
    }
    for (double& d : df) d /= std::sqrt(norm);
    mcv::BvkSign q;
    q.sg = g_r() & 1 ? 1 : -1;
    q.b = (int)(g_r() % 3);
    const double top = hwu * std::sqrt(24.0);
    double Ef = q.sg > 0 ? Ei * uni() : Ei + top * uni();
    if (i % 3 == 0) Ef = Ei - q.sg * Ei * log_uni(1e-3, 1.0);  // small energy transfers
    if (!(Ef > 0)) continue;
    const double ki = mcv::kKPerV * std::sqrt(Ei / mcv::kMeVPerV2);
    const double kf = mcv::kKPerV * std::sqrt(Ef / mcv::kMeVPerV2);
    const double ah = 0.5 * a;
    q.set_phases((float)(ah * (di[0] * ki)), (float)(ah * (di[1] * ki)), (float)(ah * (di[2] * ki)),
                 (float)(ah * df[0]), (float)(ah * df[1]), (float)(ah * df[2]));
    q.ei = (float)Ei;
    q.inv_hwu = (float)(1.0 / hwu);
    // the same in double, from the definitions
    double x[3], s[3], c[3];
    for (int k = 0; k < 3; ++k) {
      x[k] = ah * (di[k] * ki - df[k] * kf);
      s[k] = std::sin(x[k]);
      c[k] = std::cos(x[k]);
    }
    const double t = q.sg * (Ei - Ef) / hwu, lam = t * t;
    const double d0 = 4 - 2 * c[0] * (c[1] + c[2]) - lam, d1 = 4 - 2 * c[1] * (c[0] + c[2]) - lam,
                 d2 = 4 - 2 * c[2] * (c[0] + c[1]) - lam;
    const double e01 = 2 * s[0] * s[1], e02 = 2 * s[0] * s[2], e12 = 2 * s[1] * s[2];
    const double m2 = d0 * d1 - e01 * e01;
    const double m3 = d2 * m2 - e12 * (d0 * e12 - e01 * e02) + e02 * (e01 * e12 - d1 * e02);
    const float ef = (float)Ef, tf = (float)q.sg * (q.ei - ef) * q.inv_hwu;
    const int got = q(Ef);
    if (!(tf > 1e-3f * (q.ei + ef) * q.inv_hwu)) {
      open += got == 0;
      wrong += got != 0;
      continue;
    }
    const mcv::BvkMinors m = q.minors(ef, tf);
    const double pairs[6][2] = {{m.d0, d0}, {m.d1, d1}, {m.d2, d2}, {m.e01, e01}, {m.e02, e02}, {m.e12, e12}};
    for (const auto& p : pairs) r_entry = std::fmax(r_entry, std::fabs(p[0] - p[1]) / m.err);
    r_m2 = std::fmax(r_m2, std::fabs(m.m2 - m2) / m.err2);
    r_m3 = std::fmax(r_m3, std::fabs(m.m3 - m3) / m.err3);
    if (got == 0) {
      ++open;
      continue;
    }
    const int below = (d0 < 0) + ((m2 < 0) != (d0 < 0)) + ((m3 < 0) != (m2 < 0));
    wrong += got != (((below > q.b) == (q.sg > 0)) ? 1 : -1);
  }
  std::printf("{\"entry\": %.6g, \"m2\": %.6g, \"m3\": %.6g, \"wrong\": %ld, \"open\": %.6g}\n", r_entry,
              r_m2, r_m3, wrong, (double)open / n);
}
