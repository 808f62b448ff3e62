// Prints "n grid threads" of csrc/mcv_shape.h for the counts given on the command line after SMs,
// blocks per SM, threads and least warps, a line each for the waves ("w"), for one item per lane
// ("l") and for refilled lanes ("c"), and "n grid rows" for stored packets ("d").
#include <cstdio>
#include <cstdlib>

#include "mcv_shape.h"

int main(int argc, char** argv) {
  const int sms = std::atoi(argv[1]), per_sm = std::atoi(argv[2]), threads = std::atoi(argv[3]);
  const int least = std::atoi(argv[4]);
  for (int i = 5; i < argc; ++i) {
    const long long n = std::atoll(argv[i]);
    const mcv::LaunchShape w = mcv::wave_shape(n, sms, per_sm, threads, least);
    const mcv::LaunchShape l = mcv::lane_shape(n, sms, per_sm, threads);
    const mcv::LaunchShape c = mcv::chain_shape(n, sms, per_sm, threads);
    std::printf("w %lld %d %d\nl %lld %d %d\nc %lld %d %d\n", n, w.grid, w.threads, n, l.grid,
                l.threads, n, c.grid, c.threads);
    const mcv::DetectShape d = mcv::detect_shape(n, sms, threads, 4);
    std::printf("d %lld %d %d\n", n, d.grid, d.rows);
  }
}
