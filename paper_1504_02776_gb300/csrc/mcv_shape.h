// Launch shapes of the trace kernels (plain C++: a CPU test compiles it as well).
#pragma once

#include <cstdint>

namespace mcv {

struct LaunchShape {
  int grid, threads;
};

// The waves: full blocks, `blocks_per_sm` on every SM, once there are 32 neutrons for each of
// their warps.  Below that a warp for every 32 neutrons, spread over the SMs: the blocks become
// smaller, not fewer, down to `least` warps.  A warp's stages cost the same with 6 lanes as with
// 32, and full blocks on a few SMs wait for one another: FP32 powder, 3e4 neutrons, 38.3 us with
// full blocks (6 to 12 neutrons per warp), 24.4 with this; FP64 can, 1e4, 225 and 149 us.
// least: FP64 1, as a warp has its SM's FP64 pipe to itself; FP32 4, as they fetch the same code
// (phonon kernels, 1e3 neutrons: 33.9 us with one warp per block, 30.3 with two, 28.3 with four).
inline LaunchShape wave_shape(int64_t n, int sms, int blocks_per_sm, int threads, int least) {
  const int64_t room = (int64_t)sms * blocks_per_sm;
  const int64_t need = n < 1 ? 1 : (n + 31) / 32;  // warps
  int64_t warps = (need + room - 1) / room;        // per block
  if (warps < least) warps = least;
  if (warps > threads / 32) warps = threads / 32;
  const int64_t blocks = (need + warps - 1) / warps;
  return LaunchShape{(int)(blocks < room ? blocks : room), (int)(32 * warps)};
}

// One neutron per lane: blocks of `threads`, up to `blocks_per_sm` on every SM.
inline LaunchShape lane_shape(int64_t n, int sms, int blocks_per_sm, int threads) {
  const int64_t room = (int64_t)sms * blocks_per_sm;
  const int64_t need = n < 1 ? 1 : (n + threads - 1) / threads;
  return LaunchShape{(int)(need < room ? need : room), threads};
}

}  // namespace mcv
