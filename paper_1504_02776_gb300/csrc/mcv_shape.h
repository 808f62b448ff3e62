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

// One item per lane: blocks of `threads`, up to `blocks_per_sm` on every SM.
inline LaunchShape lane_shape(int64_t n, int sms, int blocks_per_sm, int threads) {
  const int64_t room = (int64_t)sms * blocks_per_sm;
  const int64_t need = n < 1 ? 1 : (n + threads - 1) / threads;
  return LaunchShape{(int)(need < room ? need : room), threads};
}

// One neutron per lane with lanes refilled as neutrons end (run_chain): two neutrons for every
// lane once each SM has a block, as lanes without a next one idle.  Stored beam into a detector,
// 1e5 neutrons, one / two / four per lane: FP32 powder 53.5 / 40.5 / 48.0 us, FP32 cylinder
// 42.9 / 28.9 / 24.7, FP32 crystal 631 / 537 / 740, FP64 powder 350 / 311 / 379.  Without a
// detector the chain is short and one per lane is the faster (FP64 can, 3e4: 136 and 155 us).
inline LaunchShape chain_shape(int64_t n, int sms, int blocks_per_sm, int threads) {
  const LaunchShape one = lane_shape(n, sms, blocks_per_sm, threads);
  const LaunchShape two = lane_shape((n + 1) / 2, sms, blocks_per_sm, threads);
  return one.grid <= sms ? one : (two.grid < sms ? LaunchShape{sms, threads} : two);
}

// Stored packets (detect_kernel): up to 8 blocks per SM, each of which reads `rows` x `threads`
// slots at a time: max_rows of them once that leaves every SM two blocks, fewer where the list is
// shorter.
struct DetectShape {
  int grid, rows;
};

inline DetectShape detect_shape(int64_t n, int sms, int threads, int max_rows) {
  const int64_t room = (int64_t)sms * 8;
  int64_t rows = n / ((int64_t)sms * 2 * threads);
  rows = rows < 1 ? 1 : (rows < max_rows ? rows : max_rows);
  const int64_t need = n < 1 ? 1 : (n + rows * threads - 1) / (rows * threads);
  return DetectShape{(int)(need < room ? need : room), (int)rows};
}

// Work items of a batch, in neutrons: about 16 items per resident warp, a multiple of 32 in
// [kMinChunk, kMaxChunk] (items of one simulation follow each other in a warp without a drain,
// so small items cost little more than their queue counter update; with items of at least 256,
// 13 crystal orientations of 2e5 neutrons left the warps 3 items each: 4.34 ms, with 64: 4.13).
constexpr int64_t kMinChunk = 64, kMaxChunk = 8192;

inline int64_t bounded_chunk(int64_t c) {
  return (c < kMinChunk ? kMinChunk : (c > kMaxChunk ? kMaxChunk : c)) / 32 * 32;
}

inline int64_t default_chunk(int64_t total, int64_t warps) {
  return bounded_chunk(total / ((warps < 1 ? 1 : warps) * 16));
}

// The sizes the tuner tries on a trial of `trial` of the batch's `total` neutrons: 512 to 8192, and
// where the trial gives every warp at least two batches of 32 (a smaller one does not show how
// the load is balanced) the default and 64 to 256, as far as they stay above 32 neutrons when
// scaled to the trial.  With 512 and more alone, tuning 13 orientations of 2e4 neutrons made them
// slower, 0.91 -> 2.46 ms, and of 2e5, 3.87 -> 4.46.
struct ChunkList {
  int64_t chunk[9];
  int n;
};

inline ChunkList chunk_candidates(int64_t total, int64_t trial, int64_t warps) {
  ChunkList l{{512, 1024, 2048, 4096, 8192}, 5};
  if (trial < 64 * warps) return l;
  const int64_t small[] = {default_chunk(total, warps), 64, 128, 256};
  for (int64_t c : small) {
    bool more = (double)c * ((double)trial / (double)total) >= 32.0;
    for (int k = 0; k < l.n; ++k) more = more && l.chunk[k] != c;
    if (more) l.chunk[l.n++] = c;
  }
  return l;
}

// The size for a batch of `total` neutrons where `chunk` was the best for one of `of`: as many
// items per warp.
inline int64_t scaled_chunk(int64_t chunk, int64_t of, int64_t total) {
  if (of == total) return chunk;
  return bounded_chunk((int64_t)((double)chunk * ((double)total / (double)of)));
}

}  // namespace mcv
