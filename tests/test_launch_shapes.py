"""Launch shapes of the trace kernels (csrc/mcv_shape.h, compiled as plain C++): every neutron has a
lane, no block is larger than the kernel's or the grid than the GPU, a warp of the waves has 32
neutrons (31 where they do not divide evenly, more once the GPU is full), and small runs are
spread over the SMs.  Work items of batches: the tuner's candidates hold the default size of a
batch that its trial can tell apart, and a tuned size follows the batch's neutrons."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1504_02776_gb300", "csrc")


@pytest.mark.parametrize("sms,per_sm,threads,least", [(152, 1, 640, 4), (152, 1, 384, 1), (7, 2, 128, 1)])
def test_shapes_fill_warps_and_sms(tmp_path, sms, per_sm, threads, least):
    exe = str(tmp_path / "launch_shape_check")
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-I" + CSRC, "-x", "c++",
                    os.path.join(HERE, "launch_shape_check.cpp"), "-o", exe], check=True)
    room = sms * per_sm
    full = 32 * room * (threads // 32)
    counts = [1, 31, 32, 33, 1000, 3001, 10000, 32 * room, 32 * room + 1, 30011, 60000, full - 31,
              full, full + 1, 100003, 10 ** 8, 2 ** 40]
    out = subprocess.run([exe, str(sms), str(per_sm), str(threads), str(least)] + [str(n) for n in counts],
                         check=True, capture_output=True, text=True).stdout
    for line in out.splitlines():
        kind, n, grid, block = line[0], *map(int, line[2:].split())
        if kind == "d":  # block: the rows; no idle block, and no longer rows than leave two per SM
            assert 1 <= block <= 4 and 1 <= grid <= 8 * sms, line
            assert grid == 8 * sms or (grid - 1) * block * threads < n <= grid * block * threads, line
            assert block == 1 or n >= 2 * sms * threads * block, line
            continue
        assert 1 <= grid <= room and 32 <= block <= threads and block % 32 == 0, line
        lanes = grid * block
        if kind == "l":
            assert lanes >= n or grid == room, line
            continue
        if kind == "c":
            assert grid == room or (grid >= min(sms, (n + threads - 1) // threads)
                                    and 2 * lanes >= n), line
            continue
        if n >= full:
            assert lanes == full, line
            continue
        warps, batches = lanes // 32, (n + 31) // 32
        assert batches <= warps < batches + block // 32, line  # no block without a batch
        assert grid >= min((batches + least - 1) // least, (room + 1) // 2), line


_CHUNKS = """
#include <cstdio>
#include <cstdlib>
#include "mcv_shape.h"
int main(int, char** v) {
  const long long total = std::atoll(v[1]), trial = std::atoll(v[2]), warps = std::atoll(v[3]);
  const mcv::ChunkList l = mcv::chunk_candidates(total, trial, warps);
  std::printf("%lld %lld %lld %lld", (long long)mcv::default_chunk(total, warps),
              (long long)mcv::scaled_chunk(512, total, total), (long long)mcv::scaled_chunk(512, total, total / 4),
              (long long)mcv::scaled_chunk(512, total, 1ll << 40));
  for (int k = 0; k < l.n; ++k) std::printf(" %lld", (long long)l.chunk[k]);
}
"""


@pytest.mark.parametrize("total,trial", [(260_000, 260_000), (2_600_000, 2_600_000), (75_100, 40_000),
                                         (362_000_000, 20_000_000), (855_000_000, 20_000_000), (1, 1)])
def test_work_items_of_batches(tmp_path, total, trial):
    src, exe, warps = tmp_path / "chunks.cpp", str(tmp_path / "chunks"), 3040
    src.write_text(_CHUNKS)
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-I" + CSRC, str(src), "-o", exe], check=True)
    out = subprocess.run([exe, str(total), str(trial), str(warps)], check=True, capture_output=True,
                         text=True).stdout
    default, same, quarter, huge, *tried = map(int, out.split())
    assert default == max(64, min(8192, total // (16 * warps))) // 32 * 32
    assert same == 512 and quarter == (128 if total > 3 else 64) and huge == 8192
    assert tried[:5] == [512, 1024, 2048, 4096, 8192] and len(set(tried)) == len(tried)
    apart = trial >= 64 * warps
    if apart and default * trial >= 32 * total:
        assert default in tried
    assert all(apart and 64 <= c <= 8192 and c * trial >= 32 * total for c in tried[5:])
