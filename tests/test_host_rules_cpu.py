"""Host-side rules of the library, compiled from its headers into a small program
that needs no GPU: which copies a kernel may make, how many values a thread
adds into one window of FP32 words, and what a tile sweep computes beyond its cells."""
import os
import subprocess

import pytest

from paper_1004_1680_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include "fp32_sums.cuh"
#include "mhd_launch.h"
int main() {
  // fields on device a (all but field 5) and b (field 5), current device, the box's device
  const int cases[][4] = {{0, 0, 0, 0}, {1, 1, 1, 0}, {1, 1, 0, 1}, {0, 0, 1, 0}, {0, 1, 0, 0}, {-1, -1, 0, 0}, {0, -1, 0, 0}};
  for (auto& c : cases)
    std::printf("local %d\n", (int)mhd::all_on_device(c[2], c[3], [&](int q) { return q == 5 ? c[1] : c[0]; }));
  for (long long n : {0LL, 1LL, 255LL, 256LL, 257LL, 155648LL, 155649LL, 262144LL, 39845888LL, 39845889LL, 39911425LL,
                      134217728LL, 2147483647LL})
    std::printf("sums %lld %d %d %d\n", n, mhd::sum_blocks(n), mhd::kSumThreads, mhd::kWin);
  for (int n : {1, 2, 3, 4, 5, 8, 9, 32, 40, 41, 96, 98, 130})
    std::printf("pad %d %.6f %.6f %.6f\n", n, mhd::fluid_tile_padding(2, n, n > 64 ? 256 : 128),
                mhd::fluid_tile_padding(0, (n + 3) / 4 * 4, 128), mhd::mag_tile_padding(n));
  return 0;
}
"""


@pytest.fixture(scope="module")
def printed(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    src, exe = str(d / "rules.cu"), str(d / "rules")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.check_call([build.nvcc(), *build.ARCH, "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, src, "-o", exe])
    return subprocess.run([exe], check=True, capture_output=True, text=True, env=dict(os.environ)).stdout.splitlines()


def test_fields_are_copied_by_a_kernel_only_on_the_boxs_own_device(printed):
    """One device throughout; not with the box elsewhere (fields and current device
    agreeing does not help: the kernel would read another device's memory), a
    field elsewhere, or host memory."""
    assert [ln for ln in printed if ln.startswith("local")] == [f"local {v}" for v in (1, 0, 0, 0, 0, 0, 0)]


def test_no_thread_adds_more_values_than_a_window_holds(printed):
    """The error bound of the FP32 words is for windows of kWin values."""
    rows = [tuple(int(v) for v in ln.split()[1:]) for ln in printed if ln.startswith("sums")]
    assert len(rows) == 13
    for n, blocks, threads, win in rows:
        assert blocks >= 1 and -(-n // (blocks * threads)) <= win
    grid = {r[0]: r[1] for r in rows}  # one grid from 155,648 values to 39.8 M
    assert grid[262144] == grid[39845888] == 608 and grid[2147483647] == 32768


def test_tile_estimates_count_what_a_block_computes(printed):
    """Whole pencils of a multiple of 4 cells have no padding; others a halo thread
    of 4 cells at each end of every segment."""
    rows = {int(ln.split()[1]): [float(v) for v in ln.split()[2:]] for ln in printed if ln.startswith("pad")}
    z = {n: 4 * (-(-n // 4) + 2) / n for n in (1, 2, 3, 5, 9, 41)}
    z.update({4: 1, 8: 1, 32: 1, 40: 1, 96: 1, 98: 4 * 27 / 98, 130: 2 * 4 * 19 / 130})
    mag = {n: -(-n // 4) * 4 / n if n <= 40 else 1 for n in rows}
    for n, (fluid_z, fluid_x, m) in rows.items():
        assert fluid_z == pytest.approx(z[n], abs=1e-6) and fluid_x == 1.0 and m == pytest.approx(mag[n], abs=1e-6)
