"""Host-side rules of the library, compiled from its headers into a small program
that needs no GPU: which copies a kernel may make."""
import os
import subprocess

import pytest

from paper_1004_1680_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include "mhd_launch.h"
int main() {
  // fields on device a (all but field 5) and b (field 5), current device, the box's device
  const int cases[][4] = {{0, 0, 0, 0}, {1, 1, 1, 0}, {1, 1, 0, 1}, {0, 0, 1, 0}, {0, 1, 0, 0}, {-1, -1, 0, 0}, {0, -1, 0, 0}};
  for (auto& c : cases)
    std::printf("local %d\n", (int)mhd::all_on_device(c[2], c[3], [&](int q) { return q == 5 ? c[1] : c[0]; }));
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
