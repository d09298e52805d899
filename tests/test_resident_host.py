"""Host build of the per-kernel cache of launch sizes (csrc/ac_resident.h)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_0710_0736_gb300", "csrc")

HARNESS = r"""
#include "ac_resident.h"
#include <cstdio>
template <int N> void kernel(float *) {}
static int calls = 0;
int query(void (*k)(float *), int threads) {
  ++calls;
  return threads + (k == kernel<2> ? 2 : k == kernel<3> ? 3 : 0);
}
int main() {
  for (int pass = 0; pass < 2; ++pass)
    printf("%d %d %d ", ac::once_per_kernel<kernel<2>, 100>(query), ac::once_per_kernel<kernel<3>, 100>(query),
           ac::once_per_kernel<kernel<2>, 200>(query));
  printf("%d", calls);
}
"""


def test_kernels_of_one_type_keep_their_own_value(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no host compiler")
    (tmp_path / "h.cpp").write_text(HARNESS)
    subprocess.run([gxx, "-O2", "-std=c++17", "-I", CSRC, str(tmp_path / "h.cpp"), "-o", str(tmp_path / "h")], check=True)
    out = subprocess.run([str(tmp_path / "h")], capture_output=True, text=True, check=True).stdout
    assert out.split() == ["102", "103", "202"] * 2 + ["3"]


def test_no_launch_size_is_cached_by_the_type_of_a_kernel():
    """The launchers' only cache of a kernel's launch size is the one above."""
    src = open(os.path.join(CSRC, "ac_launch.cuh")).read()
    assert "static const int" not in src
    assert "once_per_kernel<K, THREADS>(resident_blocks" in src
