"""Host build of the outer node update (paper_0710_0736_gb300/csrc/ac_df64.cuh):
its warp-wide operations are reached equally often by every lane."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_0710_0736_gb300", "csrc")

HARNESS = r"""
#include "ac_df64.cuh"
#include <cstdio>
#include <cstdlib>
using namespace ac;
// in: rows of N doubles u and N doubles delta (cast to float); out: per row
// the calls of any_or, the return value and u
template <int N>
void rows() {
  double in[2 * N];
  while (fread(in, 8, 2 * N, stdin) == 2 * N) {
    double u[N], out[2 + N];
    float d[N];
    for (int i = 0; i < N; ++i) {
      u[i] = in[i];
      d[i] = (float)in[N + i];
    }
    int calls = 0;
    const int path = outer_update_node<N>(u, d, [&](unsigned m) { ++calls; return m; });
    out[0] = calls;
    out[1] = path;
    for (int i = 0; i < N; ++i) out[2 + i] = u[i];
    fwrite(out, 8, 2 + N, stdout);
  }
}
int main(int, char **argv) {
  switch (atoi(argv[1])) {
    case 2: rows<2>(); break;
    case 4: rows<4>(); break;
    default: rows<8>(); break;
  }
}
"""


@pytest.mark.parametrize("N", [2, 4, 8])
def test_every_lane_takes_part_in_every_warp_operation(tmp_path, N):
    """any_or is a warp reduction over the lanes that run together: a lane
    that leaves before the last one while the others wait for it is undefined.
    Nodes of every kind: kept set found in float, near ties (binary64
    iteration), pure, not finite, and no kept component (u = delta = 0, which
    is returned as zeros for the caller to project)."""
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no host compiler")
    (tmp_path / "h.cpp").write_text(HARNESS)
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, str(tmp_path / "h.cpp"), "-o",
                    str(tmp_path / "h")], check=True)
    rng = np.random.default_rng(N)
    u = rng.dirichlet(np.ones(N), 200)
    d = rng.normal(0, 0.1, (200, N)) / N
    d -= d.mean(1, keepdims=True)
    u[:20], d[:20] = 1.0 / N, 0.0
    u[20:40] = np.eye(N)[rng.integers(0, N, 20)]
    d[20:40] = -u[20:40] + np.eye(N)[rng.integers(0, N, 20)]
    u[40:60], d[40:60] = 0.0, 0.0
    u[60:70, 0] = np.nan
    d[70:80, 1] = np.inf
    out = subprocess.run([str(tmp_path / "h"), str(N)], input=np.hstack([u, d]).tobytes(), capture_output=True,
                         check=True).stdout
    out = np.frombuffer(out).reshape(-1, 2 + N)
    assert len(out) == 200
    assert (out[:, 0] == out[0, 0]).all()
    assert (out[40:60, 1] == 2).all() and (out[40:60, 2:] == 0).all()
    assert (out[:40, 1] != 2).all()
