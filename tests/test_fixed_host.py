"""Host build of the 64-bit fixed-point helpers of the FP64 form's nodal
problem (paper_0710_0736_gb300/csrc/ac_df64.cuh): conversions and the simplex
projection against exact rationals, and its error against that of the
binary64 iteration."""
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_0710_0736_gb300", "csrc")

HARNESS = r"""
#include "ac_df64.cuh"
#include <cstdio>
#include <cstdlib>
#include <vector>
using namespace ac;
// in: rows of N doubles; out: per row N doubles x and one double, 1 if a value was out of range
template <int N>
void rows(const std::vector<double> &in) {
  for (size_t r = 0; r + N <= in.size(); r += N) {
    int64_t z[N], theta;
    unsigned keep;
    bool bad = false;
    for (int i = 0; i < N; ++i) z[i] = f64_to_fix<57, 2>(in[r + i], bad);
    fixed_simplex<N, 57>(z, keep, theta);
    double x[N + 1];
    for (int i = 0; i < N; ++i) x[i] = ((keep >> i) & 1u) ? fix_to_f64<57>(z[i] - theta) : 0.0;
    x[N] = bad;
    fwrite(x, 8, N + 1, stdout);
  }
}
int main(int argc, char **argv) {
  std::vector<double> in;
  double d;
  while (fread(&d, 8, 1, stdin) == 1) in.push_back(d);
  switch (atoi(argv[1])) {
    case 0:  // phase values: to 2^-60 and back, and whether out of range
      for (double v : in) {
        bool bad = false;
        const int64_t f = f64_to_fix<60, 1>(v, bad);
        double o[2] = {(f < 0 ? -1.0 : 1.0) * fix_to_f64<60>(f < 0 ? -f : f), (double)bad};
        fwrite(o, 8, 2, stdout);
      }
      break;
    case 2: rows<2>(in); break;
    case 3: rows<3>(in); break;
    case 4: rows<4>(in); break;
    case 5: rows<5>(in); break;
    case 6: rows<6>(in); break;
    case 7: rows<7>(in); break;
    default: rows<8>(in); break;
  }
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("fixed")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, str(d / "h.cpp"), "-o", str(d / "h")],
                   check=True)

    def run(mode, x):
        out = subprocess.run([str(d / "h"), str(mode)], input=np.ascontiguousarray(x, np.float64).tobytes(),
                             capture_output=True, check=True).stdout
        return np.frombuffer(out, np.float64)

    return run


def test_phase_values_round_trip(harness):
    """Within half a unit of 2^-60 (rounded to nearest), exact from 2^-7 up;
    out of range at 2 and above, infinities and NaN."""
    rng = np.random.default_rng(0)
    v = np.concatenate([rng.uniform(-1, 1, 2000), np.ldexp(rng.uniform(0.5, 1, 2000), -rng.integers(0, 70, 2000)),
                        [0.0, -0.0, 1.0, 5e-324, 2.0 ** -61, 2.0 ** -60, np.nextafter(2, 0)]])
    o = harness(0, v).reshape(-1, 2)
    assert not o[:, 1].any()
    for a, b in zip(v, o[:, 0]):
        assert abs(Fraction(a) - Fraction(b)) <= Fraction(1, 2 ** 61)
    big = np.abs(v) >= 2.0 ** -7
    assert np.array_equal(v[big], o[big, 0])
    assert harness(0, [2.0, -2.0, 1e300, np.inf, -np.inf, np.nan]).reshape(-1, 2)[:, 1].all()


def _exact(z):
    z = [Fraction(v) for v in z]
    keep = list(range(len(z)))
    while True:
        t = (sum(z[i] for i in keep) - 1) / len(keep)
        left = [i for i in keep if z[i] > t]
        if left == keep:
            return [z[i] - t if i in keep else Fraction(0) for i in range(len(z))]
        keep = left


def _binary64(z):
    n, keep = len(z), list(range(len(z)))
    for _ in range(n):
        t = (sum(z[i] for i in keep) - 1.0) * (1.0 / len(keep))
        left = [i for i in keep if z[i] - t > 0]
        if left == keep or not left:
            break
        keep = left
    return [z[i] - t if i in keep else 0.0 for i in range(n)]


@pytest.mark.parametrize("N", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("scale", [0.3, 1.0, 3.9])
def test_projection_is_closer_than_binary64(harness, N, scale):
    """Against the exact projection: z rounded to 2^-58, theta a mean of such
    values rounded to 2^-58, the result to 2^-54 of at most 1, so at most
    (1/2 + 1/2) 2^-57 + 2^-54 < 9e-17; sums to 1 within N such errors; and
    no further off than the binary64 iteration, at worst and on average."""
    rng = np.random.default_rng(N)
    z = rng.uniform(-scale, scale, (400, N))
    z[:40] = np.trunc(z[:40] * 4) / 4  # ties
    z[40:60] = 1.0 / N
    z[60:80] = 0.0
    o = harness(N, z).reshape(-1, N + 1)
    assert not o[:, N].any()
    off, off64 = [], []
    for row, x in zip(z, o[:, :N]):
        e = _exact(row)
        off.append(max(abs(Fraction(a) - b) for a, b in zip(x, e)))
        off64.append(max(abs(Fraction(a) - b) for a, b in zip(_binary64(list(row)), e)))
    assert float(max(off)) <= 9e-17
    assert np.abs(o[:, :N].sum(1) - 1).max() <= N * 9e-17 + 4e-16
    assert max(off) <= max(off64) and sum(off) <= sum(off64)
    assert harness(N, np.where(np.arange(N) == 0, 4.0, 0.0)[None]).reshape(-1, N + 1)[0, N] == 1.0
