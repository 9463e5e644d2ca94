"""The FP32 screen of a DE step (csrc/screen.h), compiled for the host with a base-2 logarithm of the
worst error that the device's is documented to have: the screened point stays within the margin of
the exact one, and with the room that the header derives, in one dimension and more."""
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_04336_gb300", "csrc")

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include "screen.h"
using namespace gwns;
// __log2f: absolute error at most 2^-22 for x in [0.5, 2], at most 2 ulp elsewhere
struct WorstLog2 {
  int sign;
  float operator()(float x) const {
    const double l = std::log2((double)x);
    if (x >= 0.5f && x <= 2.0f) return (float)(l + sign * 0x1p-22);
    const float f = (float)l, to = sign * INFINITY;
    return std::nextafterf(std::nextafterf(f, to), to);
  }
};
// draws 4 x uint64 a line; prints the largest |x32 - x| / margin over c = 2.38 / sqrt(2 D)
int main(int argc, char** argv) {
  const int D = atoi(argv[1]);
  const float c32 = (float)(2.38 / std::sqrt(2.0 * D));
  const long double c = 2.38 / std::sqrt(2.0 * D);
  uint64_t v[4];
  double worst = 0.0;
  while (fread(v, 8, 4, stdin) == 4) {
    long double l = 0.0L;
    for (int i = 0; i < 4; ++i) l += std::log(((long double)(v[i] >> 12) + 0.5L) * 0x1p-52L);
    const long double s = c * (-0.25L * l);
    for (int sign = -1; sign <= 1; sign += 2) {
      const float s32 = screen_scale(v, c32, WorstLog2{sign});
      // a step along the whole cube and along a tenth of it
      const double d[2][3] = {{0.7, 1.0, 0.0}, {0.3, 0.25, 0.35}};
      for (auto& q : d) {
        const long double x = q[0] + s * ((long double)q[1] - q[2]);
        const float x32 = (float)q[0] + s32 * ((float)q[1] - (float)q[2]);
        const double r = (double)(std::fabs((long double)x32 - x) / screen_margin(s32));
        if (r > worst) worst = r;
      }
    }
  }
  printf("%.6f\n", worst);
  return 0;
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    d = tmp_path_factory.mktemp("screen")
    (d / "probe.cpp").write_text(SOURCE)
    exe = d / "probe"
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-I", CSRC, "-o", str(exe), str(d / "probe.cpp")],
                   check=True)
    return str(exe)


@pytest.mark.parametrize("D", [1, 2, 3, 4, 11])
@pytest.mark.parametrize("draws", ["uniform", "near one", "spread"])
def test_screened_point_stays_within_the_margin(probe, D, draws):
    rng = np.random.default_rng([D, len(draws)])
    n = 40000
    top = np.uint64(2 ** 64 - 1)
    v = rng.integers(0, 2 ** 64 - 1, (n, 4), dtype=np.uint64, endpoint=True)
    if draws == "near one":       # small scales: the error that does not shrink with s
        v = top - (v >> rng.integers(1, 45, (n, 4)).astype(np.uint64))
    elif draws == "spread":       # logarithms over their whole range
        v = v >> rng.integers(0, 64, (n, 4)).astype(np.uint64)
    out = subprocess.run([probe, str(D)], input=v.tobytes(), capture_output=True, check=True).stdout
    # derived in the header: 8.4e-7 s + 5.9e-7 against 1e-5 (1 + s)
    assert float(out) <= 8.4e-2, float(out)
