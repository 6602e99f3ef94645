"""The default chunk depth of one float32 D3Q19 lattice (csrc/chunks.h:
estimated_depth): a depth the column can hold, the fallback unless the
estimate is a tenth better, and the estimate's order on the cases it rests
on (a block that has an SM to itself is the cheaper the fewer planes it has).
CPU only."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
DRIVER = r"""
#include <cstdio>
#include <cstdlib>
#include "chunks.h"
int main(int, char** v) {
  const int nz = std::atoi(v[1]), sms = std::atoi(v[3]), fb = std::atoi(v[4]);
  const long cols = std::atol(v[2]);
  const int c = nlc::estimated_depth(nz, cols, sms, fb);
  std::printf("%d %.17g %.17g\n", c, nlc::estimate_step_us(nz, cols, c, sms),
              nlc::estimate_step_us(nz, cols, fb, sms));
  return 0;
}
"""


@pytest.fixture(scope="module")
def estimate(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("estimate")
    (d / "drv.cpp").write_text(DRIVER)
    subprocess.check_call([gxx, "-O1", "-std=c++17", "-I",
                           os.path.join(ROOT, "paper_1907_13415_gb300", "csrc"),
                           str(d / "drv.cpp"), "-o", str(d / "drv")])

    def run(*args):
        out = subprocess.check_output([str(d / "drv")] + [str(a) for a in args]).decode().split()
        return int(out[0]), float(out[1]), float(out[2])
    return run


@pytest.mark.parametrize("nz,cols,fallback", [(1, 1, 1), (1, 5000, 1), (2, 3, 2), (7, 152, 4),
                                              (32, 4, 4), (64, 16, 4), (117, 85, 8),
                                              (256, 256, 32), (513, 1, 4), (33, 40000, 32)])
def test_depth_fits_and_beats_the_fallback(estimate, nz, cols, fallback):
    depth, t, t0 = estimate(nz, cols, 152, fallback)
    assert 1 <= depth <= nz or depth == fallback
    assert depth == fallback or t < 0.9 * t0


def test_small_lattices_spread_over_the_sms(estimate):
    assert estimate(32, 4, 152, 4)[0] == 1      # 128 blocks on 152 SMs
    assert estimate(64, 16, 152, 4)[0] == 4     # 256 blocks, two per SM
