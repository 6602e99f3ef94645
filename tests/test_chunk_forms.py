"""The default chunk depth of one float32 D3Q19 lattice by the form of its step
(csrc/chunks.h: default_depth), on lattices whose times at these depths were
measured on 152 SMs, and the event simulation of the estimate against its
closed form for many waves.  CPU only."""
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
  const int nz = std::atoi(v[1]), tz = std::atoi(v[3]);
  const long cols = std::atol(v[2]);
  const nlc::StepForm form{v[4][0] == 'i', v[4][0] == 'p'};
  std::printf("%d %.17g %.17g\n", nlc::default_depth(nz, cols, 152, tz, form),
              nlc::estimate_step_us(nz, cols, tz, 152),
              nlc::round_robin_planes(nz, cols, tz, 304));
  return 0;
}
"""


@pytest.fixture(scope="module")
def chunks(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("forms")
    (d / "drv.cpp").write_text(DRIVER)
    subprocess.check_call([gxx, "-O1", "-std=c++17", "-I",
                           os.path.join(ROOT, "paper_1907_13415_gb300", "csrc"),
                           str(d / "drv.cpp"), "-o", str(d / "drv")])

    def run(nz, cols, tz, form="standard"):
        out = subprocess.check_output([str(d / "drv"), str(nz), str(cols), str(tz), form])
        depth, us, planes = out.decode().split()
        return int(depth), float(us), float(planes)
    return run


#: nx, ny, nz, fallback, depth with the standard and the isotropic stencils
#: and in the persistent form
MEASURED = [(128, 128, 128, 4, 14, 14, 14), (160, 160, 160, 8, 28, 28, 28),
            (70, 180, 50, 4, 12, 12, 4), (32, 32, 32, 4, 1, 1, 1), (100, 100, 100, 4, 6, 6, 6),
            (51, 67, 90, 4, 3, 4, 3), (48, 175, 34, 4, 3, 4, 3), (75, 99, 32, 4, 5, 5, 5),
            (198, 59, 137, 4, 14, 14, 14), (151, 26, 32, 4, 5, 5, 5)]


@pytest.mark.parametrize("nx,ny,nz,fallback,standard,isotropic,persistent", MEASURED)
def test_depths_of_measured_lattices(chunks, nx, ny, nz, fallback, standard, isotropic,
                                     persistent):
    cols = -(-nx // 32) * -(-ny // 8)
    assert chunks(nz, cols, fallback)[0] == standard
    assert chunks(nz, cols, fallback, "isotropic")[0] == isotropic
    assert chunks(nz, cols, fallback, "persistent")[0] == persistent


@pytest.mark.parametrize("nz,tz", [(64, 4), (50, 12), (1, 1)])
def test_simulation_meets_the_closed_form(chunks, nz, tz):
    """On both sides of the 200 blocks per SM where one replaces the other; the
    last wave is a hundredth of the time there."""
    per = -(-nz // tz)
    below, above = 200 * 152 // per, 200 * 152 // per + 1
    us = [chunks(nz, c, tz)[1] / c for c in (below, above)]
    assert us[0] == pytest.approx(us[1], rel=0.02)


@pytest.mark.parametrize("nz,cols,tz,planes", [(50, 69, 12, 17.0), (50, 69, 4, 16.5),
                                               (4, 10, 4, 5.5), (9, 304, 4, 13.5)])
def test_busiest_block_of_the_persistent_kernel(chunks, nz, cols, tz, planes):
    assert chunks(nz, cols, tz)[2] == planes
