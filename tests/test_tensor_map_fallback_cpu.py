"""Where tensor maps cannot be made, large FP16 lattices take the vectorised kernel (which has a form
without tensor copies) with the wall pass apart instead of failing.  Here the driver that makes the maps
is missing: the host side must get as far as a kernel launch, whose error is then the missing driver's."""
import os
import pathlib
import shutil
import subprocess

import pytest

from conftest import cuda_available
from paper_1908_09235_gb300 import _build

CUDA_ERROR_NOT_SUPPORTED = 801

SOURCE = r"""
#include <stdio.h>
#include "lbm_internal.h"
using namespace lbm;
int main() {
  alignas(256) static char lattice[2][512];  // (addresses only: nothing is launched without a driver)
  DevParams p{};
  p.nx = 1600;
  p.ny = 1601;
  p.N = p.nx * p.ny;
  p.eos = LBM_EOS_CS;
  int err = 0;
  const int march = step_march_supported(LBM_FP16_DEV, p.eos, p.nx, p.ny);
  const int front = step_front_supported(LBM_FP16_DEV, p.eos, p.nx, p.ny, lattice[0], lattice[1]);
  const int front32 =
      step_front_supported(LBM_FP32_DEV, LBM_EOS_NONE, p.nx, p.ny, lattice[0], lattice[1]);
  for (int path : {0, 4, 3})
    printf("%d %d %d %d\n", march, front, front32,
           (int)launch_step(LBM_FP16_DEV, p, lattice[0], lattice[1], nullptr, nullptr, nullptr,
                            nullptr, false, nullptr, path, &err));
}
"""


def test_large_fp16_lattices_run_without_tensor_maps():
    if cuda_available():
        pytest.skip("needs a machine without a CUDA driver")
    if not shutil.which("g++"):
        pytest.skip("no C++ compiler")
    lib = _build.build()
    cuda_inc = os.path.join(os.path.dirname(os.path.dirname(_build._nvcc())), "include")
    root = os.path.dirname(_build.HERE)
    work = pathlib.Path(_build.LIBDIR) / "map_check"
    work.mkdir(parents=True, exist_ok=True)
    (work / "maps.cpp").write_text(SOURCE)
    exe = str(work / "maps")
    subprocess.check_call(["g++", "-std=c++17", "-I" + cuda_inc, "-I" + _build.CSRC,
                           "-I" + os.path.join(root, "include"), str(work / "maps.cpp"), lib,
                           "-Wl,-rpath," + _build.LIBDIR, "-o", exe])
    rows = [tuple(map(int, r.split()))
            for r in subprocess.check_output([exe], text=True).splitlines()]
    assert len(rows) == 3
    for march, front, front32, error in rows:
        assert march == 1 and front == 0 and front32 == 1
        assert error not in (0, CUDA_ERROR_NOT_SUPPORTED)
    assert len({r[3] for r in rows}) == 1  # path 3 is the vectorised kernel without tensor copies
