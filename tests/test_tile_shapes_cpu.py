"""Every tile shape that is picked for a lattice has its kernels: over formats, fluid models and sizes,
the launch of the shape picked is refused for the missing CUDA driver only, not for the shape."""
import os
import pathlib
import shutil
import subprocess

import pytest

from conftest import cuda_available
from paper_1908_09235_gb300 import _build

CUDA_ERROR_INVALID_VALUE = 1

SOURCE = r"""
#include <stdio.h>
#include "lbm_internal.h"
using namespace lbm;
int main() {
  alignas(256) static char lattice[2][512];  // (addresses only: nothing is launched without a driver)
  WallIn wi{};
  for (int precision : {LBM_FP64, LBM_FP32_DEV, LBM_FP16_DEV})
    for (int eos : {LBM_EOS_NONE, LBM_EOS_EXP, LBM_EOS_CS})
      for (int nx = 4; nx <= 2100; nx += nx < 64 ? 1 : nx / 17 + 3)
        for (int ny : {4, 5, nx / 3 + 4, nx, 2 * nx + 1}) {
          int tw = 0, th = 0;
          const int shape = pick_step_tiles(precision, eos, nx, ny, &tw, &th);
          if (shape < 0) continue;
          DevParams p{};
          p.nx = nx;
          p.ny = ny;
          p.N = nx * ny;
          p.eos = eos;
          for (const WallIn* w : {(const WallIn*)nullptr, (const WallIn*)&wi})
            printf("%d %d %d %d\n", precision, eos, shape,
                   (int)launch_step_tiles(shape, precision, p, lattice[0], lattice[1], nullptr, nullptr,
                                          nullptr, nullptr, w, nullptr));
        }
}
"""


def test_every_shape_picked_has_its_kernels():
    if cuda_available():
        pytest.skip("needs a machine without a CUDA driver")
    if not shutil.which("g++"):
        pytest.skip("no C++ compiler")
    lib = _build.build()
    cuda_inc = os.path.join(os.path.dirname(os.path.dirname(_build._nvcc())), "include")
    root = os.path.dirname(_build.HERE)
    work = pathlib.Path(_build.LIBDIR) / "shape_check"
    work.mkdir(parents=True, exist_ok=True)
    (work / "shapes.cpp").write_text(SOURCE)
    exe = str(work / "shapes")
    subprocess.check_call(["g++", "-std=c++17", "-I" + cuda_inc, "-I" + _build.CSRC,
                           "-I" + os.path.join(root, "include"), str(work / "shapes.cpp"), lib,
                           "-Wl,-rpath," + _build.LIBDIR, "-o", exe])
    rows = {tuple(map(int, r.split()))
            for r in subprocess.check_output([exe], text=True).splitlines()}
    # shapes of single phase and of either psi: FP64 0, 1 and 4; FP32 2, 4, 5 and 3; FP16 2, 4 and 3
    assert len({r[:3] for r in rows}) == (2 + 3 + 3) + (3 + 4 + 4) + (2 + 3 + 3)
    assert all(r[3] not in (0, CUDA_ERROR_INVALID_VALUE) for r in rows)
