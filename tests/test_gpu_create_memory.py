"""What lbm_create takes for the step kernels that do the wall pass themselves (tables, second set of
moments): a lattice whose steps never use it takes none, and without it a lattice still runs."""
import numpy as np
import pytest

from paper_1908_09235_gb300 import lbm, workloads
from test_gpu_faults import FailingMemory

pytestmark = pytest.mark.gpu


def _lattice(nx, ny, precision, scheme="mod_a", circles=None, memory=None, path=0):
    eos = lbm.make_eos(lbm.EOS_CS, **workloads.CS)
    rl, rv = lbm.lbm_coexistence(eos)
    eos.rho_wall = rv
    circles = circles or [(0.5 * nx, 0.35 * ny, 0.15 * min(nx, ny))]
    lat = lbm.Lattice(nx, ny, 1.0, scheme, circles=circles, eos=eos, precision=precision,
                      memory=memory, kernel_path=path)
    lat.init_droplet(0.5 * nx, 0.6 * ny, 0.25 * min(nx, ny), 4.0, rl, rv)
    return lat


def _run(lat, steps=35):
    lat.step(steps)
    out = lat.fields()
    mass, solid = lat.mass(), lat.flags() & 1 == 1
    assert all(np.array_equal(np.isnan(x), solid) for x in out)
    lat.close()
    return out + (np.float64(mass),)


def _same(a, b):
    return all(np.array_equal(x, y, equal_nan=True) for x, y in zip(a, b))


@pytest.mark.parametrize("precision", [lbm.FP64, lbm.FP32_DEV, lbm.FP16_DEV])
def test_a_lattice_without_memory_for_the_tables_runs_with_the_wall_pass_apart(gpu_lib, precision):
    want = _run(_lattice(96, 64, precision))
    mem = FailingMemory(0)
    _lattice(96, 64, precision, memory=mem).close()
    assert mem.calls == 3  # lattices, links, tables
    mem = FailingMemory(3)
    assert _same(_run(_lattice(96, 64, precision, memory=mem)), want)
    assert mem.calls == 3 and not mem.live


@pytest.mark.parametrize("nx,ny,scheme,circles", [
    (96, 64, "zhao_yong", None),  # its wall pass reads the lattice that the next step overwrites
    # 16 bodies in one 32 x 32 tile: its tables would take 57 KB of shared memory
    (1301, 1000, "mod_a", [(66.3 + 8.5 * i, 66.1 + 8.5 * j, 3.25) for i in range(4) for j in range(4)]),
])
def test_tables_that_no_step_uses_take_no_memory(gpu_lib, nx, ny, scheme, circles):
    def make(path):
        return _lattice(nx, ny, lbm.FP32_DEV, scheme, circles, path=path)

    here, apart = make(0), make(1)
    assert here.info()["device_bytes"] == apart.info()["device_bytes"]
    assert _same(_run(here, 5), _run(apart, 5))


def test_nothing_is_under_way_when_creation_with_tables_returns(gpu_lib):
    # the tables are uploaded from host memory that is given back before lbm_create returns
    import torch
    s = torch.cuda.Stream()
    lat = lbm.Lattice(1500, 1600, 1.0, "mod_a", circles=[(750.0, 560.0, 225.0)],
                      eos=lbm.make_eos(lbm.EOS_NONE), precision=lbm.FP64, stream=s.cuda_stream)
    idle = s.query()
    lat.close()
    assert idle
