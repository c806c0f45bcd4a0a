"""A channel's blob restored into a channel that already steps with another inflow velocity: the steps
inside captured graphs take the restored velocity as the remainder steps do."""
import numpy as np
import pytest

from paper_1908_09235_gb300 import lbm

pytestmark = pytest.mark.gpu


# the channel ends in the tiles (96 x 48), in front of them (700 x 610) and as a launch of their own
@pytest.mark.parametrize("precision", [lbm.FP64, lbm.FP32_DEV])
@pytest.mark.parametrize("nx,ny,path", [(96, 48, 0), (96, 48, 1), (700, 610, 0)])
def test_a_blob_brings_its_inflow_velocity_into_captured_steps(gpu_lib, precision, nx, ny, path):
    def lattice(u_in):
        lat = lbm.Lattice(nx, ny, 0.8, "mod_b", circles=[(0.32 * nx, 0.49 * ny, 0.13 * ny)],
                          eos=lbm.make_eos(lbm.EOS_NONE), precision=precision, kernel_path=path)
        lat.init_fields(np.ones(nx * ny))
        lat.set_inflow(u_in)
        return lat

    a = lattice(0.04)
    a.step(64)
    blob = a.save_state()
    a.step(80)
    want = a.fields() + (np.array(a.force()),)
    a.close()
    b = lattice(0.08)
    b.step(64)  # two graphs, captured with 0.08
    b.load_state(blob)
    b.step(80)
    got = b.fields() + (np.array(b.force()),)
    b.close()
    solid = np.isnan(want[0])
    assert np.isfinite(want[1][~solid]).all()
    for x, y in zip(got, want):
        assert np.array_equal(x, y, equal_nan=True)
