"""A bounded wait of a step kernel that gave up fails every blocking read of the lattice with
LBM_ETIMEOUT, until its state is set anew.  The wait for the wall pass in front of the tiles is run on a
count that nothing raises, with a short limit."""
import time

import numpy as np
import pytest

from paper_1908_09235_gb300 import lbm

pytestmark = pytest.mark.gpu

NX, NY = 700, 610  # single-phase FP32 of this size has its wall pass in front of the tiles
READS = {"mass": lambda lat: lat.mass(), "fields": lambda lat: lat.fields(),
         "force": lambda lat: lat.force(), "save_state": lambda lat: lat.save_state()}


def _channel():
    lat = lbm.Lattice(NX, NY, 0.8, "mod_b", circles=[(0.3 * NX, 0.5 * NY, 40.5)],
                      eos=lbm.make_eos(lbm.EOS_NONE), precision=lbm.FP32_DEV)
    lat.init_fields(np.ones(NX * NY))
    lat.set_inflow(0.05)
    return lat


def _expire(lat):
    t0 = time.perf_counter()
    assert lbm.lbm_selftest_front_wait(lat.ctx, 50_000_000, 0) == (5, 0)
    assert 0.045 < time.perf_counter() - t0 < 10.0


@pytest.mark.parametrize("read", sorted(READS))
def test_a_wait_that_gave_up_fails_the_next_read(gpu_lib, read):
    lat = _channel()
    assert lbm.lbm_selftest_front_wait(lat.ctx, 50_000_000, 1) == (0, 1)
    lat.step(3)
    READS[read](lat)
    _expire(lat)
    lat.step(3)
    with pytest.raises(lbm.LBMError) as e:
        READS[read](lat)
    assert e.value.status == 5  # LBM_ETIMEOUT, and sticky
    with pytest.raises(lbm.LBMError):
        lat.step(1)
    lat.close()


@pytest.mark.parametrize("how", ["init", "load"])
def test_a_new_state_waits_again(gpu_lib, how):
    lat = _channel()
    lat.step(5)
    blob = lat.save_state()
    lat.step(35)
    want = lat.fields()
    _expire(lat)
    if how == "init":
        lat.init_fields(np.ones(NX * NY))
        lat.step(5)
    else:
        lat.load_state(blob)
    lat.step(35)
    assert lbm.lbm_selftest_front_wait(lat.ctx, 50_000_000, 1) == (0, 1)
    for x, y in zip(lat.fields(), want):
        assert np.array_equal(x, y, equal_nan=True)
    lat.close()


def test_self_test_arguments(gpu_lib):
    lat = _channel()
    for limit in (0, -1, 10 ** 11):
        assert lbm.lbm_selftest_front_wait(lat.ctx, limit, 1)[0] == 1
    lat.close()
