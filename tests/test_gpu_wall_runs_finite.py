"""The runs that tests/test_gpu_wall_tiles.py compares bit for bit are runs of a finite fluid: the mass
ledger accepts each of them, and density and velocity are finite exactly at the fluid nodes.  And the
wall pass in front of the tiles with more bodies than its tiles test for (every tile then waits)."""
import numpy as np
import pytest

from paper_1908_09235_gb300 import lbm
from test_gpu_wall_tiles import CASES, SCHEMES, _lattice, _run, _same

pytestmark = pytest.mark.gpu


def _assert_finite(steps, *args):
    lat = _lattice(*args)
    lat.step(steps)
    solid = lat.flags() & 1 == 1
    mass = lat.mass()  # raises where a fluid density is not finite or not positive
    for x in lat.fields():
        assert np.array_equal(np.isfinite(x), ~solid)
    lat.close()
    assert mass > 0


@pytest.mark.parametrize("precision", [lbm.FP64, lbm.FP32_DEV, lbm.FP16_DEV])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "%dx%d-%s" % c[:3])
def test_small_lattices_stay_finite(gpu_lib, precision, case):
    nx, ny, kind, circles, walls = case
    for scheme in SCHEMES:
        _assert_finite(7, nx, ny, precision, scheme, 0, kind, circles, walls)


@pytest.mark.parametrize("precision,nx,ny,kind,steps,schemes", [
    (lbm.FP64, 250, 250, "cs", 35, ("mls", "mod_a", "mod_b")),
    (lbm.FP64, 400, 400, "none", 35, ("mls", "mod_a", "mod_b")),
    (lbm.FP32_DEV, 700, 700, "exp", 35, ("mls", "mod_a", "mod_b")),
    (lbm.FP32_DEV, 1301, 1000, "cs", 35, ("mls", "mod_a", "mod_b")),
    (lbm.FP16_DEV, 700, 700, "cs", 35, ("mls", "mod_a", "mod_b")),
    (lbm.FP16_DEV, 1451, 1400, "cs", 35, ("mls", "mod_a", "mod_b")),
    (lbm.FP16_DEV, 1124, 1125, "exp", 5, ("bouzidi_q", "mod_a", "mod_b")),
    (lbm.FP16_DEV, 1128, 1125, "cs", 5, ("bouzidi_q", "mod_a", "mod_b")),
    (lbm.FP32_DEV, 700, 610, "none", 5, ("bouzidi_q", "mod_a", "mod_b")),
    (lbm.FP16_DEV, 136, 9161, "exp", 7, ("mod_b", "zhao_yong")),
])
def test_larger_lattices_stay_finite(gpu_lib, precision, nx, ny, kind, steps, schemes):
    circles = [(0.3 * nx, 0.35 * ny, 0.11 * nx), (0.75 * nx, 0.3 * ny, 0.05 * nx)]
    for scheme in schemes:
        _assert_finite(steps, nx, ny, precision, scheme, 0, kind, circles, False)


@pytest.mark.parametrize("precision,nx,ny,kind", [
    (lbm.FP16_DEV, 1160, 1080, "cs"), (lbm.FP32_DEV, 700, 610, "none")])
@pytest.mark.parametrize("n", [4, 5, 16])
def test_more_bodies_than_the_tiles_in_front_test_for(gpu_lib, precision, nx, ny, kind, n):
    circles = [((0.1 + 0.2 * (k % 4)) * nx, (0.12 + 0.22 * (k // 4)) * ny, 9.3 + k) for k in range(n)]
    for scheme in ("bouzidi_q", "mod_b"):
        args = (nx, ny, precision, scheme)
        assert _same(_run([2, 1, 32], *args, 0, kind, circles, False),
                     _run([35], *args, 4, kind, circles, False)), scheme
    # (with 16 bodies, several of them inside the liquid, quadratic Bouzidi diverges in the oracle too)
    _assert_finite(35, nx, ny, precision, "mod_b", 0, kind, circles, False)
