"""The wall pass inside the step kernels of small lattices (kernel_path 0) against the wall pass as a
launch of its own after the scalar tiles (kernel_path 1): the same bits.  Sizes on both sides of
every tile shape's range, with bodies and flat walls on tile edges and across the periodic seam,
several bodies in a tile, and runs of every length that ends in another set of moments."""
import numpy as np
import pytest

from paper_1908_09235_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu

SCHEMES = ["hbb", "mls", "bouzidi_l", "bouzidi_q", "zhao_yong", "mod_a", "mod_b", "bao",
           "bouzidi_l_a"]


def _lattice(nx, ny, precision, scheme, path, kind, circles, walls):
    kw = dict(circles=circles, precision=precision, kernel_path=path)
    if walls:
        kw.update(wall_q_lo=0.3, wall_q_hi=0.8)
    if kind == "none":
        lat = lbm.Lattice(nx, ny, 0.8, scheme, eos=lbm.make_eos(lbm.EOS_NONE, gx=1e-5, gy=-1e-4),
                          **kw)
        rng = np.random.default_rng(workloads.SEED)
        lat.init_fields(1.0 + 0.01 * rng.standard_normal(nx * ny))
        return lat
    if kind == "exp":
        eos = lbm.make_eos(lbm.EOS_EXP, **workloads.PAPER_E2["eos"], rho_wall=1.5)
        rl, rv = 2.783, 0.3675
    else:
        eos = lbm.make_eos(lbm.EOS_CS, **workloads.CS)
        rl, rv = lbm.lbm_coexistence(eos)
        eos.rho_wall = rv
    lat = lbm.Lattice(nx, ny, 1.0, scheme, eos=eos, **kw)
    lat.init_droplet(0.5 * nx, 0.6 * ny, 0.3 * min(nx, ny), 4.0, rl, rv)
    return lat


def _run(parts, *args):
    lat = _lattice(*args)
    for n in parts:
        lat.step(n)
    out = [np.nan_to_num(a, nan=-7.0) for a in lat.fields()]
    if args[3] != "zhao_yong":  # every population; Zhao-Yong's path 0 is the vector kernel, which
        out.append(lat.save_state())  # leaves other values in slots of solid nodes
    try:
        out.append(np.float64(lat.mass()))
    except lbm.LBMError as e:
        out.append(np.float64(-e.status))
    lat.close()
    return out


def _same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


# bodies: on the corners of 16- and 32-node tiles, three in one tile, near the periodic seam
CASES = [
    (100, 50, "none", [], True),
    (33, 37, "cs", [(16.0, 15.5, 6.2)], False),
    (64, 48, "cs", [(9.1, 8.2, 3.3), (22.4, 9.0, 4.1), (15.7, 22.9, 5.0), (45.5, 31.5, 8.0)], False),
    (40, 35, "exp", [(31.6, 16.1, 4.9)], True),
    (31, 90, "none", [(15.5, 60.25, 9.0)], True),
    (5, 30, "none", [], True),
]


@pytest.mark.parametrize("precision", [lbm.FP64, lbm.FP32_DEV, lbm.FP16_DEV])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "%dx%d-%s" % c[:3])
def test_wall_pass_in_the_tiles_gives_the_bits_of_the_wall_kernel(gpu_lib, precision, case):
    nx, ny, kind, circles, walls = case
    for scheme in SCHEMES:
        args = (nx, ny, precision, scheme)
        apart = _run([7], *args, 1, kind, circles, walls)
        assert _same(_run([7], *args, 0, kind, circles, walls), apart), scheme
        assert _same(_run([1, 2, 3, 1], *args, 0, kind, circles, walls), apart), scheme


@pytest.mark.parametrize("precision,nx,ny,kind", [
    (lbm.FP64, 250, 250, "cs"), (lbm.FP64, 630, 640, "cs"), (lbm.FP64, 400, 400, "none"),
    (lbm.FP32_DEV, 460, 460, "cs"), (lbm.FP32_DEV, 700, 700, "exp"),
    (lbm.FP32_DEV, 1301, 1000, "cs"), (lbm.FP32_DEV, 1003, 500, "none"),
    (lbm.FP16_DEV, 470, 460, "cs"), (lbm.FP16_DEV, 700, 700, "cs"), (lbm.FP16_DEV, 1451, 1400, "cs"),
])
def test_every_tile_shape_gives_the_bits_of_the_wall_kernel(gpu_lib, precision, nx, ny, kind):
    circles = [(0.3 * nx, 0.35 * ny, 0.11 * nx), (0.75 * nx, 0.3 * ny, 0.05 * nx)]
    for scheme in ("mls", "mod_a", "mod_b"):
        args = (nx, ny, precision, scheme)
        # a graph of 32 steps and a remainder
        assert _same(_run([35], *args, 0, kind, circles, False),
                     _run([35], *args, 1, kind, circles, False)), scheme


@pytest.mark.parametrize("precision,nx,ny,kind", [
    (lbm.FP32_DEV, 1600, 1603, "cs"), (lbm.FP16_DEV, 1124, 1125, "exp"),
    (lbm.FP16_DEV, 1128, 1125, "cs"), (lbm.FP32_DEV, 700, 610, "none"),
    (lbm.FP16_DEV, 644, 509, "none"), (lbm.FP32_DEV, 2056, 1250, "exp"),
])
def test_walls_in_front_of_the_tiles_give_the_bits_of_the_wall_kernel(gpu_lib, precision, nx, ny,
                                                                      kind):
    # large lattices (vector and marching kernel): ragged tiles in x and y, walls along the seam, two
    # bodies, one of them on tile edges; kernel_path 4 is the same kernel with the wall pass apart
    circles = [(0.3 * nx, 0.35 * ny, 0.11 * nx), (640.0 if nx > 700 else 512.0, 0.3 * ny, 20.5)]
    for scheme in ("bouzidi_q", "mod_a", "mod_b"):
        for walls in (False, True):
            args = (nx, ny, precision, scheme)
            apart = _run([5], *args, 4, kind, circles, walls)
            assert _same(_run([5], *args, 0, kind, circles, walls), apart), (scheme, walls)
            assert _same(_run([2, 1, 2], *args, 0, kind, circles, walls), apart), (scheme, walls)


@pytest.mark.parametrize("precision,nx,ny,kind", [
    (lbm.FP16_DEV, 1160, 1080, "cs"), (lbm.FP32_DEV, 700, 610, "none"), (lbm.FP64, 100, 90, "cs"),
])
def test_a_circle_round_the_fluid_may_cross_the_seam(gpu_lib, precision, nx, ny, kind):
    # the fluid inside a circle that leaves the lattice on the left, or at a corner: boundary nodes all
    # along the seam, far from the circle
    for circle in ((0.34 * nx, 0.5 * ny, 0.52 * nx, 1), (0.26 * nx, 0.28 * ny, 0.43 * nx, 1)):
        for scheme in ("bouzidi_q", "mod_b"):
            args = (nx, ny, precision, scheme)
            assert _same(_run([5], *args, 0, kind, [circle], False),
                         _run([5], *args, 4 if nx > 100 else 1, kind, [circle], False)), scheme


@pytest.mark.parametrize("precision", [lbm.FP64, lbm.FP32_DEV, lbm.FP16_DEV])
@pytest.mark.parametrize("nx,ny", [(120, 64), (121, 75), (800, 500)])
def test_channel_ends_in_the_tiles_give_the_bits_of_their_kernel(gpu_lib, precision, nx, ny):
    def run(path):
        lat = lbm.Lattice(nx, ny, 0.8, "mod_b", circles=[(0.4 * nx, 0.5 * ny, 0.1 * ny)],
                          eos=lbm.make_eos(lbm.EOS_NONE), precision=precision, kernel_path=path)
        lat.init_fields(np.ones(nx * ny), np.full(nx * ny, 0.05))
        lat.set_inflow(0.05)
        lat.step(35)
        out = [np.nan_to_num(a, nan=-7.0) for a in lat.fields()] + [np.array(lat.force())]
        lat.close()
        return out

    assert _same(run(0), run(1))


@pytest.mark.parametrize("nx,ny,kind", [(128, 9740, "cs"), (136, 9161, "exp"), (8, 65530, "cs"),
                                        (1048, 1189, "cs"), (1272, 1000, "exp")])
def test_the_marching_kernel_gives_the_bits_of_the_scalar_tiles(gpu_lib, nx, ny, kind):
    # FP16 lattices just above the size from which kernel_path 0 and 4 march: whole strips, a last
    # strip of one lane or 30, one strip of two lanes (its left and right neighbours itself), and
    # heights that are no multiple of a strip's rows; seven steps and their wall pass
    circles = [(0.5 * nx, 0.35 * ny, 0.2 * nx)] if nx > 8 else []
    for scheme in ("mod_b", "zhao_yong"):
        args = (nx, ny, lbm.FP16_DEV, scheme)
        a = _run([7], *args, 4, kind, circles, False)
        b = _run([7], *args, 1, kind, circles, False)
        assert _same(a[:3], b[:3]) and a[-1] == b[-1], scheme
