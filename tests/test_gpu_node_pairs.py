"""k_collide_node2 (two nodes per thread, wide FP32 lattices of the
cavity-model class) gives the bits of the paired strips where its index
arithmetic can go wrong: odd widths, whose last pair has one node, the wraps of
periodic sides in either direction, walls on one pair of sides only and
second-order extrapolation.  And several tiles per CTA of the FP64 collision,
which only a lattice of more than 64 fills of the GPU has."""
import numpy as np
import pytest

from paper_1809_08683_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def cavity_class_box(nx, ny, walls=None):
    c = W.periodic_box(nx, ny, precision=1, visc_law=2, force=(0.0, -1e-5), force_mode=1)
    if walls:
        c["walls"] = walls
    return c


WARM, COLD = W.wall((0, 0), 1.02, 0, 1), W.wall((0, 0), 0.98, 0, 2)
CASES = {
    "cavity-187": lambda: W.cavity(N=187, Ra=1e5, eps=0.4, precision=1),
    "cavity-189-order2": lambda: W.cavity(N=189, Ra=1e5, eps=0.4, order=2, precision=1),
    "box-201x167": lambda: cavity_class_box(201, 167),
    "box-200x165": lambda: cavity_class_box(200, 165),
    "box-161x205": lambda: cavity_class_box(161, 205),
    "walls-in-y-201x170": lambda: cavity_class_box(201, 170, [WARM, COLD, W.periodic(), W.periodic()]),
    "walls-in-x-203x171": lambda: cavity_class_box(203, 171, [W.periodic(), W.periodic(), COLD, WARM]),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_pairs_equal_paired_strips(name):
    from paper_1809_08683_gb300 import lbm
    cfg = CASES[name]()
    a, b = lbm.Lattice(cfg), lbm.Lattice(cfg)
    assert a.tile()[2] == 1                      # paired strips are the default shape
    assert lbm.Batch([a]).kernels()[0] == "k_collide_node2"
    b.set_tile(128, 7, 1)
    f, g = W.df_noise(cfg["nx"], cfg["ny"], 5, 1e-4)
    for lat in (a, b):
        lat.init_macros(*W.random_macros(cfg["nx"], cfg["ny"], 4))
        f0, g0 = lat.get_state()
        lat.set_state(f0 + f, g0 + g)
        lat.step(7)
        lat.step(4)
        lat.sync()
    for x, y in zip(a.get_state(), b.get_state()):
        assert np.array_equal(x, y)
    a.close()
    b.close()


def test_several_tiles_per_cta_of_a_large_fp64_lattice():
    from paper_1809_08683_gb300 import lbm
    cfg = W.periodic_box(2801, 2703)
    out = []
    for tile in (None, (128, 8, 0)):
        lat = lbm.Lattice(cfg)
        if tile:
            lat.set_tile(*tile)
        lat.init_macros(*W.random_macros(2801, 2703, 6))
        lat.step(3)
        out.append(lat.macros())
        lat.close()
    assert all(np.array_equal(out[0][k], out[1][k]) for k in out[0])
