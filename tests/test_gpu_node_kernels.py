"""The node kernels (k_prep, k_collide_node) give the bits of the strip
kernels: the same node arithmetic, contraction written out, so the states are
compared for equality, over both storage precisions, every EOS, viscosity law
and force mode, walls on either pair of sides, second-order extrapolation,
the smallest lattices and sizes around a CTA of 128 nodes."""
import numpy as np
import pytest

from paper_1809_08683_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    from paper_1809_08683_gb300 import lbm as m
    return m


def configs(precision):
    p = {"precision": precision}
    yield W.periodic_box(1, 1, **p)
    yield W.periodic_box(5, 3, eos=(W.EOS_DECOUPLING, ()), **p)
    yield W.periodic_box(127, 9, eos=(W.EOS_CS, ()), force=(1e-5, -2e-5), **p)
    yield W.periodic_box(130, 67, eos=(W.EOS_CUBIC, (0.05, 0.2)), visc_law=2, force=(1e-5, 2e-5), force_mode=1, **p)
    yield W.periodic_box(33, 20, corrections=0, **p)
    yield W.cavity(N=4, Ra=10.0, eps=0.02, tau0=0.8, **p)
    yield W.cavity(N=67, Ra=1e4, eps=0.6, **p)
    yield W.cavity(N=186, Ra=1e5, eps=0.4, eos=(W.EOS_CUBIC, (0.05, 0.2)), **p)   # cavity-model instance
    yield W.cavity(N=40, Ra=1e4, eps=0.1, order=2, tau0=0.8, **p)
    yield W.couette_variable_mu(nx=1, ny=32, **p)
    yield W.periodic_box(64, 64, **p)                                             # most nodes of one cluster in FP32
    yield W.cavity(N=65, Ra=1e4, eps=0.3, **p)                                    # one row and column beyond
    yield W.poiseuille(nx=16, ny=128, **p)                                        # most nodes of one cluster in FP64
    yield W.poiseuille(nx=4, ny=128, **p)
    yield W.poiseuille(nx=200, ny=61, Th=1.01, **p)
    c = W.periodic_box(37, 29, **p)                                               # walls in x, periodic in y
    c["walls"] = [W.periodic(), W.periodic(), W.wall((0, 0.02), 1.02, 0, 2), W.wall((0, 0), 1.0, 1, 1)]
    yield c


def start(lat, cfg, seed):
    f, g = W.df_noise(cfg["nx"], cfg["ny"], seed, 1e-4)
    lat.init_macros(*W.random_macros(cfg["nx"], cfg["ny"], seed))
    f0, g0 = lat.get_state()
    lat.set_state(f0 + f, g0 + g)


@pytest.mark.parametrize("precision", [0, 1])
def test_node_kernels_equal_strips(lbm, precision):
    for k, cfg in enumerate(configs(precision)):
        a, b, c = lbm.Lattice(cfg), lbm.Lattice(cfg), lbm.Lattice(cfg)
        _, _, pair = a.tile()
        # strips that give the default shape's bits, and the node kernels by name
        b.set_tile(*((128, 7, 1) if pair == 1 else (30, 5, 4) if k % 2 else (64, 6, 0)))
        c.set_tile(128, 1, 6)
        for lat in (a, b, c):
            start(lat, cfg, 100 + k)
            lat.step(7)
            lat.step(300 if 1 < cfg["nx"] < 40 else 4)   # 300: more than one cluster launch
            lat.sync()
        for x, y in zip(a.get_state(), b.get_state()):
            assert np.array_equal(x, y), (k, cfg["nx"], cfg["ny"])
        if pair != 1:   # pair 6 rounds FP32 stores with the draws of pairs 0 and 4
            for x, y in zip(a.get_state(), c.get_state()):
                assert np.array_equal(x, y), (k, cfg["nx"], cfg["ny"])
        assert c.tile() == (128, 1, 6)
        for lat in (a, b, c):
            lat.close()


@pytest.mark.parametrize("graph_steps", [0, 4])
def test_batch_of_node_and_strip_members_equals_alone(lbm, graph_steps):
    import torch
    st = torch.cuda.Stream()
    cfgs = [W.cavity(N=48, Ra=1e4, eps=0.5, precision=1), W.poiseuille(nx=9, ny=40, precision=0),
            W.cavity(N=200, Ra=1e5, eps=0.5, precision=1), W.periodic_box(33, 31, precision=1),
            W.cavity(N=50, Ra=1e4, eps=0.5, precision=0)]
    alone = [lbm.Lattice(c, stream=st) for c in cfgs]
    mixed = [lbm.Lattice(c, stream=st) for c in cfgs]
    for lats in (alone, mixed):
        lats[3].set_tile(32, 6, 0)      # strips beside node members
        lats[4].set_tile(30, 8, 4)
        for k, lat in enumerate(lats):
            start(lat, cfgs[k], 7 + k)
    batch = lbm.Batch(mixed, graph_steps=graph_steps)
    for n in (8, 4):
        batch.step(n)
        for lat in alone:
            lat.step(n)
    for x, y in zip(alone, mixed):
        assert all(np.array_equal(p, q) for p, q in zip(x.get_state(), y.get_state()))
        assert x.steps == y.steps == 12
    batch.close()


@pytest.mark.parametrize("cfg", [W.poiseuille(nx=499, ny=421, precision=1), W.cavity(N=520, Ra=1e6, eps=0.5, precision=0)],
                         ids=["fp32", "fp64-prep"])
def test_several_tiles_per_cta(lbm, cfg):
    a, b = lbm.Lattice(cfg), lbm.Lattice(cfg)
    b.set_tile(64, 8, 0)
    for lat in (a, b):
        lat.init_macros(*W.random_macros(cfg["nx"], cfg["ny"], 3))
        lat.step(3)
    for x, y in zip(a.get_state(), b.get_state()):
        assert np.array_equal(x, y)
    a.close()
    b.close()


def test_narrow_members_beside_many_wide_nodes(lbm):
    """More than 600,000 nodes of up to 160 columns beside as many wider ones:
    node kernels and strips in one batch, against each in its strips alone."""
    import torch
    st = torch.cuda.Stream()
    cfgs = [W.periodic_box(160, 2000, precision=1), W.poiseuille(nx=100, ny=3001, precision=1),
            W.periodic_box(161, 3800, precision=1)]
    alone = [lbm.Lattice(c, stream=st) for c in cfgs]
    mixed = [lbm.Lattice(c, stream=st) for c in cfgs]
    for k, (a, b) in enumerate(zip(alone, mixed)):
        a.set_tile(*((30, 8, 4) if k < 2 else (128, 8, 0)))
        for lat in (a, b):
            lat.init_macros(*W.random_macros(cfgs[k]["nx"], cfgs[k]["ny"], 60 + k))
    batch = lbm.Batch(mixed, graph_steps=2)
    batch.step(4)
    for a, b in zip(alone, mixed):
        a.step(4)
        assert all(np.array_equal(p, q) for p, q in zip(a.get_state(), b.get_state()))
    batch.close()
    for lat in alone + mixed:
        lat.close()
