"""Which launch shapes give one set of bits: the one-node kernels (pairs 0, 3,
4, 6 and the default of a lattice without paired strips) in the generic
instance of the node arithmetic, however FP32 stores round."""
import numpy as np
import pytest

from paper_1809_08683_gb300 import workloads as W

pytestmark = pytest.mark.gpu
ONE_NODE = [None, (128, 1, 6), (60, 5, 4), (64, 7, 3)]


@pytest.mark.parametrize("cfg", [W.cavity(N=100, Ra=1e4, eps=0.4, precision=1),
                                 W.periodic_box(301, 201, visc_law=2, force=(1e-5, 2e-5), force_mode=1, precision=1),
                                 W.periodic_box(130, 101, eos=(W.EOS_CS, ()), force=(1e-5, -2e-5), precision=1)],
                         ids=["cavity", "box", "carnahan-starling"])
@pytest.mark.parametrize("nearest", [False, True])
def test_generic_instance(cfg, nearest):
    from paper_1809_08683_gb300 import lbm

    def run(tile):
        lat = lbm.Lattice(cfg)
        if tile:
            lat.set_tile(*tile)
        lat.set_rounding(lbm.ROUND_NEAREST if nearest else lbm.ROUND_STOCHASTIC)
        lat.init_macros(*W.random_macros(cfg["nx"], cfg["ny"], 3))
        lat.step(40)
        lat.sync()
        state = lat.get_state()
        lat.close()
        return state

    ref = run((128, 7, 0))
    for tile in ONE_NODE:
        assert all(np.array_equal(a, b) for a, b in zip(run(tile), ref)), tile
