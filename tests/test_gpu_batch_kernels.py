"""lbm_batch_kernels names the kernels that a batch launches: a member's
reported shape is that of its strips also while node kernels step it."""
import ctypes as C

import pytest

from paper_1809_08683_gb300 import workloads as W


def test_null_batch_is_refused():
    from paper_1809_08683_gb300 import lbm
    lbm.build()
    assert lbm.load().lbm_batch_kernels(None, None, 0, None, None) == lbm.LBM_EINVAL


@pytest.mark.gpu
def test_names_and_launches():
    import torch
    from paper_1809_08683_gb300 import lbm
    st = torch.cuda.Stream()

    def kernels(cfgs, tiles=()):
        lats = [lbm.Lattice(c, stream=st) for c in cfgs]
        for lat, t in zip(lats, tiles):
            if t:
                lat.set_tile(*t)
        b = lbm.Batch(lats)
        b.step(2)
        out = b.kernels()
        if out == ("k_collide_node+k_collide_pair", 4, 1):   # names cut to the room given
            short = C.create_string_buffer(15)
            assert b.L.lbm_batch_kernels(b.h, short, 15, None, None) == lbm.LBM_OK and short.value == b"k_collide_node"
        b.close()
        for lat in lats:
            lat.close()
        return out

    c = lambda n, p: W.cavity(N=n, Ra=1e5, eps=0.5, precision=p)  # noqa: E731
    assert kernels([c(200, 0)]) == ("k_collide_node", 2, 1)
    assert kernels([c(200, 0)], [(128, 8, 0)]) == ("k_collide_stream", 2, 0)
    assert kernels([c(200, 1)]) == ("k_collide_node2", 2, 1)
    assert kernels([c(100, 1), c(200, 1), c(100, 0)]) == ("k_collide_node+k_collide_node2", 5, 2)
    assert kernels([c(1024, 1), c(100, 1)]) == ("k_collide_node+k_collide_pair", 4, 1)
    assert kernels([c(100, 1), c(100, 1)], [(30, 4, 4), (60, 4, 5)]) == ("k_collide_warp+k_collide_warp2", 3, 0)
