"""What bench.py reports about the kernels that it timed."""
import pytest

import bench


@pytest.mark.gpu
def test_fp64_path_times_the_kernels_that_step_fp64_lattices():
    out = bench.fp64_path(n_side=192, steps=2)
    assert out["kernel"] == "k_collide_node" and out["ms_per_step"] > 0
    assert 0 < out["frac_of_fp64_rate"] < 1.1
