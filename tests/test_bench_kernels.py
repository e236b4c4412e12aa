"""What bench.py reports about the kernels that it timed."""
import pytest

import bench


def test_traffic_is_reported_for_the_measured_shape_only(tmp_path, monkeypatch):
    (tmp_path / "profiles").mkdir()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    monkeypatch.setattr(bench, "kernel_source_hash", lambda: "abc")
    path = tmp_path / "profiles" / "traffic_w.txt"
    text = "kernel = k_collide_pair\nworkload = w\nsource_sha256 = abc\ndram_bytes_per_launch = 5\n"
    path.write_text(text + "shape = default\n")
    assert bench.read_traffic("w", "k_collide_pair", None) == 5.0
    assert bench.read_traffic("w", "k_collide_pair", (128, 48, 1)) is None
    path.write_text(text + "shape = 128,48,1\n")
    assert bench.read_traffic("w", "k_collide_pair", (128, 48, 1)) == 5.0
    assert bench.read_traffic("w", "k_collide_pair", None) is None
    path.write_text(text)                        # a summary that names no shape is of the default one
    assert bench.read_traffic("w", "k_collide_pair", (128, 48, 1)) is None


@pytest.mark.gpu
def test_fp64_path_times_the_kernels_that_step_fp64_lattices():
    out = bench.fp64_path(n_side=192, steps=2)
    assert out["kernel"] == "k_collide_node" and out["ms_per_step"] > 0
    assert 0 < out["frac_of_fp64_rate"] < 1.1
