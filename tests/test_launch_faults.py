"""What the library's calls do when a launch or a copy that they issue fails:
the error comes back from that call, no step is counted and no copy stays in
flight.  The CUDA runtime is a fake in the helper (tests/launch_faults.cu),
which runs with no GPU visible."""
import os
import subprocess

from paper_1809_08683_gb300 import lbm

HERE = os.path.dirname(os.path.abspath(__file__))


def test_failed_launches_and_copies(tmp_path):
    exe = str(tmp_path / "launch_faults")
    # no device code is wanted: PTX alone, not optimised, compiles fastest
    subprocess.check_call([lbm._nvcc(), "-O0", "-Xcicc", "-O0", "-std=c++17", "-gencode",
                           "arch=compute_103a,code=compute_103a", "-o", exe, os.path.join(HERE, "launch_faults.cu")])
    r = subprocess.run([exe], env=dict(os.environ, CUDA_VISIBLE_DEVICES="-1"), capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
