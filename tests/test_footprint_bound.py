"""The bound under which a brick's projected footprint stands for its voxels
(csrc/footprint_bound.h: image tests left out, depths of open bricks not
looked at), against the two binary32 projections voxel by voxel on the host:
far from the world's origin they part by more than the footprint's margin."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_voxel_leaves_a_footprint_that_holds(tmp_path):
    exe = str(tmp_path / "footprint_check")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I",
                           os.path.join(ROOT, "paper_1602_06645_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "host_checks", "footprint_check.cpp"), "-o", exe])
    r = subprocess.run([exe, "150000"], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
