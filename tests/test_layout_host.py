"""Packed-code positions of the cache layout, checked on the host (no GPU): `host_layout_check.cpp` includes the
library's layout header, and verifies that every position function is a bijection and that the decode kernel's
mask arithmetic on byte-ordered rows / chunks yields code x weight for the promised (token, channel)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2602_23200_b200", "csrc")


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs a host C++ compiler")
def test_positions_are_bijections_and_operand_bytes_are_code_times_weight(tmp_path):
    exe = str(tmp_path / "host_layout_check")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-o", exe, os.path.join(HERE, "host_layout_check.cpp")],
                   check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert r.stdout.strip().endswith("0 failure(s)")


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs a host C++ compiler")
def test_division_by_the_quantisers_constants_is_correctly_rounded(tmp_path):
    exe = str(tmp_path / "div_const_check")
    subprocess.run(["g++", "-std=c++17", "-O2", "-march=native", "-ffp-contract=off", "-I", CSRC, "-o", exe,
                    os.path.join(HERE, "div_const_check.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs a host C++ compiler")
def test_every_launch_has_a_grid_whose_partials_and_tickets_fit(tmp_path):
    exe = str(tmp_path / "host_split_check")
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", CSRC, "-o", exe, os.path.join(HERE, "host_split_check.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs a host C++ compiler")
def test_decode_launches_go_without_a_cluster_that_cannot_be_placed(tmp_path):
    exe = str(tmp_path / "host_cluster_check")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-I", "/usr/local/cuda/include", "-o", exe,
                    os.path.join(HERE, "host_cluster_check.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
