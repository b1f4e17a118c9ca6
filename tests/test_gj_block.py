"""The 32 x 32 pivot elimination of the digit dielectric solve (csrc/gj_block.cuh), run on the host with 256
threads that go from barrier to barrier in several orders (tests/gj_block_check.cpp): the inverse must not
depend on the order, whichever lanes of a warp run ahead."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1602_02313_gb300", "csrc")


def test_elimination_in_any_thread_order(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "gj_block_check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-pthread", "-I", CSRC, os.path.join(HERE, "gj_block_check.cpp"), "-o", exe],
                   check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    print(r.stdout)
    assert r.returncode == 0, r.stdout
    assert "0 orders wrong" in r.stdout
