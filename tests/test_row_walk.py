"""The row walk's index arithmetic on the CPU (tests/host: one warp as 32
threads), over lists of one and several windows and of more than 2^31 entries."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HOST = os.path.join(ROOT, "tests", "host")


def test_row_walk_hands_out_every_entry_of_its_row(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    exe = str(tmp_path / "row_walk")
    subprocess.check_call([gxx, "-std=c++20", "-O1", "-w", "-pthread", "-I", HOST,
                           "-I", os.path.join(ROOT, "paper_1507_05086_gb300", "csrc"),
                           os.path.join(HOST, "row_walk.cpp"), "-o", exe])
    run = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert run.returncode == 0, run.stdout + run.stderr
