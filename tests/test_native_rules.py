"""Rules of the native code that can be run without a GPU: small C++ programs over the
library's own headers, with the CUDA side replaced by threads or fakes."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2312_02667_gb300", "csrc")


def run_native(name, tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no g++")
    exe = str(tmp_path / name)
    subprocess.run([gxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, os.path.join(HERE, "native", name + ".cpp"),
                    "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr


def test_a_warps_answer_is_the_same_on_every_lane(tmp_path):
    run_native("vote", tmp_path)


def test_what_belongs_to_a_device(tmp_path):
    run_native("device", tmp_path)
