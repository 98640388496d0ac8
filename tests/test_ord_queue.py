"""The ordered queue of the chase (csrc/lr_ordq.h) on the host, under
interleavings that a GPU rarely takes: every position of the sequence goes to
exactly one thread (tests/ord_queue_model.cc).  Needs no GPU."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2606_09318_gb300", "csrc")


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path_factory.mktemp("ordq") / "model")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, os.path.join(HERE, "ord_queue_model.cc"), "-o", exe],
                   check=True, capture_output=True)
    return exe


@pytest.mark.parametrize("what", ["held", "1500"])
def test_every_position_once(model, what):
    r = subprocess.run([model, what], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
