"""The record ring of the 128-token kernel, its real code compiled for the host: no order of the roles may stall it."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2607_24027_b200", "csrc")


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    exe = str(tmp_path_factory.mktemp("ring") / "record_ring")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, os.path.join(HERE, "record_ring.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("records", [
    "1 1 / 3 2 / 1 4",                           # a tile in every record, as in the other modes
    "20 0 0 0 0 / 20 0 0 0 0 / 0 0 0 0 0",       # one busy chunk, then more empty records than the ring holds
    "4 0 0 0 0 0 0 3 / 0 0 0 0 0 0 0 1",
    "30 0 / 0 0 / 0 0 / 2 0 / 0 2",              # empty items behind a busy one
    "10 / 0 / 0 / 0 / 0 / 1 / 0 / 0 / 0 / 0 / 0 / 2",
    "0 0 0 / 0 0 0 / 0 0 0",
])
def test_no_order_stalls(model, records):
    r = subprocess.run([model, "300", *records.split()], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
