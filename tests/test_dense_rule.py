"""Which kernel a dense call takes, from the host function that decides it."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MAIN = """
#include <stdio.h>
#include <stdlib.h>
#include "common.cuh"
int main(int, char** a) {
  printf("%d", (int)sol::dense_in_pairs(atoi(a[1]), atoi(a[2]), atoi(a[3]), atoi(a[4]), 148));
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    cxx = shutil.which("g++")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    if cxx is None or not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        pytest.skip("no host compiler or no CUDA headers")
    d = tmp_path_factory.mktemp("rule")
    (d / "rule.cpp").write_text(MAIN)
    subprocess.run([cxx, "-std=c++17", "-I", os.path.join(cuda, "include"), "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2607_24027_b200", "csrc"), str(d / "rule.cpp"), "-o", str(d / "rule")],
                   check=True)
    return lambda *args: subprocess.run([str(d / "rule"), *map(str, args)], capture_output=True, check=True).stdout == b"1"


# heads, tokens: rounds of single tiles and of pairs on 148 SMs; where pairs are the faster at d = 128 and at d = 64
@pytest.mark.parametrize("H,N,d128,d64", [
    (1, 1, False, False), (2, 4096, False, False), (24, 700, False, False),         # 1 / 1
    (48, 700, True, True), (24, 1024, True, True),                                 # 2 / 1
    (24, 2048, False, False), (12, 4096, False, False),                            # 3 / 2
    (24, 3000, True, True), (30, 4096, False, False),                              # 4 / 2, 7 / 4
    (40, 4096, False, True), (24, 8500, False, True),                              # 9 / 5, 11 / 6
    (24, 4096, True, True), (40, 8192, True, True), (40, 32760, True, True),       # 6 / 3, 18 / 9, 70 / 35
])
def test_pairs_or_single_tiles(rule, H, N, d128, d64):
    assert rule(H, N, 128, 128) == d128
    assert rule(H, N, 64, 128) == d64
    assert rule(H, N, 64, 64) == rule(H, N, 128, 64) == (H * -(-N // 64) > 148)
