"""The rule by which a BN254 handle keeps its points' images (internal.h): never where a
table of window multiples from 8 bits up would then not fit the free memory."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2501_03245_gb300", "csrc")
SRC = """
#include <cstdio>
#include <cstdlib>
#include "internal.h"
int main(int, char** v) {
  std::printf("%d\\n", (int)ecc::images_fit(std::strtoull(v[1], 0, 10), std::strtoull(v[2], 0, 10)));
}
"""


def test_images_leave_room_for_a_table(tmp_path):
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if shutil.which("g++") is None or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("no host compiler or CUDA headers")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", f"-I{CSRC}", f"-I{cuda}", str(src), "-o", str(exe)], check=True)
    fits = lambda n, free: subprocess.run([str(exe), str(n), str(free)], check=True, capture_output=True,  # noqa: E731
                                          text=True).stdout.strip() == "1"
    for n in (1, 1 << 20, (1 << 26) + 7, 1 << 28):
        windows = (254 + 8) // 8  # of 8 bits
        need = 64 * n * (2 + windows)
        assert fits(n, need) and not fits(n, need - 64 * 34)
    assert fits(0, 0) and fits(1 << 26, 260 << 30) and not fits(1 << 28, 260 << 30)
