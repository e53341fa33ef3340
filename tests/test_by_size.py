"""BySize (internal.h), the widths that a call remembers by its instances' sizes: right for
every size however many share a slot, and found once for a size that repeats."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2501_03245_gb300", "csrc")
SRC = """
#include <cstdio>
#include "internal.h"
int main() {
  ecc::BySize<int> memo;
  int calls = 0, wrong = 0;
  auto f = [&](uint64_t n) { ++calls; return (int)(n % 1000003); };
  for (int turn = 0; turn < 3; ++turn)
    for (uint64_t n = 0; n < 5000; ++n) wrong += memo.get(n, [&] { return f(n); }) != (int)n;
  for (uint64_t n : {0ull, 1ull << 28, ~0ull, 1ull << 63})
    for (int i = 0; i < 2; ++i) wrong += memo.get(n, [&] { return f(n); }) != (int)(n % 1000003);
  calls = 0;
  for (int i = 0; i < 65536; ++i) wrong += memo.get(1024 + i % 8, [&] { return f(1024 + i % 8); }) != 1024 + i % 8;
  std::printf("%d %d\\n", wrong, calls);
}
"""


def test_by_size(tmp_path):
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if shutil.which("g++") is None or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("no host compiler or CUDA headers")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", f"-I{CSRC}", f"-I{cuda}", str(src), "-o", str(exe)], check=True)
    wrong, calls = map(int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert wrong == 0 and calls <= 8
