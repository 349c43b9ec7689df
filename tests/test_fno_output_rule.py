"""Host rule for the network's output (fno_out.hpp), compiled here: the last kernel writes
device memory of the network's own device and nothing else.  Another device's memory, which
needs two GPUs to try, takes the copy."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "fno_out.hpp"
int main() {
  for (int device_memory = 0; device_memory < 2; ++device_memory)
    for (int memory = -2; memory < 3; ++memory)   // -2: cudaInvalidDeviceId
      for (int own = 0; own < 3; ++own)
        std::printf("%d %d %d %d\n", device_memory, memory, own, (int)fh::writes_directly(device_memory != 0, memory, own));
}
"""


def test_only_own_device_memory_is_written_directly(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", os.path.join(ROOT, "paper_1701_04685_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    rows = [tuple(map(int, r.split())) for r in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.splitlines()]
    assert len(rows) == 2 * 5 * 3
    for device_memory, memory, own, direct in rows:
        assert direct == (device_memory == 1 and memory == own)
