"""Host rule of the two-step passes of general lengths (gensplit.hpp), compiled here: for
every axis length to 4096 and both precisions the column tile that the dispatch takes fits
in the 227 KB a block may ask for (less the kernel's own 64 bytes), and the split covers
the length with admissible radices."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "gensplit.hpp"
int main() {
  for (int fp32 = 0; fp32 < 2; ++fp32)
    for (int nv = 3; nv <= 6; nv += 3)
      for (int N = 2; N <= 4096; ++N) {
        int R1 = 0, R2 = 0;
        const bool ok = fh::gen_split(N, fp32 != 0, &R1, &R2);
        const int ct = fh::gen_columns(N, fp32 != 0, nv);
        std::printf("%d %d %d %d %d %d %d %zu\n", fp32, nv, N, ok ? R1 : 0, ok ? R2 : 0, ct,
                    ct ? fh::gen_col_stride(R1, R2, fp32 != 0, ct) : 0, ct ? fh::gen_col_bytes(N, fp32 != 0, nv, ct) : (size_t)0);
      }
}
"""


def test_column_tiles_fit(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src = tmp_path / "sizes.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "sizes"
    subprocess.run([cxx, "-std=c++17", "-I", os.path.join(ROOT, "paper_1701_04685_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    rows = [tuple(map(int, r.split())) for r in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.splitlines()]
    assert len(rows) == 4 * 4095
    taken = set()
    for fp32, nv, N, R1, R2, ct, stride, size in rows:
        radices = set(range(4, 17)) | ({18, 20, 24, 32} if fp32 else set())
        splits = [r for r in radices if N % r == 0 and N // r in radices]
        assert (R1 * R2 == N and R1 in radices and R2 in radices) if splits else R1 == R2 == 0
        if not ct:
            continue
        taken.add((fp32, nv, N))
        assert ct in (4, 8) and stride >= R1 * (R2 | 1)
        assert size == (N + nv * ct * stride) * (8 if fp32 else 16)
        assert size + 64 <= 227 * 1024
    for N in (576, 640, 768, 1024):   # tiles of eight columns of these do not fit
        assert (1, 6, N) in taken and (1, 3, N) in taken
