"""Host rule of the cluster kernel's variants (clusterplan.cpp), compiled here, over every
grid N0 | L up to 1500 points a row: the schedules multiply to the axis lengths and use
only radices that the chosen kernel has; FP32 grids with a prime factor above 13 take the
staged kernel; a radix above 8 in FP64 only where a stage of it has more than 128
butterflies in a CTA of a cluster of 8; and the kinds of grids on both sides of each line."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1701_04685_gb300", "csrc")
POW2, GENERAL, STAGED = 0, 1, 2

PROGRAM = r"""
#include <cstdio>
#include <string>
#include "clusterkern.hpp"
namespace fh { void set_error(const std::string&) {} }
static void put(const fh::FftPlan& p) {
  std::printf(" %d", p.np);
  for (int q = 0; q < p.np; ++q) std::printf(" %d", p.r[q]);
}
int main() {
  for (int fp32 = 0; fp32 < 2; ++fp32)
    for (int nv = 3; nv <= 6; nv += 3)
      for (int N0 = 2; N0 <= 260; ++N0)
        for (int L = N0; L <= 1500; L += N0) {
          fh::ClusterChoice c;
          if (!fh::cluster_choice(N0, L, nv, fp32 != 0, &c)) return 1;
          std::printf("%d %d %d %d %d", fp32, nv, N0, L, c.kind);
          put(c.plan0);
          put(c.plan1);
          std::printf("\n");
        }
  return 0;
}
"""


def test_choice_over_all_grids(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "choice.cpp", tmp_path / "choice"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(src), os.path.join(CSRC, "clusterplan.cpp"),
                    os.path.join(CSRC, "lattice.cpp"), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    kinds = {}
    for line in out.splitlines():
        v = list(map(int, line.split()))
        fp32, nv, N0, L, kind = v[:5]
        p0 = v[6:6 + v[5]]
        p1 = v[7 + v[5]:]
        assert len(p1) == v[6 + v[5]]
        kinds[fp32, nv, N0, L] = kind
        lines = (nv * ((L // 2 + 8) // 8), ((N0 + 7) // 8 * nv + 1) // 2)
        for n, p, nl in ((N0, p0, lines[0]), (L, p1, lines[1])):
            prod = 1
            for r in p:
                prod *= r
                prime = all(r % q for q in range(2, r))
                if kind == POW2:
                    assert r in (2, 4, 8)
                elif kind == STAGED:
                    assert r in (2, 3, 4, 5, 7, 8, 11, 13) or (r > 13 and prime)
                else:
                    assert 2 <= r <= 16 or (not fp32 and r > 16 and prime)
                if not fp32 and r > 8 and not prime:
                    assert nl * (n // r) > 128
            assert prod == n
        assert (kind == POW2) == (N0 & (N0 - 1) == 0 and L & (L - 1) == 0)
        if fp32 and kind != POW2 and any(r > 13 for n in (N0, L) for r in range(17, n + 1, 2)
                                         if n % r == 0 and all(r % q for q in range(3, int(r ** 0.5) + 1, 2))):
            assert kind == STAGED
    for key, kind in {(1, 3, 17, 17): STAGED, (1, 3, 96, 96): GENERAL, (1, 3, 27, 27): STAGED, (1, 3, 162, 162): GENERAL,
                      (1, 3, 26, 26): GENERAL, (1, 3, 125, 125): STAGED, (1, 3, 5, 255): STAGED, (0, 3, 60, 60): STAGED,
                      (0, 3, 100, 100): GENERAL, (0, 3, 12, 240): STAGED, (0, 3, 22, 22): GENERAL, (0, 3, 64, 64): POW2}.items():
        assert kinds[key] == kind, key
