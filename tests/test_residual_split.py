"""The split of the refinement residual over the chip (refine_split.h, host arithmetic): every tile size, tile count and
number of right-hand sides that a matrix can have, one 64-wide tile included, gives a group width, groups that hold the
right-hand sides, at least one and at most as many column ranges as there are tile columns, and partial sums of at most 30
MB.  A division by a count that is zero for the smallest sizes ends the process here."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = """
#include <cstdio>
#include "refine_split.h"
int main() {
  long seen = 0;
  for (int nb = 64; nb <= 2048; nb += 64)
    for (int nt = 1; nt <= 2500; nt += nt < 40 ? 1 : 97)
      for (int nrhs = 1; nrhs <= 3000; nrhs += nrhs < 70 ? 1 : 331)
        for (int sm : {1, 148, 152}) {
          const ResidualSplit s = residual_split(sm, nt, nb, nrhs);
          const bool width = s.P == 1 || s.P == 4 || s.P == 8 || s.P == 16 || s.P == 32;
          if (!width || (long)s.groups * s.P < nrhs || (long)(s.groups - 1) * s.P >= nrhs || s.nz < 1 || s.nz > nt ||
              s.partial((long)nt * nb) > 12ul * 64 * 32 * sm) {
            std::printf("nb %d nt %d nrhs %d sm %d: P %d groups %d nz %d\\n", nb, nt, nrhs, sm, s.P, s.groups, s.nz);
            return 1;
          }
          seen++;
        }
  std::printf("%ld splits\\n", seen);
  return 0;
}
"""


def test_every_size_has_a_split(tmp_path):
    src, exe = tmp_path / "split.cpp", tmp_path / "split"
    src.write_text(SRC)
    inc = os.path.join(ROOT, "paper_2408_04440_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", inc, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout)
