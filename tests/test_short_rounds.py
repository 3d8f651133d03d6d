"""Which launches of the fused kernel fit the stage width to the round
(csrc/short_rounds.h, compiled for the host): the choice at sizes where both
kernels were measured apart."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2609_38477_gb300", "csrc")

# (batch, rows, columns): fitted width faster; full width faster.
FITTED = [(1, 1024, 1024), (1, 64, 8192), (1, 4096, 256), (1, 2048, 2048), (1, 6000, 128), (2, 1024, 512),
          (2, 400, 2048), (2, 6000, 256), (4, 1024, 512), (4, 64, 8192), (4, 6000, 128), (4, 6000, 256)]
FULL = [(1, 64, 128), (1, 8, 8192), (1, 33, 2048), (1, 6000, 512), (1, 6000, 1024), (1, 11008, 256),
        (1, 4096, 4096), (2, 64, 128), (2, 8, 11008), (2, 11008, 128), (4, 8, 8192), (4, 11008, 128),
        (4, 4096, 1024)]

PROGRAM = r"""
#include "short_rounds.h"
#include <algorithm>
#include <cstdio>
#include <cstdlib>

int main(int, char **argv) {
  const int n = std::atoi(argv[1]), stage = n == 1 ? 27 : n == 2 ? 21 : 15;
  const int64_t rows = std::atoll(argv[2]);
  const int nb = std::atoi(argv[3]) / 8;
  const int64_t units = (rows + 31) / 32 * nb;
  const int ctas = (int)std::min<int64_t>(152, units);
  std::printf("%d\n", (int)seedq::short_rounds(n, units, ctas, 12 * stage, 1, rows, nb));
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_choice_at_measured_sizes(tmp_path):
    src = tmp_path / "short.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "short"
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    for want, sizes in ((1, FITTED), (0, FULL)):
        for size in sizes:
            r = subprocess.run([str(exe), *map(str, size)], capture_output=True, text=True, timeout=60)
            assert r.returncode == 0 and int(r.stdout) == want, (size, r.stdout)
