"""Row/column splits of the four-step transforms (host side of mg_fftp.cuh), no GPU: every split that planning and the
autotuner may choose keeps a column's lookups inside that column's own twiddle table, its tile inside the column
buffer and its rows inside the row kernels.  Compiled with nvcc as host code."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2509_15948_gb300", "csrc")

CHECK = r'''
#include <algorithm>
#include <cstdio>
#include "mg_fftp.cuh"
using namespace mg;
int main() {
  int admitted = 0, table = 0, tile = 0, rows = 0;
  for (int f : {1, 3, 5})
    for (int logN = 10; logN <= 23; ++logN)
      for (int logN1 = 0; logN1 <= logN; ++logN1) {
        if (!split_ok(f, logN, logN1)) continue;
        ++admitted;
        const int logN2 = logN - logN1, N2 = 1 << logN2;
        const int G = std::min(8, std::min(8192 >> logN2, 1 << logN1));
        for (int gg = 0; gg < G; ++gg)
          for (int k2 = 0; k2 < N2; ++k2) {   // what the column pass multiplies: entries k2 mod 64 and 64 + k2 / 64
            const int lo = gg * kColTwS + (k2 & 63), hi = gg * kColTwS + 64 + (k2 >> 6);
            table += lo / kColTwS != gg || hi / kColTwS != gg;
          }
        tile += G < 1 || N2 * G > 8192;
        rows += (f << logN1) > (f == 1 ? 2048 : (f == 3 ? 3072 : 2560)) || logN1 < 4 || logN2 < 3;
      }
  printf("%d %d %d %d\n", admitted, table, tile, rows);
  return 0;
}
'''


def test_every_admitted_split_fits_the_column_and_row_kernels(tmp_path):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    src = tmp_path / "check.cu"
    src.write_text(CHECK)
    exe = tmp_path / "check"
    subprocess.run([nvcc, "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True, capture_output=True,
                   timeout=300)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60).stdout.split()
    admitted, table, tile, rows = map(int, out)
    assert admitted > 0 and table == 0 and tile == 0 and rows == 0, out
