"""The rows of a repeating residual that the Dense epilogue for grouped output rows fetches (csrc/residual_rows.cuh), compiled
for the host: the right one for every output row, none for the rows past the last in its last chunk of 32."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include "residual_rows.cuh"

int main() {
  const int rows[] = {32, 33, 63, 64, 100, 196, 1 << 20, 2147483647};
  for (int M = 1; M <= 300; ++M)
    for (int res_rows : rows)
      for (int row0 = 0; row0 < M; row0 += 32)
        for (int off = 0; off < 32; ++off) {
          const int got = ivit::residual_row(row0, (int)((unsigned)row0 % (unsigned)res_rows), off, M, res_rows);
          const int want = row0 + off < M ? (row0 + off) % res_rows : -1;
          if (got != want) { std::printf("M %d res_rows %d row %d: %d, not %d\n", M, res_rows, row0 + off, got, want); return 1; }
        }
  return 0;
}
"""


def test_residual_rows(tmp_path):
    (tmp_path / "t.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_2207_01405_b200", "csrc"), str(tmp_path / "t.cpp"),
                    "-o", str(tmp_path / "t")], check=True)
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
