"""The fp32 attention kernels' row / group quotient (csrc/row_division.cuh), compiled for the host: every
group size that a call may have, at the first and last row of every node."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include "row_division.cuh"
int main() {
  for (int group = 1; group <= 65535; ++group) {
    const ptd::GroupDivisor d = ptd::group_divisor(group);
    for (int node = 0; node < 128; ++node) {
      const int rows[3] = {node * group, node * group + group / 2, node * group + group - 1};
      for (int m : rows)
        if (ptd::divide_by_group(m, d) != m / group) {
          std::printf("%d / %d gives %d\n", m, group, ptd::divide_by_group(m, d));
          return 1;
        }
    }
  }
  return 0;
}
"""


def test_division_by_the_group_is_exact(tmp_path):
    src, exe = tmp_path / "division.cpp", tmp_path / "division"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2607_10661_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
