"""Block shapes of the 3D row pass on team FFTs, from the sources (no GPU)."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2103_10203_gb300", "csrc")

SRC = r"""
#include <cstdio>
#include "rf_fft3.cuh"
int main() {
#define X(L, R, M) \
  std::printf("%d %d %d %d\n", L, R * M, rfk::fft3::row_teams(R * M), rfk::fft3::row_threads(R * M));
  RF_TEAM_SIDES(X)
#undef X
}
"""


def test_row_blocks_are_whole_warps_that_hold_their_teams(tmp_path):
    """The final pass sums over the block with shuffles of all 32 lanes of each warp."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "shapes.cu", tmp_path / "shapes"
    src.write_text(SRC)
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC,
                    "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    rows = [tuple(int(v) for v in line.split()) for line in out.splitlines()]
    assert {r[0] for r in rows} >= {48, 96, 192, 384}
    for side, lanes, teams, threads in rows:
        assert threads % 32 == 0 and threads <= 256, side
        assert 0 <= threads - teams * lanes < 32, side
