"""The size of the cooperative rebuild launch (paper_2104_10231_gb300/csrc/grid.h):
every block has to be resident, so it follows from the SMs that the device
offers, whatever part the other launch shapes are tuned to."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2104_10231_gb300", "csrc")

DRIVER = r"""
#include "grid.h"
#include <cstdio>
int main() {
  int n = 0, bad = 0;
  for (int sms : {1, 7, 16, 76, 132, 148, 152, 160})
    for (int per : {1, 2, 8, 9, 16})
      for (int cells : {1, 27, 170, 1215, 1216, 1217, 40000}) {
        const int b = relres::cooperative_blocks(cells, sms, per);
        ++n;
        bad += b < 1 || b > sms * per || b > cells || (b < cells && b != sms * per);
      }
  std::printf("%d %d\n", n, bad);
  return bad ? 1 : 0;
}
"""


def test_cooperative_launches_fit_the_device(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    src = tmp_path / "grid_driver.cpp"
    src.write_text(DRIVER)
    exe = tmp_path / "grid_driver"
    subprocess.run([gxx, "-O1", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.split() == ["280", "0"], r.stdout


def test_the_rebuild_launch_is_sized_by_it():
    src = open(os.path.join(CSRC, "neighbor.cu")).read()
    body = src[src.index("cudaError_t launch_rebuild_fused("):]
    body = body[: body.index("\n}\n")]
    assert "cudaLaunchCooperativeKernel" in body and "cudaDevAttrMultiProcessorCount" in body
    assert "cooperative_blocks(" in body and "kPartSMs" not in body and "152" not in body
