"""The refill of a stage of the one-launch extraction's state ring
(csrc/refill_stage.cuh), on the host: no stage is armed and no copy started once
a wait of any lane has run out, that of the chunk's data or that of its
readers, and the lanes learn of it."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_13576_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "refill_stage.cuh"

// Two lanes stand for a warp: bit 0 / 1 of `arrived` and `freed` say whether the
// lane's waits for the data and for the readers succeed.  The vote of lane l
// takes the other lane's value from what its waits give.
int main() {
  int bad = 0;
  for (int arrived = 0; arrived < 4; ++arrived)
    for (int freed = 0; freed < 4; ++freed) {
      int copies = 0, waited = 0;
      bool back[2];
      for (int l = 0; l < 2; ++l) {
        const bool other = ((arrived & freed) >> (1 - l)) & 1;
        back[l] = mape_detail::refill_stage(
            (arrived >> l) & 1, [&] { ++waited; return ((freed >> l) & 1) != 0; },
            [&](bool b) { return b && other; }, [&] { ++copies; });
      }
      const bool fine = arrived == 3 && freed == 3;
      const bool lanes = back[0] == (((arrived & freed) & 1) != 0) && back[1] == (((arrived & freed) & 2) != 0);
      if (copies != (fine ? 2 : 0) || waited != 2 || !lanes) {
        std::printf("arrived %d freed %d: copies %d back %d %d\n", arrived, freed, copies, back[0], back[1]);
        ++bad;
      }
    }
  return bad ? 1 : 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_no_stage_is_armed_after_a_wait_ran_out(tmp_path):
    src = tmp_path / "refill.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "refill"
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
