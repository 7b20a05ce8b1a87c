"""The teams of a batched chip-resident launch and its message memory, on any number of SMs
(whole chips and slices): every team has a word inside the launch's memory and
the teams fit on the SMs.  The header is host code and is compiled as such."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include "batch_teams.h"
using namespace lap5;
int main() {
  for (int sms = 1; sms <= 160; ++sms)
    for (int split : kTeamSplits) {
      const int size = team_size(sms, split), teams = team_count(sms, size);
      const size_t end = kTeamWordOffset + (size_t)(teams - 1) * kTeamWordStride * 8 + 8;
      if (size < 1 || teams < 1 || teams * size > sms || end > kTeamLaunchBytes) {
        std::printf("%d SMs, teams of %d: %d\n", sms, size, teams);
        return 1;
      }
    }
  return 0;
}
"""


def test_every_team_has_a_word(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_1803_03797_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
