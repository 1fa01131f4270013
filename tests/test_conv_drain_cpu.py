"""The waits of a convolution CTA that gave up (cv_drain), run on the CPU against a model of its
barriers: whatever was still in flight when the K loop stopped has completed when they return."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MODEL = r"""
#include <cstdio>
#include <initializer_list>
#include "ewh_conv.cuh"
using namespace ewh;
int main() {
  long runs = 0;
  for (int steps = 1; steps <= 11; ++steps)
    for (int stages = 1; stages <= 4; ++stages)
      for (int mul = 0; mul <= steps; ++mul)                              // MMAs issued for steps < mul
        for (int iss = mul; iss <= steps && iss <= mul + stages; ++iss)   // loads requested for steps < iss
          for (int com = 0; com <= mul; ++com) {                          // commits that have completed
            if (iss > stages && com < iss - stages) continue;             // a stage is filled again after its MMAs
            for (int arrived = mul; arrived <= iss; ++arrived) {          // loads that have landed
              int landed = arrived, commits = com;
              bool ran_out = false;
              // phases that a barrier has completed, given what has landed / completed
              auto phases = [&](CvBar kind, int stage) {
                int n = 0;
                if (kind == CV_DONE) return commits == steps ? 1 : 0;
                for (int s = stage; s < (kind == CV_FULL ? landed : commits); s += stages)
                  n += kind == CV_FULL || s + 1 < steps;
                return n;
              };
              cv_drain(iss, mul, steps, stages, [&](CvBar kind, int stage, unsigned parity) {
                // in flight: loads land and commits complete in order, one by one, while a wait lasts
                while ((phases(kind, stage) & 1) == (int)parity) {
                  if (kind == CV_FULL && landed < iss) ++landed;
                  else if (kind != CV_FULL && commits < mul) ++commits;
                  else { ran_out = true; return; }
                }
              });
              if (ran_out || landed != iss || commits != mul) {
                printf("steps %d stages %d multiplied %d issued %d: landed %d, committed %d%s\n", steps, stages, mul, iss,
                       landed, commits, ran_out ? ", a wait ran out" : "");
                return 1;
              }
              ++runs;
            }
          }
  printf("%ld\n", runs);
  return 0;
}
"""


def test_drain_covers_everything_in_flight(tmp_path):
    cuda = "/usr/local/cuda/include"
    if not shutil.which("g++") or not os.path.isdir(cuda):
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = tmp_path / "drain.cpp", str(tmp_path / "drain")
    src.write_text(MODEL)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2205_12344_gb300", "csrc"), "-I", cuda,
                    str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout) > 1000
