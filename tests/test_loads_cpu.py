"""A warp's pending copies (csrc/fds_loads.h): after it gives up on one, it waits once more for exactly
those that were issued and have not arrived -- the one it gave up on too, and none that never was."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1512_02951_gb300", "csrc")

# Runs of subtiles as restore loads them (private parts in one or two buffers), where copy number
# `bad` never arrives; the barriers keep the number of phases announced and completed.
DRIVER = r"""
#include "fds_loads.h"
#include <cstdio>
using namespace fds;
struct Bars {
  int announced[3] = {0, 0, 0}, completed[3] = {0, 0, 0}, copies = 0, bad;
  bool stuck[3] = {false, false, false};
  void copy(Loads& ld, int i) {
    ld.issued(i);
    ++announced[i];
    if (copies++ == bad) stuck[i] = true; else ++completed[i];
  }
  // mbarrier.try_wait.parity: the phase of that parity is the last completed one
  bool wait(int i, unsigned parity) { return completed[i] > 0 && ((completed[i] - 1) & 1u) == parity; }
};
int main() {
  int checks = 0;
  for (int twice = 0; twice < 2; ++twice)
    for (int runs = 1; runs <= 4; ++runs)
      for (int len = 1; len <= 3; ++len)
        for (int bad = -1; bad < runs * (len + 1); ++bad) {
          Bars b;
          b.bad = bad;
          Loads ld;
          bool lost = false;
          int half = 0;
          b.copy(ld, 0);
          b.copy(ld, 1);
          for (int r = 0; r < runs && !lost; ++r) {
            const bool more = r + 1 < runs;
            if (twice && more) b.copy(ld, 1 + (half ^ 1));
            if (!b.wait(1 + half, ld.parity(1 + half))) { lost = true; break; }
            ld.arrived(1 + half);
            for (int t = 0; t < len; ++t) {
              if (!b.wait(0, ld.parity(0))) { lost = true; break; }
              ld.arrived(0);
              if (t + 1 < len || more) b.copy(ld, 0);
              if (!twice && more && t + 1 == len) b.copy(ld, 1);
            }
            if (twice) half ^= 1;
          }
          if (lost != (bad >= 0)) return printf("lost %d of copy %d\n", lost, bad), 1;
          // under way: announced and not yet waited for, i.e. pending
          int waited[3] = {0, 0, 0};
          ld.drain(3, [&](int i, unsigned parity) {
            ++waited[i];
            // either it has arrived, or it is the one that never does and the parity is its phase's
            if (!b.wait(i, parity) && !(b.stuck[i] && parity == ((unsigned)b.completed[i] & 1u))) waited[i] = 100;
          });
          for (int i = 0; i < 3; ++i) {
            if (waited[i] > 1) return printf("wrong phase on barrier %d\n", i), 1;
            if (waited[i] != (ld.pending(i) ? 1 : 0)) return printf("barrier %d\n", i), 1;
            if (b.stuck[i] && !waited[i]) return printf("copy given up on is left (barrier %d)\n", i), 1;
            if (waited[i] && b.announced[i] == 0) return printf("no copy was issued on barrier %d\n", i), 1;
          }
          if (!lost && (waited[0] || waited[1] || waited[2])) return printf("a copy is left\n"), 1;
          ++checks;
        }
  printf("ok %d\n", checks);
  return 0;
}
"""


def test_drain_waits_for_what_is_under_way(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "loads.cpp", tmp_path / "loads"
    src.write_text(DRIVER)
    subprocess.run([gxx, "-std=c++17", "-O1", "-I" + CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0 and out.stdout.startswith("ok"), out.stdout


@pytest.mark.parametrize("unit", ["fds_protect_warp.cu", "fds_restore_warp.cu"])
def test_warp_kernels_wait_through_their_pending_copies(unit):
    with open(os.path.join(CSRC, unit)) as f:
        text = f.read()
    assert not re.search(r"\bmbar_wait\(", text)      # load_wait and load_drain only
    kernels = len(re.findall(r"__global__ void", text))
    assert len(re.findall(r"if \((?:BULK && )?lost\) load_drain\(ld, ", text)) == kernels
