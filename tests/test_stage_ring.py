"""The operand loader's walk over its ring of stages (csrc/stage_ring.h), compiled for the host and run
against a model of the mbarriers: when the reader of the stages stops after any number of them, the loader
arms nothing after the wait that gave up, never a stage whose reader is not done, and its closing waits
outlast every copy."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2009_12505_gb300", "csrc")

MODEL = r"""
#include <cstdio>
#include <vector>
#include "stage_ring.h"
// A barrier's phase `done` runs; a wait for parity p is over when the last finished phase has parity p.
struct Bar { int done = 0; bool over(uint32_t p) const { return ((done - 1) & 1) == (int)p; } };
template <int N> int run(int total, int batch, int reader) {
  Bar full[N], empty[N];
  std::vector<int> armed, landed;  // steps
  int read = 0, gave_up = 0;
  StageRing<N> r;
  auto land = [&] { int t = armed[landed.size()]; landed.push_back(t); ++full[t % N].done; };
  auto turn = [&](int) {
    // the reader keeps N - 1 stages behind until it stops for good
    while (read < reader && read < (int)armed.size() && (int)armed.size() - read >= N) {
      while ((int)landed.size() <= read) land();
      ++empty[read % N].done;
      ++read;
    }
    if (!r.fresh() && !empty[r.s].over(r.ph)) { ++gave_up; return false; }
    if (gave_up) return std::puts("armed after a wait that gave up"), true;
    if (r.step >= N && read < r.step - N + 1) std::puts("armed a stage that is still read");
    armed.push_back(r.step);
    return true;
  };
  for (int q = 0; q < total; q += batch)
    if (!ring_stages(r, total - q < batch ? total - q : batch, turn, [](bool c) { return c; })) break;
  if (r.step != (int)armed.size()) std::puts("the ring moved past a stage that was not armed");
  for (int t = r.pending(); t < r.step; ++t)
    while (!full[t % N].over((uint32_t)((t / N) & 1))) {
      if (landed.size() == armed.size()) return std::puts("a closing wait never ends"), 1;
      land();
    }
  if (landed.size() != armed.size()) std::puts("copies outlive the loader");
  const int want = reader + N < total ? reader + N : total;
  if ((int)armed.size() != want) std::printf("%d stages armed, not %d\n", (int)armed.size(), want);
  return 0;
}
int main() {
  for (int total : {1, 2, 5, 31, 32, 33, 70, 129})
    for (int batch : {1, 3, 32})
      for (int reader = 0; reader <= total; ++reader)
        run<3>(total, batch, reader), run<4>(total, batch, reader), run<5>(total, batch, reader);
  std::puts("done");
}
"""


def test_walk_stops_at_a_wait_that_gives_up(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    (tmp_path / "ring.cpp").write_text(MODEL)
    exe = str(tmp_path / "ring")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC,
                    str(tmp_path / "ring.cpp"), "-o", exe], check=True)
    assert subprocess.run([exe], check=True, capture_output=True, text=True).stdout == "done\n"
