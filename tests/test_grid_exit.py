"""Which status a launch reports when CTAs meet at barriers with a time limit (csrc/zgr_grid_exit.h, host logic compiled with g++)."""
import itertools
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_12917_b200", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "zgr_grid_exit.h"
struct Words {
  unsigned out = 0; bool failed = false;
  void fail() { failed = true; }
  bool count_out(unsigned n) { const bool last = out == n - 1; out = last ? 0 : out + 1; return last; }
  bool take_failed() { const bool f = failed; failed = false; return f; }
};
int main(int argc, char** argv) {           // statuses of the CTAs in the order in which they leave; every launch runs twice
  Words words;
  for (int launch = 0; launch < 2; ++launch)
    for (int i = 1; i < argc; ++i) {
      int status = launch == 0 ? std::atoi(argv[i]) : 0;
      if (zgr::leave_grid(words, argc - 1, status)) std::printf("%d:%d ", i, status);
    }
}
"""


def test_a_cta_that_gave_up_fails_the_launch_whoever_leaves_last(tmp_path):
    src, exe = tmp_path / "exit.cpp", tmp_path / "exit"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    # all passed, dependent columns (the same verdict everywhere), and every mix of CTAs that gave up with one that passed late
    for statuses in [(0,), (0, 0, 0), (5, 5, 5)] + list(itertools.product((0, -1), repeat=3)):
        out = subprocess.run([str(exe)] + [str(s) for s in statuses], check=True, capture_output=True, text=True).stdout.split()
        n = len(statuses)
        assert out == [f"{n}:{-1 if -1 in statuses else statuses[-1]}", f"{n}:0"]      # and the next launch starts clean
