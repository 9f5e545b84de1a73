"""The rule by which cooperative kernels are chained to the kernel before them, with launches that fail on purpose."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "ts_launch.h"
int pair_error, plain_error, pair_calls, plain_calls;
int launch(bool chained) { ++(chained ? pair_calls : plain_calls); return chained ? pair_error : plain_error; }
void call(int& refused) {
  pair_calls = plain_calls = 0;
  const int e = ts::launch_chained(refused, launch);
  std::printf("%d %d %d %d\n", e, refused, pair_calls, plain_calls);
}
int main() {
  int refused = 0;
  call(refused);                                        // both fine
  pair_error = plain_error = 900; call(refused);        // the launch itself cannot be made
  pair_error = plain_error = 0; call(refused);          // ... and says nothing about the pair
  pair_error = 801; call(refused);                      // the pair is refused
  call(refused);                                        // and not asked for again
}
"""


def test_only_a_refusal_of_the_pair_is_remembered(tmp_path):
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2609_22098_b200", "csrc"), "-o", str(exe), str(src)])
    got = [tuple(map(int, line.split())) for line in subprocess.check_output([str(exe)], text=True).splitlines()]
    assert got == [(0, 0, 1, 0),      # (error, remembered, chained attempts, plain attempts)
                   (900, 0, 1, 1),
                   (0, 0, 1, 0),
                   (0, 1, 1, 1),
                   (0, 1, 0, 1)]
