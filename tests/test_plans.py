"""The kernels' shared-memory plans, asked of the library itself (host code; 148 SMs with 227 KB of shared memory a block)."""
import os
import subprocess

import pytest

from paper_2609_22098_b200 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SMS, SMEM = 148, 232448

TREE = r"""
#include <cstdio>
#include "ts_tree.cuh"
int main() {
  ts_config c{}; c.D = 8;
  while (std::scanf("%d %d %d %d %d", &c.V, &c.r, &c.K, &c.Nmax, &c.max_batch) == 5) {
    ts::TreePlan p{};
    const bool ok = ts::tree_plan(c, SMS, SMEM, &p);
    std::printf("%d %d %d %d\n", ok ? 1 : 0, p.BN, p.nW, p.ring_nW);
  }
}
"""


def ask(tmp_path, program, lines):
    """Compiles `program` against the library and runs it on `lines`; one tuple of numbers a line of its output."""
    lib = build.build()
    src, exe = tmp_path / "plan.cu", tmp_path / "plan"
    src.write_text(program)
    subprocess.check_call(["nvcc", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", f"-DSMS={SMS}", f"-DSMEM={SMEM}", "-I", build.CSRC, "-I", os.path.join(ROOT, "include"),
                           "-o", str(exe), str(src), lib, "-Xlinker", "-rpath=" + os.path.dirname(lib)])
    out = subprocess.run([str(exe)], input="\n".join(" ".join(map(str, x)) for x in lines), capture_output=True, text=True, check=True).stdout
    return [tuple(map(int, line.split())) for line in out.splitlines()]


# (V, r, K, Nmax, max_batch) -> tokens a block, stages of W, stages of W beside the base-logit ring: sizes at which a row's lists
# longer by one word would cost the ring or the blocks of 128 tokens, and two whose odd stage of W is left out
def test_the_expansions_plan_has_room_for_its_rings(tmp_path):
    want = {(64000, 48, 14, 64, 128): (1, 128, 8, 2), (64000, 224, 14, 64, 96): (1, 64, 3, 2), (64000, 200, 14, 64, 32): (1, 128, 2, 0),
            (64000, 160, 14, 64, 32): (1, 128, 2, 2), (64000, 128, 2, 64, 32): (1, 128, 4, 4)}
    got = dict(zip(want, ask(tmp_path, TREE, list(want))))
    assert got == want
