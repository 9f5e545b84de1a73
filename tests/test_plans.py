"""The kernels' shared-memory plans, asked of the library itself (host code; 148 SMs with 227 KB of shared memory a block)."""
import os
import subprocess


from helpers import WALK_SHAPES
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


WALK = r"""
#include <cstdio>
#include "ts_walk.cuh"
int main() {
  ts_ctx c{}; c.num_sms = SMS; c.max_smem = SMEM; c.cfg.D = 8; c.cfg.K = 8; c.cfg.Nmax = 64; c.cfg.max_batch = 4096;
  int B, tma;
  while (std::scanf("%d %d %d %d", &c.cfg.V, &c.cfg.r, &B, &tma) == 4) {
    c.vt_TV = ((c.cfg.V + SMS - 1) / SMS + 63) / 64 * 64; c.vt_n = (c.cfg.V + c.vt_TV - 1) / c.vt_TV;
    ts::WalkPlan p{};
    const bool ok = ts::walk_plan(&c, B, tma != 0, &p);
    std::printf("%d %d %d %d %d %d %d %d %d\n", ok ? 1 : 0, p.ring, p.req, p.cols, 1 << p.lsets, p.tr, (int)p.smem, c.vt_TV, c.vt_n);
  }
}
"""


def test_walk_forms_that_the_parity_tests_stand_for(tmp_path):
    got = ask(tmp_path, WALK, [(*s, int(s[0] % 8 == 0)) for s in WALK_SHAPES])
    for shape, want, g in zip(WALK_SHAPES, WALK_SHAPES.values(), got):
        assert g[0] == 1 and (int(g[1] > 0), g[2], g[4], g[5]) == want, (shape, g)


def test_every_walk_whose_weights_fit_has_a_tensor_core_plan(tmp_path):
    """A range of W in shared memory beside one tile of head rows and the walks' state is all that the walk needs at least: a
    plan must be found wherever that much fits (ranks padded to 64, 16 KB of static memory, the state of an owner 360 bytes),
    resident where there is no tensor map (ragged rows, or none to be had)."""
    grid = [(V, r, B, tma) for V0 in (*range(100, 4000, 300), *range(4000, 262000, 6000)) for V, tma in ((V0 // 8 * 8, 1), (V0 // 8 * 8, 0), (V0 | 1, 0)) for r in (8, 24, 56, 64, 96, 128, 160, 192, 256) for B in (1, 3, 8, 16, 17, 32, 33, 64, 128, 400, 1500, 4096)]
    missing = []
    for (V, r, B, tma), (ok, ring, req, cols, sets, tr, smem, TV, n) in zip(grid, ask(tmp_path, WALK, grid)):
        slab, ntile = (r + 63) // 64 * 8192, (TV + 127) // 128
        least = max(TV // 64 * slab, 17 * 1024) + slab + 512 + 1024 + (B + n - 1) // n * 360
        if tma:   # streamed otherwise
            least = min(least, 2 * 2 * slab + slab + 1536 + (B + n - 1) // n * 360)
        if not ok:
            missing += [(V, r, B, tma)] if least <= SMEM - 16 * 1024 else []
            continue
        real = (r + 15) // 16 * 2048   # bytes of 64 tokens of W
        assert smem <= SMEM - 2048 and sets * tr * cols <= 512 and sets in (1, 2, 4) and 1 <= tr <= 3 and cols >= max(req, 16)
        assert sets * tr >= ntile or sets == 4   # several rounds only where all sets have tiles
        assert smem >= (ring * 2 if ring else ntile * 2) * real   # the MMAs of a half tile read the other half's place too
        assert tma or ring == 0
    assert not missing, (len(missing), missing[:8])
