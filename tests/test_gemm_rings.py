"""Stages of the GEMM's rings (csrc/rings.h), as a host program: rings are whole rounds of the dequantization groups, so a few KB that something else takes
can halve what is on its way to a CTA, which no result shows."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_11357_b200", "csrc")

# (bits, groups per tile, width of the instantiation, token rows) -> stages of activations, of packed weights
STAGES = {
    (4, 1, 32, 32): (4, 8), (4, 1, 64, 64): (4, 8), (4, 1, 128, 80): (4, 8), (4, 1, 128, 96): (4, 6), (4, 1, 128, 112): (4, 6), (4, 1, 128, 128): (4, 4),
    (4, 2, 64, 64): (4, 8), (4, 2, 128, 80): (4, 6), (4, 2, 128, 112): (4, 6), (4, 2, 128, 128): (4, 4),
    (4, 4, 64, 64): (4, 8), (4, 4, 128, 64): (4, 8), (4, 4, 128, 80): (4, 6), (4, 4, 128, 128): (4, 4),
    (8, 1, 64, 64): (4, 8), (8, 1, 128, 80): (4, 8), (8, 1, 128, 96): (4, 4), (8, 1, 128, 128): (4, 4),
    (4, 1, 256, 128): (8, 4), (4, 1, 256, 176): (8, 4), (4, 1, 256, 208): (7, 4), (4, 1, 256, 240): (6, 4), (4, 1, 256, 256): (5, 4),
    (4, 2, 256, 176): (8, 4), (4, 2, 256, 208): (7, 4), (4, 2, 256, 240): (6, 4), (4, 4, 256, 176): (8, 4), (4, 4, 256, 240): (6, 4),
    (8, 1, 256, 128): (8, 4), (8, 1, 256, 240): (5, 4), (8, 1, 256, 256): (4, 4),
}

PROGRAM = r"""
#include "rings.h"
#include <cstdio>
using namespace tf;
int main() {
    int bits, G, width, rows;
    while (std::scanf("%d %d %d %d", &bits, &G, &width, &rows) == 4) {
        const GemmRings r = gemm_rings(bits, width, rows, G);
        const int used = kGemmSmemFixed + r.act_stages * r.act_stage_bytes + r.wp_stages * wp_stage_bytes(bits, width, G);
        const bool fits = used == r.smem_bytes && used <= kGemmSmemMax && r.wp_stages % (kGroups / chunk_tiles(bits, width)) == 0;
        std::printf("%d %d %d\n", r.act_stages, r.wp_stages, fits);
    }
}
"""


def test_stages(tmp_path):
    source, program = tmp_path / "rings.cpp", tmp_path / "rings"
    source.write_text(PROGRAM)
    res = subprocess.run(["g++", "-std=c++17", "-O1", "-I" + CSRC, str(source), "-o", str(program)], capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    res = subprocess.run([str(program)], input="\n".join("%d %d %d %d" % key for key in STAGES), capture_output=True, text=True, timeout=60)
    got = {key: tuple(map(int, line.split())) for key, line in zip(STAGES, res.stdout.splitlines())}
    assert got == {key: (*value, 1) for key, value in STAGES.items()}
