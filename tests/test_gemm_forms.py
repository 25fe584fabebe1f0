"""The forms of the GEMM: token tiles up to 256 columns wide, by one CTA or by a pair, whole tiles, tiles cut in equal ranges and tiles with a row of CTAs
each.  csrc/split.h chooses, by an estimate; so each shape here is listed with the form that it is for, which a host program compares with the
choice (for the 148 SMs of a B200): when the estimate changes and a shape gets another form, that test fails, and the shape is to be replaced."""
import os
import subprocess

import numpy as np
import pytest
import torch

from helpers import bf16_bits_to_f64
from paper_2606_11357_b200 import binding as tf
from paper_2606_11357_b200 import workloads as wl

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_11357_b200", "csrc")

# (M, K, N) -> (width of the kernel, token columns of a tile, pair, how the work is cut); ragged tokens and columns, odd numbers of 128-column tiles, whose
# last pair has a half without columns
PAIRS = {
    (300, 4096, 14344): (256, 160, True, "ranges"),
    (600, 8192, 8200): (256, 224, True, "ranges"),
    (300, 1024, 32760): (256, 160, True, "whole"),
    (300, 8192, 4104): (256, 160, True, "rows"),
    (190, 8192, 9000): (256, 192, True, "rows"),
}
ALONE = {
    (160, 2048, 20008): (256, 160, False, "ranges"),
    (200, 512, 16392): (256, 208, False, "whole"),
    (250, 1024, 16392): (256, 256, False, "whole"),
    (160, 8192, 4104): (256, 160, False, "rows"),
    (300, 256, 12800): (128, 112, False, "whole"),
}
# shapes of the other GPU tests that are there for their form
OTHERS = {
    (1000, 4096, 4104): (256, 256, True, "whole"),
    (256, 32768, 2184): (256, 256, True, "rows"),
    (512, 32768, 4096): (256, 256, True, "ranges"),
    (2048, 4096, 14336): (256, 256, True, "ranges"),
    (200, 8192, 2048): (128, 112, False, "rows"),
    (96, 2944, 1096): (64, 48, False, "rows"),
}
FORMATS = [(4, 128), (4, 64), (4, 32), (8, 128)]

PROGRAM = r"""
#include "split.h"
#include <cstdio>
using namespace tf;
int main() {
    int M, K, N;
    while (std::scanf("%d %d %d", &M, &K, &N) == 3) {
        const GemmTiling t = choose_gemm_tiling(M, (N + 127) / 128, K / kTileK, 148);
        std::printf("%d %d %d %s\n", t.width, t.bt, t.pair, t.split.whole_tiles ? "whole" : t.split.rows > 1 ? "rows" : "ranges");
    }
}
"""


def test_each_shape_takes_the_form_that_it_is_listed_for(tmp_path):
    source, program = tmp_path / "forms.cpp", tmp_path / "forms"
    source.write_text(PROGRAM)
    res = subprocess.run(["g++", "-std=c++17", "-O1", "-I" + CSRC, str(source), "-o", str(program)], capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    want = {**PAIRS, **ALONE, **OTHERS}
    res = subprocess.run([str(program)], input="\n".join("%d %d %d" % shape for shape in want), capture_output=True, text=True, timeout=60)
    got = {}
    for shape, line in zip(want, res.stdout.splitlines()):
        width, bt, pair, cut = line.split()
        got[shape] = (int(width), int(bt), pair == "1", cut)
    assert got == want


@pytest.mark.gpu
@pytest.mark.parametrize("bits,group", FORMATS)
@pytest.mark.parametrize("M,K,N", [*PAIRS, *ALONE])
def test_forms(bits, group, M, K, N):
    import test_gpu_gemm
    test_gpu_gemm.test_gemm_cuts(bits, group, M, K, N)


@pytest.mark.gpu
@pytest.mark.parametrize("bits,group", FORMATS)
@pytest.mark.parametrize("M,K,N", [(300, 8192, 4104), (300, 1024, 32760), (200, 512, 16392), (300, 256, 12800)])
def test_integers_are_exact(bits, group, M, K, N):
    """s = 1 and small-integer activations: operands, products and fp32 sums (below 2^24) are exact, so a misplaced element of either operand shows."""
    import gpu_util as gu
    rng = np.random.default_rng(M + N)
    ai = rng.integers(-4, 5, size=(M, K))
    p = wl.make_w4(M, K, N, seed=6, group_size=group, keep_raw=True) if bits == 4 else wl.make_w8(M, K, N, seed=6, keep_raw=True)
    p.scales_f16 = np.ones_like(p.scales_f16)
    blob, a = torch.from_numpy(gu.pack(p)).cuda(), gu.to_device_bf16(wl.f32_to_bf16_bits(ai.astype(np.float32)))
    y = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device="cuda")
    ws = torch.zeros(tf.tf_workspace_size(tf.TF_OP_GEMM_W4A16 if bits == 4 else tf.TF_OP_GEMM_W8A16, M, K, N), dtype=torch.uint8, device="cuda")
    if group == 128:
        getattr(tf, f"tf_gemm_w{bits}a16")(blob, a, y, M, K, N, ws)
    else:
        tf.tf_gemm_w4a16_grouped(blob, a, y, M, K, N, group, ws)
    assert tf.tf_device_status(ws) == 0
    q = p.raw["q"].astype(np.float32)
    if bits == 4:
        q -= np.repeat(p.raw["z"].astype(np.float32), group, 0)
    exact = ai.astype(np.float32) @ q                        # in any order: whole numbers below 2^24
    assert np.array_equal(bf16_bits_to_f64(gu.bits_of(y)), bf16_bits_to_f64(wl.f32_to_bf16_bits(exact)))


@pytest.mark.gpu
@pytest.mark.parametrize("bits,M,K,N", [(4, 300, 4096, 14344), (8, 300, 8192, 4104), (4, 160, 2048, 20008)])
def test_waits_run_out_where_tiles_are_cut(bits, M, K, N):
    """Waits for the parts of another pair, or of another CTA with a wide token tile: whoever gives up first, all reach their end and the next call is right."""
    import test_gpu_failure
    try:
        test_gpu_failure.test_bounded_wait_runs_out_and_the_library_recovers("gemm", bits, M, K, N)
        test_gpu_failure.test_waits_that_run_out_while_the_data_arrives("gemm", bits, M, K, N)
    finally:
        tf.tf_debug_inject(0, False)


@pytest.mark.gpu
@pytest.mark.parametrize("M,K,N", [(300, 4096, 14344), (190, 8192, 9000)])
def test_cut_tiles_of_pairs_on_two_streams_at_once(M, K, N):
    """The launches of two streams share the SMs in any mixture; every call finishes and gives what it gives alone."""
    import gpu_util as gu
    p = wl.make_w4(M, K, N, seed=12)
    blob, a = torch.from_numpy(gu.pack(p)).cuda(), gu.to_device_bf16(p.a_bf16)
    want = gu.run(p, "gemm", blob_dev=blob)
    size = tf.tf_workspace_size(tf.TF_OP_GEMM_W4A16, M, K, N)
    lanes = [(torch.cuda.Stream(), torch.zeros(size, dtype=torch.uint8, device="cuda"), torch.empty((M, N), dtype=torch.bfloat16, device="cuda")) for _ in range(2)]
    torch.cuda.synchronize()
    for _ in range(50):
        for stream, ws, y in lanes:
            tf.tf_gemm_w4a16(blob, a, y, M, K, N, ws, stream=stream)
    torch.cuda.synchronize()
    for _, ws, y in lanes:
        assert tf.tf_device_status(ws) == 0
        assert np.array_equal(gu.bits_of(y), want)
