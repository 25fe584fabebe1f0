"""How the GEMM's and the GEMV's work is dealt out (csrc/split.h), as a host program.  The owner of a cut tile waits for every CTA that
holds a part of it, so a range without a unit would be a wait for something that nobody stores."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_11357_b200", "csrc")

PRELUDE = r"""
#include "split.h"
#include <cstdio>
#include <initializer_list>
using namespace tf;
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return false; } } while (0)
// every CTA has a unit, the ranges follow one another, and owner() is the CTA whose range it is (asked at the ends of every range)
static bool sound(const Ranges& r, int units, int ctas) {
    CHECK(r.start(0) == 0 && r.start(ctas) == units);
    for (int c = 0; c < ctas; ++c) {
        CHECK(r.start(c) < r.start(c + 1));
        CHECK(r.owner(r.start(c)) == c && r.owner(r.start(c + 1) - 1) == c);
    }
    return true;
}
"""

CASES = {
    "ranges": r"""
        for (int units = 1; units <= 400; ++units)
            for (int ctas = 1; ctas <= units && ctas <= 160; ++ctas)
                for (int late : {0, 1, 10})
                    for (int less : {-6, -3, -1, 0, 1, 4, 6})
                        if (late < ctas && !sound(Ranges::make(units, ctas, late, less), units, ctas)) {
                            std::printf("units %d ctas %d late %d less %d\n", units, ctas, late, less);
                            return 1;
                        }
    """,
    "the GEMV's late CTAs": r"""
        for (int tiles = 24 * 148; tiles <= 256 * 512; tiles += 7)
            if (!sound(Ranges::make(tiles, 148, 10, 6), tiles, 148)) return std::printf("%d tiles\n", tiles), 1;
    """,
    "split": r"""
        for (int sms : {160, 148, 132, 80, 16})
            for (int ktiles = 1; ktiles <= 256; ++ktiles)
                for (int tiles = 1; tiles <= 4096; tiles += tiles < 330 ? 1 : 97)
                    for (int bt = 16; bt <= 256; bt += 16) {
                        const GemmSplit s = split_gemm(tiles, ktiles, bt, sms);
                        bool ok = s.grid >= 1 && s.grid <= sms && s.rows >= 1 && s.grid % s.rows == 0;
                        if (s.whole_tiles) ok = ok && s.rows == 1 && sound(s.ranges, tiles, s.grid);
                        else if (s.rows > 1) ok = ok && s.rows == tiles && sound(s.ranges, ktiles, s.grid / s.rows);      // a row of CTAs per tile
                        else ok = ok && sound(s.ranges, tiles * ktiles, s.grid);
                        if (!ok) return std::printf("%d tiles of %d k-tiles, bt %d, %d SMs\n", tiles, ktiles, bt, sms), 1;
                    }
    """,
    "token tiles": r"""
        for (int sms : {160, 148, 80, 16})
            for (int ktiles : {1, 3, 8, 32, 112, 256})
                for (int n_tiles : {1, 2, 9, 32, 87, 256})
                    for (int M = 1; M <= 4096; M += M < 300 ? 1 : 61) {
                        const GemmTiling t = choose_gemm_tiling(M, n_tiles, ktiles, sms);
                        const int tiles = (t.pair ? (n_tiles + 1) / 2 : n_tiles) * t.m_tiles;
                        // a kernel that exists, a slot that the workspace has room for, every token in a tile and no tile without one
                        bool ok = t.width <= gemm_widest_tile(M) && (t.width == 32 || t.width == 64 || t.width == 128 || t.width == 256);
                        ok = ok && t.bt % (t.pair ? 32 : 16) == 0 && (!t.pair || (t.width == 256 && 2 * t.split.grid <= sms)) && t.bt >= 16 && t.bt <= t.width && t.bt * t.m_tiles >= M && t.bt * (t.m_tiles - 1) < M;
                        if (t.split.whole_tiles) ok = ok && sound(t.split.ranges, tiles, t.split.grid);
                        else if (t.split.rows > 1) ok = ok && t.split.rows == tiles && sound(t.split.ranges, ktiles, t.split.grid / t.split.rows);
                        else ok = ok && sound(t.split.ranges, tiles * ktiles, t.split.grid);
                        if (!ok) return std::printf("M %d, %d n-tiles of %d k-tiles, %d SMs\n", M, n_tiles, ktiles, sms), 1;
                    }
    """,
}


@pytest.mark.parametrize("name", CASES)
def test_every_cta_has_work_and_every_unit_an_owner(name, tmp_path):
    source, program = tmp_path / "split.cpp", tmp_path / "split"
    source.write_text(PRELUDE + "int main() {" + CASES[name] + "return 0; }\n")
    res = subprocess.run(["g++", "-std=c++17", "-O2", "-I" + CSRC, str(source), "-o", str(program)], capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    res = subprocess.run([str(program)], capture_output=True, text=True, timeout=300)
    assert res.returncode == 0, res.stdout
