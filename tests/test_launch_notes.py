"""What the launchers remember about a stream (csrc/launch_notes.h), as a host program: a GEMV or GEMM may start early only where
one is known to have been launched on the stream since the last packing there."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_11357_b200", "csrc")

PRELUDE = r"""
#include "launch_notes.h"
#include <cstdio>
using namespace tf;
static LaunchNotes n;
static StreamName on(unsigned long long stream, unsigned long long capture = 0) { return {stream, capture, true}; }
static const StreamName nobody = {0, 0, false};
static bool early(const StreamName& s) { return n.look(s).kind != LaunchKind::kNone; }
static void gemv(const StreamName& s, LaunchKind kind = LaunchKind::kHalfSm) { n.launched(s, n.look(s), kind); }
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main() {
"""

CASES = {
    "a stream not seen before, one with a GEMV, one with a packing behind it": r"""
        CHECK(!early(on(1)));
        gemv(on(1)); CHECK(early(on(1)) && n.look(on(1)).kind == LaunchKind::kHalfSm && !early(on(2)));
        gemv(on(1), LaunchKind::kWholeSm); CHECK(n.look(on(1)).kind == LaunchKind::kWholeSm);
        n.packed(on(1)); CHECK(!early(on(1)));
        gemv(on(1)); CHECK(early(on(1)));
    """,
    "other streams may push an entry out, and never a packing": r"""
        gemv(on(1)); n.packed(on(1));
        for (int s = 2; s < 2 + 3 * LaunchNotes::kEntries; ++s) { gemv(on(s)); CHECK(early(on(s)) && !early(on(1))); }
        gemv(on(1));
        for (int s = 2; s < 2 + 3 * LaunchNotes::kEntries; ++s) gemv(on(s));
        CHECK(!early(on(1)));
    """,
    "a packing leaves the other streams alone": r"""
        gemv(on(1)); gemv(on(2)); n.packed(on(1));
        CHECK(!early(on(1)) && early(on(2)));
    """,
    "what is captured on a stream says nothing about what runs on it": r"""
        gemv(on(1)); n.packed(on(1));
        gemv(on(1, 7)); CHECK(early(on(1, 7)) && !early(on(1)) && !early(on(1, 8)));
        gemv(on(1)); n.packed(on(1, 7)); CHECK(early(on(1)) && !early(on(1, 7)));
    """,
    "a captured packing: every stream of the capture is forgotten": r"""
        gemv(on(1, 7)); gemv(on(2, 7)); gemv(on(2, 8)); n.packed(on(1, 7));
        CHECK(!early(on(1, 7)) && !early(on(2, 7)) && early(on(2, 8)));
    """,
    "a packing by another thread between a launch's question and its note": r"""
        gemv(on(1));
        const LaunchNotes::Seen before = n.look(on(1));
        n.packed(on(1));
        n.launched(on(1), before, LaunchKind::kWholeSm); CHECK(!early(on(1)));
        const LaunchNotes::Seen unseen = n.look(on(3));
        n.packed(on(3));
        n.launched(on(3), unseen, LaunchKind::kWholeSm); CHECK(!early(on(3)));
    """,
    "a stream that the runtime could not name": r"""
        gemv(on(1)); gemv(nobody); CHECK(!early(nobody) && early(on(1)));
        n.packed(nobody); CHECK(!early(on(1)));
    """,
}


@pytest.mark.parametrize("name", CASES)
def test_notes(name, tmp_path):
    source, program = tmp_path / "notes.cpp", tmp_path / "notes"
    source.write_text(PRELUDE + CASES[name] + "return 0; }\n")
    res = subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-Wno-unused", "-I" + CSRC, str(source), "-o", str(program)], capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    res = subprocess.run([str(program)], capture_output=True, text=True, timeout=60)
    assert res.returncode == 0, res.stdout
