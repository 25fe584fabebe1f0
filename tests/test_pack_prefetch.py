"""What the host packer asks for ahead (csrc/pack.cpp), as a host program in which every prefetch is recorded: bytes show none of it."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_11357_b200", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdint>
#include <cstdlib>
#include <mutex>
#include <vector>
static std::mutex lock;
static std::vector<const uint8_t*> asked;
static void record(const void* p) { std::lock_guard<std::mutex> hold(lock); asked.push_back(static_cast<const uint8_t*>(p)); }
#define __builtin_prefetch(p) record(p)
#include "pack.cpp"
int main(int argc, char** argv) {
    const int bits = atoi(argv[1]), K = atoi(argv[2]), N = atoi(argv[3]), g = 128;
    const size_t row = (size_t)N * bits / 8;
    std::vector<uint32_t> q((size_t)K * row / 4 + 1), z((size_t)(K / g) * N / 8 + 1);
    std::vector<uint16_t> s((size_t)(K / g) * N);
    std::vector<uint8_t> out(tf_packed_size(bits, K, N, g));
    const tf_status st = bits == 4 ? tf_pack_awq(q.data(), s.data(), z.data(), K, N, g, out.data(), out.size())
                                   : tf_pack_w8(reinterpret_cast<const int8_t*>(q.data()), s.data(), K, N, g, out.data(), out.size());
    const uint8_t* base = reinterpret_cast<const uint8_t*>(q.data());
    long outside = 0, wrapped = 0;        // behind the matrix; in the next row, whose first line is no strip's successor
    for (const uint8_t* p : asked) {
        if (p < base || p >= base + (size_t)K * row) ++outside;
        else if ((size_t)(p - base) % row < 64) ++wrapped;
    }
    std::printf("%d %zu %ld %ld\n", (int)st, asked.size(), outside, wrapped);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    folder = tmp_path_factory.mktemp("prefetch")
    (folder / "prefetch.cpp").write_text(PROGRAM)
    res = subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I" + CSRC, str(folder / "prefetch.cpp"), "-o", str(folder / "prefetch")],
                         capture_output=True, text=True)
    assert res.returncode == 0, res.stderr

    def asked(bits, K, N):
        res = subprocess.run([str(folder / "prefetch"), str(bits), str(K), str(N)], capture_output=True, text=True, timeout=120)
        status, count, outside, wrapped = map(int, res.stdout.split())
        assert status == 0
        return count, outside, wrapped
    return asked


def test_int8_asks_ahead_for_large_blobs_only(program):
    assert program(8, 512, 512)[0] == 0 and program(8, 2048, 2048)[0] == 0
    assert program(8, 1024, 8256)[0] > 0


@pytest.mark.parametrize("bits,K,N", [(4, 256, 64), (4, 256, 128), (4, 256, 192), (4, 256, 200), (4, 256, 520), (4, 1024, 16384 + 64), (8, 1024, 8192), (8, 1024, 8264)])
def test_nothing_is_asked_for_behind_the_last_strip(program, bits, K, N):
    count, outside, wrapped = program(bits, K, N)
    assert (outside, wrapped) == (0, 0)
    assert count > 0 or N <= 128
