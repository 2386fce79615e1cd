"""Placement in the descriptor ring (csrc/stage_ring.cuh): the arrays that one
launch reads never share bytes, whatever their sizes and wherever the ring
stands, and lie inside the ring; a launch that cannot fit is refused.  (The case
that went wrong: descriptors of 15.9 MB and their offsets of 0.7 MB in 16 MB.)"""
import os
import subprocess

import paper_2402_09356_gb300 as tlr

CSRC = os.path.join(os.path.dirname(tlr.__file__), "csrc")

PROGRAM = r"""
#include <cstdio>
#include <random>
#include "stage_ring.cuh"
using namespace tlr;
int main() {
    std::mt19937_64 g(1);
    int bad = 0, refused = 0, restarts = 0, wrong = 0;
    for (size_t cap : {(size_t)4096, (size_t)65536, (size_t)16 << 20}) {
        size_t off = 0;
        for (int t = 0; t < 20000; ++t) {
            size_t b[3];
            for (size_t &v : b) v = g() % (t % 3 ? cap / 4 : cap) + 1;
            if (cap > 65536 && t == 0) b[0] = 170000 * 96, b[1] = 170001 * 4, b[2] = 1;
            bool restart = false;
            const size_t before = off, need = ring_bytes(b[0]) + ring_bytes(b[1]) + ring_bytes(b[2]);
            const bool ok = ring_room(cap, off, {b[0], b[1], b[2]}, restart);
            if (ok != (need <= cap)) ++wrong;
            if (!ok) {
                ++refused;
                if (off != before || restart) ++wrong;
                continue;
            }
            if (restart != (before + need > cap)) ++wrong;
            restarts += restart;
            size_t end = off;
            for (size_t v : b) {  // as the pushes of the launch place them
                bool again = false;
                if (!ring_room(cap, off, {v}, again) || again || off < end || off + v > cap) ++bad;
                off += ring_bytes(v);
                end = off;
            }
        }
    }
    std::printf("%d %d %d %d\n", bad, wrong, refused > 0, restarts > 0);
}
"""


def test_arrays_of_a_launch_do_not_overlap(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split() == ["0", "0", "1", "1"]
