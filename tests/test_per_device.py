"""PerDevice (csrc/per_device.cuh): what a kernel launch needs from a device is
asked of every device of the process, once each, by whichever thread comes
first; a device past the table is asked every time."""
import os
import subprocess

import paper_2402_09356_gb300 as tlr

CSRC = os.path.join(os.path.dirname(tlr.__file__), "csrc")

PROGRAM = r"""
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.cuh"
int main() {
    tlr::PerDevice<int> p;
    std::atomic<int> asked[80] = {}, wrong{0};
    auto use = [&](int d) {
        if (p.get(d, [&] { ++asked[d]; return 100 + d; }) != 100 + d) ++wrong;
    };
    std::vector<std::thread> t;
    for (int k = 0; k < 8; ++k) t.emplace_back([&] { for (int r = 0; r < 50; ++r) for (int d : {0, 3, 63}) use(d); });
    for (auto &x : t) x.join();
    use(70);
    use(70);
    std::printf("%d %d %d %d %d\n", asked[0].load(), asked[3].load(), asked[63].load(), asked[70].load(), wrong.load());
}
"""


def test_once_per_device(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split() == ["1", "1", "1", "2", "0"]


def test_orderings_and_solve_ask_each_device():
    """Their attributes are not behind a flag of the process."""
    for name in ("order.cu", "solve.cu"):
        text = open(os.path.join(CSRC, name)).read()
        assert "PerDevice<bool>" in text and "once_flag" not in text
