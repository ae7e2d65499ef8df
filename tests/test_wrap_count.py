"""The grid barrier's arrival count passes 2^32 in a long decode (456 arrivals
an early-terminated iteration on 152 SMs: after 9.4 million iterations).  The
comparison that its blocks poll with (csrc/wrap_count.h), compiled for the
host, walked through a wrap: a barrier opens at its last arrival, never
before."""
import os
import subprocess

HDR = os.path.join(os.path.dirname(os.path.abspath(__file__)), os.pardir, "paper_1711_01783_gb300", "csrc")

SRC = r"""
#include "wrap_count.h"
#include <cstdio>
int main() {
    const uint32_t grids[] = {1, 2, 115, 152};
    for (uint32_t grid : grids) {
        uint32_t count = 0u - 3u * grid - 1u, target = count;  // three barriers before the wrap, past it after
        for (int bar = 0; bar < 8; ++bar) {
            target += grid;
            for (uint32_t i = 0; i < grid; ++i) {
                if (mld::count_reached(count, target)) { std::printf("open early %u %d %u\n", grid, bar, i); return 1; }
                ++count;
            }
            // open from the last arrival on, while the next barrier's blocks arrive
            for (uint32_t i = 0; i < grid; ++i)
                if (!mld::count_reached(count + i, target)) { std::printf("shut %u %d %u\n", grid, bar, i); return 1; }
        }
    }
    return 0;
}
"""


def test_a_barrier_opens_at_its_last_arrival_across_the_wrap(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", HDR, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
