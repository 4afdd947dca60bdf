"""The few-orbit kernel's chunks cover every step of a run once and end, also
for runs whose length is within a chunk of 2^32 (a loop counting up in 32
bits by eight passes from 2^32 - 8 to 0 and starts again)."""
import os
import subprocess

from paper_1908_03869_gb300 import build

PROGRAM = r"""
#include <initializer_list>
#include "split_chunks.h"
int main() {
    const uint32_t top = 0xffffffffu;
    for (uint32_t steps : {0u, 1u, 7u, 8u, 9u, 16u, 17u, top - 8, top - 7, top - 1, top}) {
        uint64_t covered = 0, chunks = 0;
        sdeb::SplitChunks c(steps);
        for (; !c.done() && chunks <= steps / 8ull + 1; c.next(), ++chunks) {
            if (c.from != covered || c.last() != (covered + 8 >= steps)) return 1;
            covered += c.count();
        }
        if (!c.done() || covered != steps || chunks != (steps + 7ull) / 8) return 1;
    }
    return 0;
}
"""


def test_chunks_cover_the_run_and_end(tmp_path):
    src, exe = str(tmp_path / "chunks.cpp"), str(tmp_path / "chunks")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.abspath(build.CSRC), src, "-o", exe], check=True)
    assert subprocess.run([exe], timeout=120).returncode == 0
