"""Arc arithmetic at the largest graphs (csrc/arc_index.h, compiled for the host): a row that
ends at 2^31 - 2 arcs is walked with every stride the kernels use, each arc once and none
past the end."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_14895_gb300", "csrc")
PROGRAM = r"""
#include <cstdio>
#include "arc_index.h"
using namespace fsgp;
int main() {
    const int32_t e = 2147483646;
    const int strides[] = {1, 8, 16, 32, 256};
    for (int stride : strides)
        for (int32_t len = 0; len < 600; ++len) {
            const int32_t b0 = e - len;
            int64_t seen = 0;
            uint32_t b = (uint32_t)b0;
            int rounds = 0;
            while (b < (uint32_t)e && ++rounds < 1000) {
                for (int lane = 0; lane < stride; ++lane)
                    if (arc_in((int32_t)b, lane, e)) {
                        const uint32_t a = b + (uint32_t)lane;
                        if (a < (uint32_t)b0 || a >= (uint32_t)e) { std::printf("arc %u of row %d\n", a, b0); return 1; }
                        ++seen;
                    }
                b += (uint32_t)stride;
            }
            if (seen != len) { std::printf("stride %d len %d: %lld arcs\n", stride, len, (long long)seen); return 1; }
        }
    if (arc_chunks(e, 65535) != 32769 || arc_chunks(0, 32) != 0 || arc_chunks(33, 32) != 2) { std::printf("chunks\n"); return 1; }
    return 0;
}
"""


def test_last_row_of_the_largest_graph(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(tmp_path / "t")], check=True)
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
