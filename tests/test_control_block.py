"""The clearing of the control block at the start of a batch, compiled for the host with checked array
bounds: what a batch counts starts from zero whatever the number of threads, what persists is kept."""
import os
import subprocess

import pytest

from paper_2305_07238_gb300 import build as B

PROGRAM = r"""
#include "pmc_internal.h"
#include <cstring>
using namespace pmc;
int main() {
    constexpr uint32_t N = sizeof(Control) / 4, EPOCH = offsetof(Control, epoch) / 4, MID = offsetof(Control, mid_count) / 4;
    for (uint32_t T : {1u, 7u, 32u, 33u, 256u, 1024u})
        for (int rounds = 0; rounds < 2; ++rounds) {
            Control c;
            std::memset(&c, 0xA5, sizeof(c));
            for (uint32_t t = 0; t < T; ++t) clear_control(&c, rounds, t, T);
            uint32_t w[N];
            std::memcpy(w, &c, sizeof(c));
            for (uint32_t i = 0; i < N; ++i)
                if (w[i] != (i < EPOCH || (rounds && i >= MID) ? 0u : 0xA5A5A5A5u)) return 1;
        }
    return 0;
}
"""


def test_clear_control(tmp_path):
    try:
        nvcc = B.nvcc_path()
    except RuntimeError:
        pytest.skip("no nvcc")
    src, exe = tmp_path / "clear.cpp", tmp_path / "clear"
    src.write_text(PROGRAM)
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    # an index past an array's end ends the program
    subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=bounds", "-fsanitize-undefined-trap-on-error", "-I", B.CSRC,
                    "-I", B.INCLUDE, "-I", inc, "-o", str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
