"""The rule for one or two points per lane, compiled for the host: at the sizes where both were measured
(152 SMs) it takes the faster one, or one at most 12 % slower."""
import os
import subprocess

import pytest

from paper_2305_07238_gb300 import build as B

PROGRAM = r"""
#include "cache_impl.h"
#include <cstdio>
int main() {
    int mode;
    unsigned n, mats, forced;
    double uneven, mean;
    while (std::scanf("%d %u %u %lf %lf %u", &mode, &n, &mats, &uneven, &mean, &forced) == 6) {
        pmc_cache c;
        c.num_sms = 152;
        c.n_mats = mats;
        c.uneven[0] = c.uneven[1] = uneven;
        c.mean_cost[0] = c.mean_cost[1] = mean;
        pmc::BatchArgs a{};
        a.n = n;
        a.use_cache = mode != 0;
        a.split = 1;
        a.keys_inline = mode == 1;
        a.one_point = a.roots_one_point = (int)forced;
        set_order(&c, &a);
        std::printf("%d %d\n", a.one_point, a.roots_one_point);
    }
}
"""

PLAIN, FIRST, OUTER = 0, 1, 2
# mode, points, networks, longest / mean program, mean program, us with two points per lane, with one
MEASURED = [
    (FIRST, 30720, 1, 1.0, 473, 17.6, 16.1), (FIRST, 65536, 1, 1.0, 473, 20.0, 22.0), (FIRST, 115200, 1, 1.0, 473, 25.5, 32.4),
    (FIRST, 230400, 1, 1.0, 473, 32.7, 39.7), (FIRST, 30720, 1, 1.0, 1596, 20.8, 19.1), (FIRST, 65536, 1, 1.0, 1596, 24.2, 24.6),
    (FIRST, 115200, 1, 1.0, 1596, 28.5, 31.3), (FIRST, 147456, 1, 1.0, 1596, 33.2, 40.5), (FIRST, 115200, 1, 1.0, 8363, 96.6, 75.7),
    (FIRST, 147456, 1, 1.0, 8363, 98.0, 85.0), (FIRST, 184320, 1, 1.0, 8363, 99.9, 117.6), (FIRST, 65536, 16, 1.65, 1388, 40.0, 30.3),
    (FIRST, 230400, 16, 1.65, 1388, 44.7, 49.0), (FIRST, 230400, 64, 2.47, 9656, 306.8, 185.0), (FIRST, 1040000, 64, 2.3, 9656, 384, 421),
    (FIRST, 518400, 512, 4.4, 20000, 556, 286), (FIRST, 2073600, 512, 4.4, 20000, 658, 759), (FIRST, 1040000, 1024, 6, 60000, 3182, 2666),
    (FIRST, 2073600, 1024, 6, 60000, 4650, 4976), (PLAIN, 16384, 1, 1.0, 473, 10.2, 10.1), (PLAIN, 115200, 1, 1.0, 473, 13.4, 15.3),
    (PLAIN, 147456, 1, 1.0, 473, 14.6, 17.4), (PLAIN, 115200, 1, 1.0, 1596, 21.8, 19.2), (PLAIN, 230400, 1, 1.0, 1596, 24.6, 26.8),
    (PLAIN, 147456, 1, 1.0, 8363, 77.0, 58.0), (PLAIN, 184320, 64, 2.47, 9656, 169.4, 147.9), (OUTER, 115200, 1, 1.0, 0, 10.1, 12.3),
    (OUTER, 115200, 1, 1.0, 567, 14.3, 16.4), (OUTER, 131072, 1, 1.0, 2307, 32.8, 24.6), (OUTER, 230400, 1, 1.0, 2307, 34.8, 36.8),
    (OUTER, 400000, 64, 2.91, 2296, 75.8, 57.3),
]


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    try:
        nvcc = B.nvcc_path()
    except RuntimeError:
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("rule")
    (d / "rule.cpp").write_text(PROGRAM)
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", B.CSRC, "-I", B.INCLUDE, "-I", inc, "-o", str(d / "rule"),
                    str(d / "rule.cpp")], check=True)

    def run(rows):
        text = "\n".join("%d %d %d %g %g %d" % r for r in rows)
        r = subprocess.run([str(d / "rule")], input=text, capture_output=True, text=True)
        return [tuple(map(int, line.split())) for line in r.stdout.splitlines()]
    return run


def test_measured_sizes(rule):
    got = rule([m[:5] + (0,) for m in MEASURED])
    for m, (one, roots) in zip(MEASURED, got, strict=True):
        assert m[6 if one else 5] <= 1.12 * min(m[5:]), m
        assert not roots   # the batched misses have a rule of their own


def test_asked_for(rule):
    assert rule([(mode, n, 1, 1.0, 473, 1) for mode in (PLAIN, FIRST, OUTER) for n in (1000, 10**7)]) == [(1, 1)] * 6
