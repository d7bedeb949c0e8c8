"""The rule for the cells per bin of the binned insert, compiled for the host: the sizes it was measured
at, and for any table and batch no more bins than the cache reserves room for and every cell in one."""
import os
import random
import subprocess

import pytest

from paper_2305_07238_gb300 import build as B

PROGRAM = r"""
#include "cache_impl.h"
#include <cstdio>
int main() {
    unsigned long long cells, n, roots, mats;
    while (std::scanf("%llu %llu %llu %llu", &cells, &n, &roots, &mats) == 4) {
        pmc_cache c;
        c.desc.n_cells = cells;
        c.n_mats = (uint32_t)mats;
        c.root_info.resize(roots);
        c.max_roots = (uint32_t)roots;   // one network has them all
        pmc::BatchArgs a{};
        a.n = (uint32_t)n;
        a.probe_cap = 0xFFFFFFFFu;
        set_bins(&c, &a);
        std::printf("%u %u %u\n", a.bin_shift, a.n_bins, pmc::insert_bins_max(cells));
    }
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    try:
        nvcc = B.nvcc_path()
    except RuntimeError:
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("bins")
    (d / "bins.cpp").write_text(PROGRAM)
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", B.CSRC, "-I", B.INCLUDE, "-I", inc, "-o", str(d / "bins"),
                    str(d / "bins.cpp")], check=True)

    def run(rows):   # cells, points, cacheable nodes of all networks, networks
        r = subprocess.run([str(d / "bins")], input="\n".join("%d %d %d %d" % p for p in rows), capture_output=True,
                           text=True)
        return [tuple(map(int, line.split())) for line in r.stdout.splitlines()]
    return run


# table cells, points, cacheable nodes per network (mean): cells per bin that measured fastest, or
# within a few percent of it
MEASURED = [(65536, 403200, 7.28, 32), (65536, 403200, 2.67, 64), (131072, 206755, 2.69, 256), (50021, 99301, 2.67, 256),
            (524288, 1050000, 1.70, 256), (262144, 403200, 7.28, 128), (262144, 1050000, 4.33, 64), (16384, 99301, 7.28, 32),
            (1024, 35000, 7.28, 4), (4096, 210000, 1.0, 16), (300000, 230400, 2.0, 256)]


def test_measured_sizes(rule):
    got = rule([(cells, n, int(roots * 100), 100) for cells, n, roots, _ in MEASURED])
    assert [1 << s for s, _, _ in got] == [m[3] for m in MEASURED]


def test_any_table_and_batch(rule):
    rng = random.Random(1)
    pairs = [(c, p) for c in (1, 2, 255, 256, 257, 8191, 8192, 8193, 65536, 1 << 21, (1 << 21) + 1, (1 << 32) - 1)
             for p in (0, 1, 1536, 1537, 10**5, 10**7, (1 << 32) - 1)]
    pairs += [(int(2 ** rng.uniform(0, 31)), int(2 ** rng.uniform(0, 32))) for _ in range(2000)]
    for (cells, probes), (s, bins, most) in zip(pairs, rule([(c, p, 1, 1) for c, p in pairs]), strict=True):
        assert s <= 8 and bins <= most
        assert (bins - 1) << s < cells <= bins << s
        assert s == 8 or bins <= 8192
        assert s == 8 or probes > 1536 * -(-cells >> (s + 1))   # no smaller than asked for
