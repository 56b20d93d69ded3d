"""How the FP64 kernel stages R (csrc/plan64.cuh, plain C++): compiled with g++ and read on the CPU.

The rows of a chunk are what its latency is spread over, so a plan holds as many of them as fit
(up to four) before it holds several chunks.
"""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0811_1081_gb300", "csrc")
OPTIN = 232448  # bytes of shared memory a CTA may ask for
STATIC = 1024   # of which the kernel's own arrays take at most this

PROBE = r"""
#include <cstdio>
#include "plan64.cuh"
using namespace gspca;
int main() {
    int rows, ldr, ldk, slice;
    long avail;
    while (std::scanf("%d %d %d %d %ld", &rows, &ldr, &ldk, &slice, &avail) == 5) {
        const Chunks64 p = plan_chunks64(rows, ldr, ldk, slice, avail);
        std::printf("%d %d %zu %zu %zu\n", p.rc, p.nbuf, p.bytes, smem64_bytes(ldr, 1, 1, ldk, slice),
                    smem64_bytes(ldr, p.nbuf, p.rc + 1, ldk, slice));
    }
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan64")
    src, exe = d / "probe.cpp", d / "probe"
    src.write_text(PROBE)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)

    def run(shapes, rows=20):
        """[(N, K, G)], the rows of a CTA -> [(rows per chunk, chunks, bytes, bytes of one row, bytes of one row more)]"""
        lines = ["%d %d %d %d %d" % (rows, (n + 1) // 2 * 2, (k + 1) // 2 * 2, (n + g - 1) // g + 1, OPTIN - STATIC)
                 for n, k, g in shapes]
        out = subprocess.run([str(exe)], input="\n".join(lines), capture_output=True, text=True, check=True).stdout
        return [tuple(int(x) for x in line.split()) for line in out.splitlines()]

    return run


def test_rows_before_overlap(plan):
    shapes = [(n, k, g) for n in [1, 2, 60, 257, 511, 1500, 2000, 2055, 2500, 3000, 3601, 4097, 5000, 5699, 5801, 7000,
                                  8191, 8192] for k in [1, 50, 700] for g in [1, 8, 152]]
    for (n, k, g), (rc, nbuf, used, one, more) in zip(shapes, plan(shapes)):
        limit = OPTIN - STATIC
        if one > limit:
            assert rc == 0, (n, k, g)
            continue
        assert rc >= 1 and used <= limit, (n, k, g)
        if rc < 4:  # nothing but the next row's room keeps it from more
            assert nbuf == 1 and more > limit, (n, k, g, rc, nbuf)


def test_every_column_count_fits(plan):
    """Up to 8192 columns with K to 300: at least one row per chunk (K a little less where one CTA owns every column)."""
    shapes = [(n, k, 152) for n in range(300, 8193, 131) for k in (2, 300)]
    assert all(p[0] >= 1 for p in plan(shapes + [(8192, 300, 152), (8192, 2, 8)]))


def test_short_rows_share_a_stage(plan):
    """Rows of up to 256 doubles are staged 32 at a time, whatever K and the grid, unless a CTA has at
    most eight; longer ones at most four."""
    shapes = [(n, k, g) for n in [1, 2, 3, 31, 60, 129, 255, 256] for k in {1, min(n, 34), n} for g in [1, 2, 152]]
    for s, (rc, nbuf, used, _, _), few in zip(shapes, plan(shapes, rows=9), plan(shapes, rows=8)):
        assert (rc, nbuf) == (32, 3) and used <= OPTIN - STATIC, s
        assert few[:2] == (4, 3), s
    assert all(p[0] == 4 for p in plan([(257, 5, 152), (258, 257, 1), (1500, 50, 152)]))
