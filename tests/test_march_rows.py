"""The rule that cuts a 2D grid into chunks of rows (march_rows, csrc/march.cuh),
compiled here by the host compiler: every row in one chunk, no chunk below the
least height or past the grid, no long one-wave marches on grids far beyond a
wave's worth of short chunks, and one wave where that is the faster."""
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    src = open(os.path.join(ROOT, "paper_2510_11042_gb300", "csrc", "march.cuh")).read()
    least = re.search(r"constexpr int kMarchMinRows = (\d+);",
                      open(os.path.join(ROOT, "paper_2510_11042_gb300", "csrc", "lbem_internal.cuh")).read())
    rule = re.search(r"^constexpr double kSlowest.*?^}\n", src, re.M | re.S)
    d = tmp_path_factory.mktemp("rows")
    (d / "rows.cpp").write_text("#include <algorithm>\n#include <cstdio>\n" + least.group(0) + "\n" + rule.group(0) +
                                "int main() { int ny, s; long long c;\n"
                                "while (scanf(\"%d %d %lld\", &ny, &s, &c) == 3) printf(\"%d\\n\", march_rows(ny, s, c)); }\n")
    subprocess.run(["g++", "-O1", "-std=c++17", str(d / "rows.cpp"), "-o", str(d / "rows")], check=True)

    def call(cases):
        out = subprocess.run([str(d / "rows")], input="\n".join("%d %d %d" % c for c in cases), text=True,
                             capture_output=True, check=True).stdout
        return [int(v) for v in out.split()]
    return call


def test_chunks_cover_the_grid(rows):
    cases = [(ny, s, cap) for ny in (2, 3, 4, 5, 17, 333, 1024, 4097, 100003) for s in (1, 2, 19, 74, 600, 40000)
             for cap in (1, 38, 152, 304)]
    for (ny, _, _), r in zip(cases, rows(cases)):
        assert 4 <= r and (r == 4 or r <= ny)


@pytest.mark.parametrize("n", [2048, 2800, 4096])
def test_no_single_wave_of_long_chunks(rows, n):
    assert rows([(n, -(-n // 56), 152)])[0] <= n // 4


@pytest.mark.parametrize("n,least", [(520, 35), (1000, 125), (1024, 128)])
def test_one_wave_where_it_is_faster(rows, n, least):
    assert rows([(n, -(-n // 56), 152)])[0] == least
