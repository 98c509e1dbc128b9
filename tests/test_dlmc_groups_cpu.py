"""The groups of outer samples of the double loop (csrc/dlmc_groups.h), compiled for the host: whole
tiles of 64 rows, no more than 65535 of them (the second dimension of a grid), no more distances
than 2^25 or one tile's, from one sample to the largest counts an int holds."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
BIG = 2 ** 31 - 1
SIZES = [(n, m) for n in (1, 63, 64, 65, 4096, 4194240, 4194241, 4194304, 4793491, 9000001, 2 ** 25, 2 ** 30, BIG - 63, BIG)
         for m in (1, 2, 3, 7, 8, 9, 64, 4096, 524288, 524289, 5000000, BIG)]


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    cc = shutil.which("g++")
    if cc is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("groups")
    src = d / "groups.cpp"
    src.write_text(PROGRAM)
    subprocess.run([cc, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1502_07873_gb300", "csrc"), str(src), "-o",
                    str(d / "groups")], check=True)
    return str(d / "groups")


PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "dlmc_groups.h"
int main(int argc, char **argv)
{
    for (int k = 1; k + 1 < argc; k += 2) {
        const int N = atoi(argv[k]), M = atoi(argv[k + 1]);
        long long calls = 0, covered = 0, bad = 0;
        oed::dlmc_for_groups(N, M, [&](int n0, int n1) {
            bad += n0 != covered || n1 <= n0 || n1 > N || n1 - n0 > oed::dlmc_group_rows(N, M);
            covered = n1;
            if (++calls > 40000000) exit(1);
        });
        printf("%d %lld %lld %lld\n", oed::dlmc_group_rows(N, M), calls, covered, bad);
    }
}
"""


def _run(exe):
    args = [str(v) for s in SIZES for v in s]
    lines = subprocess.run([exe, *args], check=True, capture_output=True, text=True, timeout=60).stdout.split("\n")
    return [tuple(map(int, l.split())) for l in lines if l]


def test_rows_of_a_group(exe):
    for (n, m), (rows, *_) in zip(SIZES, _run(exe), strict=True):
        assert 1 <= rows <= n and (rows % 64 == 0 or rows == n), (n, m, rows)
        assert (rows + 63) // 64 <= 65535, (n, m, rows)
        assert rows * m <= max(2 ** 25, 64 * m), (n, m, rows)
        assert rows == n or (rows + 64) * m > 2 ** 25 or rows == 65535 * 64, (n, m, rows)   # no smaller than need be


def test_groups_cover_the_rows_once(exe):
    for (n, m), (rows, calls, covered, bad) in zip(SIZES, _run(exe), strict=True):
        assert bad == 0 and covered == n and calls == -(-n // rows), (n, m, rows, calls, covered, bad)
