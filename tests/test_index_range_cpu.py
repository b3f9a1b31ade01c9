"""The walk over a row's particles at the largest particle number that a context takes, compiled for the host."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = """
#include <cstdio>
#include <cstdlib>
#include "pm_rows.cuh"
int main(int, char **v)
{
    const int n = atoi(v[1]);
    long groups = 0, last = -32, bad = 0;
    pm::for_groups(n, [&](int c) {
        bad += c != last + 32 || c >= n;
        last = c;
        if (++groups > (1l << 26)) { printf("endless"); exit(1); }
    });
    printf("%ld %ld %ld", groups, last, bad);
}
"""


@pytest.fixture(scope="module")
def walk(tmp_path_factory):
    d = tmp_path_factory.mktemp("walk")
    (d / "t.cpp").write_text(SRC)
    exe = str(d / "t")
    subprocess.check_call(["g++", "-O1", "-std=c++20", "-I", os.path.join(ROOT, "paper_2607_17929_gb300", "csrc"),
                           str(d / "t.cpp"), "-o", exe])
    return lambda n: subprocess.run([exe, str(n)], capture_output=True, text=True, timeout=60).stdout


@pytest.mark.parametrize("n", [0, 1, 31, 32, 33, 2 ** 31 - 33, 2 ** 31 - 32, 2 ** 31 - 31, 2 ** 31 - 1])
def test_groups_of_a_row(walk, n):
    """Every group once, the last one below n, and an end: the particle numbers c .. c + 31 fit an int."""
    groups = (n + 31) // 32
    assert walk(n) == f"{groups} {32 * (groups - 1)} 0"
    assert n == 0 or 32 * (groups - 1) + 31 < 2 ** 31


def test_offsets_of_a_mass_tile_fit_their_type(tmp_path):
    """Where the mass deposit counts a tile's particles in 32 bits, the count and the end of its last chunk fit."""
    (tmp_path / "m.cpp").write_text("""
#include <cstdio>
#include <cstdlib>
#include "pm_rows.cuh"
int main(int, char **v) { printf("%d %d", (int)pm::mass_wide(atoi(v[1]), atoll(v[2])), pm::MCAP); }
""")
    exe = str(tmp_path / "m")
    subprocess.check_call(["g++", "-std=c++20", "-I", os.path.join(ROOT, "paper_2607_17929_gb300", "csrc"),
                           str(tmp_path / "m.cpp"), "-o", exe])
    for n in (8, 16, 24, 128, 1024):
        for np_ in (1, 512, 2 ** 27, 2 ** 28 - 200, 2 ** 28 - 1, 2 ** 28, 2 ** 31 - 2000, 2 ** 31 - 900, 2 ** 31 - 1):
            wide, cap = map(int, subprocess.check_output([exe, str(n), str(np_)], text=True).split())
            # cells x0 - 1 .. x0 + 7 along an axis: on 8 cells one of them is there twice
            most = np_ * (8 if n == 8 else 1)
            assert wide or most + cap < 2 ** 31, (n, np_)
            assert not wide or most > 2 ** 31 - 2000, (n, np_)   # only where it is needed
