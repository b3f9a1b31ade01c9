"""The list that both the accepted mesh sizes and the compiled FFT passes come from, compiled for the host."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = """
#include <cstdio>
#include "pm_sizes.cuh"
int main()
{
    for (int n = -8; n <= 2048; n++) {
        int got = 0;
        const bool ran = pm::with_mesh_size(n, [&]<int N>() { got = N; });
        if (ran != pm::is_mesh_size(n) || got != (ran ? n : 0)) return 1;
        if (ran) printf("%d ", n);
    }
}
"""


def test_every_accepted_size_is_compiled(tmp_path):
    (tmp_path / "t.cpp").write_text(SRC)
    exe = str(tmp_path / "t")
    subprocess.check_call(["g++", "-std=c++20", "-I", os.path.join(ROOT, "paper_2607_17929_gb300", "csrc"),
                           str(tmp_path / "t.cpp"), "-o", exe])
    got = [int(v) for v in subprocess.check_output([exe], text=True).split()]
    assert got == sorted(2 ** a * 3 ** b for a in range(3, 11) for b in range(7) if 2 ** a * 3 ** b <= 1024)
