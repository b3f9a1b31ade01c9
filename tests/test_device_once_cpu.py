"""Per-device set-up against a second thread that comes while the first is at it, compiled for the host."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = """
#include <chrono>
#include <cstdio>
#include <thread>
#include "pm_once.cuh"
using namespace std::chrono_literals;
int main()
{
    pm::DeviceOnce once;
    std::atomic<int> set[2] = {0, 0}, began{0}, second{-1};
    // the first thread is still in its set-up when the second comes
    std::thread a([&] { once(0, [&] { began = 1; std::this_thread::sleep_for(300ms); set[0] = 1; }); });
    while (!began) std::this_thread::yield();
    std::thread b([&] { once(0, [&] { set[0] = 1; }); second = set[0].load(); });
    b.join();
    a.join();
    int again = 0, other = 0, far = 0;
    once(0, [&] { again++; });                       // done: not again
    once(1, [&] { other++; });                       // another device: its own
    for (int i = 0; i < 2; i++) once(64, [&] { far++; });   // beyond the mask: each time, and no other device's bit
    printf("%d %d %d %d", second.load(), again, other, far);
}
"""


def test_second_thread_finds_the_set_up_done(tmp_path):
    (tmp_path / "t.cpp").write_text(SRC)
    exe = str(tmp_path / "t")
    subprocess.check_call(["g++", "-O1", "-std=c++20", "-pthread", "-I",
                           os.path.join(ROOT, "paper_2607_17929_gb300", "csrc"), str(tmp_path / "t.cpp"), "-o", exe])
    assert subprocess.check_output([exe], text=True, timeout=60) == "1 0 1 2"
