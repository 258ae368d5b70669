"""What a launch site remembers of its kernel's occupancy (csrc/hfs_resident.h)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <cstdio>
#include "hfs_resident.h"
int main()
{
    static hfs::ResidentSlot slot;
    int asked = 0, bad = 0;
    auto get = [&](int dev, int threads, uint64_t smem, int answer, int status) {
        int ctas = -1;
        const int s = slot.get(dev, threads, smem, [&](int *n) { ++asked; *n = answer; return status; }, &ctas);
        if (s != status || (s == 0 && ctas != answer)) ++bad;
    };
    // two models with the same shared memory and other CTA sizes, in turn
    for (int i = 0; i < 10; ++i) {
        get(0, 64, 10944, 152 * 16, 0);
        get(0, 128, 10944, 152 * 8, 0);
    }
    printf("%d %d\n", asked, bad);
    // other sizes and devices; a failure is not remembered
    asked = 0;
    for (int i = 0; i < 3; ++i) {
        get(0, 512, 144 * 1024, 152, 0);
        get(1, 512, 144 * 1024, 132, 0);
        get(0, 512, 227 * 1024, 304, 0);
        get(0, 256, 0, 0, 7);
        get(70, 256, 1024, 5, 0);
    }
    printf("%d %d\n", asked, bad);
    // more keys than entries: right answers all the same
    for (int i = 0; i < 60; ++i) get(0, 32, 16 * (i % 20), 100 + i % 20, 0);
    printf("%d\n", bad);
}
"""


def test_every_size_gets_its_own_grid(tmp_path):
    src, exe = tmp_path / "slot.cpp", tmp_path / "slot"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror",
                    "-I" + os.path.join(ROOT, "paper_1007_3470_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["2", "0", str(3 + 3 + 3), "0", "0"]
