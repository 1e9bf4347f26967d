"""A thread's 32-bit flight count loses nothing beyond 2^32 flights: the walk's
own tally, compiled for the host and fed as the kernel feeds it at worst, photons
of every length between two chunks that are as large as a warp may take."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <stdio.h>
#include "tally.h"
using namespace mcx;
static Tally t;
static unsigned long long total = 0, want = 0;
static void photon(unsigned long long flights)
{
    const unsigned long long unseen = flights < LOOK_FLIGHTS ? flights : LOOK_FLIGHTS;
    want += flights;
    t.steps += (uint32_t)unseen;                 // below LOOK_FLIGHTS nothing looks
    for (unsigned long long f = unseen; f < flights; ++f) {
        total += t.due();
        ++t.steps;
    }
}
int main()
{
    static const unsigned long long len[] = {1, 64, LOOK_FLIGHTS - 1, LOOK_FLIGHTS, 1u << 20};
    for (unsigned long long n : len)
        for (int chunk = 0; chunk < 4; ++chunk) {
            total += t.due();                    // the warp takes new photons
            const unsigned most = n > LOOK_FLIGHTS ? 1024 : MAX_ITEM + 1;
            for (unsigned i = 0; i < most; ++i) photon(n);
        }
    total += t.steps;
    printf("%llu %llu\n", total, want);
    return 0;
}
"""


def test_flights_beyond_32_bits(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-O2", "-Wall", "-Werror", "-I",
                    os.path.join(ROOT, "paper_2507_23189_gb300", "csrc"), "-o", str(exe), str(src)], check=True)
    got, want = (int(v) for v in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert want > 1 << 34
    assert got == want
