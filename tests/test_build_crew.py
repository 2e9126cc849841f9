"""The build's thread crew (csrc/lc_crew.h) when memory or threads run out while it starts: its
constructor either throws std::bad_alloc or leaves a crew of fewer threads that does the work; it
never ends the process."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1804_09996_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <new>
#include "lc_crew.h"

static std::atomic<int> left{1 << 30};              // allocations until one fails

void *operator new(std::size_t n)
{
    if (left.fetch_sub(1) == 0) throw std::bad_alloc();
    if (void *p = std::malloc(n ? n : 1)) return p;
    throw std::bad_alloc();
}
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, std::size_t) noexcept { std::free(p); }

int main()
{
    int thrown = 0, ran = 0;
    for (int fail = 0; fail < 24; fail++) {
        left = fail;
        try {
            lc::Crew crew(8);
            left = 1 << 30;
            std::atomic<long> sum{0};
            for (int r = 0; r < 3; r++)
                crew.run(1000, 7, [&](int64_t a, int64_t b, int) { for (; a < b; a++) sum += a; });
            if (sum != 3 * 499500) return 2;
            ran++;
        } catch (const std::bad_alloc &) {
            thrown++;
        }
        left = 1 << 30;
    }
    std::printf("%d %d\n", ran, thrown);
    return 0;
}
"""


@pytest.mark.skipif(not shutil.which("g++"), reason="needs g++")
def test_crew_survives_failing_allocations(tmp_path):
    src, exe = tmp_path / "crew.cpp", tmp_path / "crew"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stderr
    ran, thrown = map(int, r.stdout.split())
    assert ran + thrown == 24 and ran > 0
