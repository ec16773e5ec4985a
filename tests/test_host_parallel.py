"""The host threads of the field and checkpoint conversions: every element once, also where a thread cannot
be started for want of memory (operator new throws while the threads are created)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <new>
#include <vector>

#include "klb_host.h"

static std::atomic<int> left{-1};  // allocations until one fails; < 0: none fails

void *operator new(std::size_t n)
{
    if (left.load() >= 0 && left.fetch_sub(1) == 0) throw std::bad_alloc();
    if (void *p = std::malloc(n ? n : 1)) return p;
    throw std::bad_alloc();
}
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, std::size_t) noexcept { std::free(p); }

int main()
{
    for (std::size_t n : {0ul, 1ul, 5ul, 1001ul})
        for (int fail = -1; fail < 9; ++fail) {
            std::vector<std::atomic<int>> hits(n);
            left = fail;
            klb::host_parallel(n, 64ul << 20, [&](std::size_t a, std::size_t b) {
                for (std::size_t k = a; k < b; ++k) ++hits[k];
            });
            left = -1;
            for (auto &h : hits)
                if (h != 1) return std::printf("n %zu fail %d: an element %d times\n", n, fail, (int)h), 1;
        }
    return 0;
}
"""


def test_every_element_once_without_memory_for_threads(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-pthread", "-I",
                           os.path.join(ROOT, "paper_2403_15768_gb300", "csrc"), str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
