"""The setup's loop over substructures (csrc/for_each_sub.h) when memory runs
out: a failed start of a thread is done without, a failed call comes back as an
exception, and the process goes on."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0911_5730_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <new>
#include "for_each_sub.h"

// the calling thread's allocation number `fail` fails
static thread_local long count = 0, fail = -1;
void *operator new(std::size_t n) {
    if (++count == fail) throw std::bad_alloc();
    if (void *p = std::malloc(n ? n : 1)) return p;
    throw std::bad_alloc();
}
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, std::size_t) noexcept { std::free(p); }

int main() {
    static int hits[2000];
    for (long k = 0; k < 40; ++k) {
        for (int &h : hits) h = 0;
        count = 0;
        fail = k;
        bddc::for_each_sub(2000, [&](int s) { ++hits[s]; });
        fail = -1;
        for (int h : hits) if (h != 1) return 1;
    }
    int thrown = 0;
    try {
        bddc::for_each_sub(2000, [&](int s) { if (s == 777) throw 7; });
    } catch (int e) { thrown = e; }
    return thrown == 7 ? 0 : 2;
}
"""


def test_threads_that_cannot_start(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I" + CSRC, str(src), "-o", str(exe)], check=True)
    p = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert p.returncode == 0, (p.returncode, p.stderr)
