"""The set-up's host threads: an exception of any item comes back to the caller
(the C entry points turn it into an error code) instead of ending the process,
and the work is done when no thread can be had."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1707_04228_gb300", "csrc")

PROGRAM = r"""
#include <cerrno>
#include <cstdio>
#include <cstring>
#include <new>
#include <stdexcept>

#include "host_parallel.h"

#ifdef NO_THREADS
extern "C" int pthread_create(pthread_t *, const pthread_attr_t *, void *(*)(void *), void *) { return EAGAIN; }
#endif

struct Own { int code; };

int main() {
    for (int n : {0, 1, 2, 33, 1000}) {
        std::vector<int> hit(n, 0);
        gl::parallel_for(n, [&](int i) { hit[i] += 1; });
        for (int h : hit) if (h != 1) return 1;
        for (int bad = 0; bad < std::min(n, 3); ++bad) {
            try {
                gl::parallel_for(n, [&](int i) { if (i == bad) throw std::bad_alloc(); });
                return 2;
            } catch (const std::bad_alloc &) {
            }
        }
        if (n) try {
            gl::parallel_for(n, [&](int) { throw Own{-4}; });
            return 3;
        } catch (const Own &e) {
            if (e.code != -4) return 4;
        }
    }
    if (gl::in_background([] { return 7; }).get() != 7) return 5;
    auto f = gl::in_background([]() -> int { throw Own{-2}; });
    try {
        f.get();
        return 6;
    } catch (const Own &e) {
        if (e.code != -2) return 7;
    }
    return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
@pytest.mark.parametrize("flags", [[], ["-DNO_THREADS"]])
def test_exceptions_come_back(tmp_path, flags):
    src, exe = tmp_path / "p.cpp", tmp_path / "p"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", *flags, "-I", CSRC, str(src), "-o", str(exe), "-lpthread"], check=True)
    assert subprocess.run([str(exe)], timeout=60).returncode == 0
