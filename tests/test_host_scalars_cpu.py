"""The page-locked read-back memory (csrc/host_scalars.h), compiled here for
the host with an allocator that can fail."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_02135_gb300", "csrc")
MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "host_scalars.h"
int live = 0;
bool fail_next = false;
int alloc(void** p, size_t bytes) {
    if (fail_next) { *p = nullptr; return 2; }
    ++live;
    *p = std::malloc(bytes);
    return 0;
}
int release(void* p) { --live; std::free(p); return 0; }
#define CHECK(x) if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; }
int main() {
    double* p = nullptr;
    size_t n = 0;
    CHECK(lmk::grow_host_doubles<int>(&p, &n, 64, alloc, release) == 0 && p && n == 64 && live == 1);
    double* const first = p;
    p[0] = 1.0; p[63] = 2.0;
    CHECK(lmk::grow_host_doubles<int>(&p, &n, 64, alloc, release) == 0 && p == first && live == 1);
    fail_next = true;    // an allocation that fails leaves the old memory in use
    CHECK(lmk::grow_host_doubles<int>(&p, &n, 1000, alloc, release) == 2);
    CHECK(p == first && n == 64 && live == 1 && p[0] == 1.0 && p[63] == 2.0);
    fail_next = false;
    CHECK(lmk::grow_host_doubles<int>(&p, &n, 1000, alloc, release) == 0 && n == 1000 && live == 1);
    p[999] = 3.0;
    release(p);
    return live;
}
"""


def test_failed_growth_keeps_the_memory(tmp_path):
    src, exe = tmp_path / "h.cpp", tmp_path / "h"
    src.write_text(MAIN)
    subprocess.run(["g++", "-O1", "-std=c++17", "-fsanitize=address,undefined", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr

