"""The kernel tables' construction when an allocation fails, whichever one: no exception
leaves it (it is called from a C entry), the caller gets NULL, or a table with fewer
threads at work, and a later call builds the same table.  Host code only."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2110_10749_gb300", "csrc")

SOURCE = r"""
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <initializer_list>
#include <new>
#include "fx.h"
static std::atomic<long> left{-1};
void *operator new(std::size_t n) {
    if (left >= 0 && left-- == 0) throw std::bad_alloc();
    if (void *p = std::malloc(n ? n : 1)) return p;
    throw std::bad_alloc();
}
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, std::size_t) noexcept { std::free(p); }
int main(int, char **argv) {
    left = std::atol(argv[1]);
    const ssd::FxI4 *t = ssd::fx_table_host();
    const bool first = t != nullptr;
    left = -1;
    if (!t) t = ssd::fx_table_host();
    if (!t) return 1;
    unsigned long long h = 1469598103934665603ull;
    for (int i = 0; i < ssd::kFxTabEntries * ssd::kFxEntry; ++i)
        for (int v : {t[i].x, t[i].y, t[i].z, t[i].w}) h = (h ^ (unsigned)v) * 1099511628211ull;
    std::printf("%d %llx\n", first ? 1 : 0, h);
    return 0;
}
"""


def test_failing_allocations(tmp_path):
    cc = shutil.which("g++")
    if not cc:
        pytest.skip("no g++")
    src, exe = tmp_path / "check.cpp", tmp_path / "check"
    src.write_text(SOURCE)
    subprocess.run([cc, "-O2", "-std=c++17", "-I", CSRC, str(src), "-x", "c++", os.path.join(CSRC, "fx_table.cu"),
                    "-o", str(exe), "-lpthread"], check=True)
    out = {k: subprocess.run([str(exe), str(k)], capture_output=True, text=True, check=True).stdout.split()
           for k in (-1, *range(0, 260))}
    assert len({h for _, h in out.values()}) == 1
    assert out[-1][0] == "1" and out[0][0] == "0"
