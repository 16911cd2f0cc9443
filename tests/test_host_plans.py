"""Host code of the plans, compiled by itself and run on the CPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1902_08933_gb300", "csrc")


def run_cpp(tmp_path, code):
    """Compiles code (C++, the headers of csrc/) and runs it; its output."""
    from paper_1902_08933_gb300 import build
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(code)
    r = subprocess.run([cxx, "-std=c++17", "-O2", "-Wall", "-Werror", "-I", CSRC, "-isystem", cuda, str(src), "-o",
                        str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
    return r.stdout


def test_persistent_monitor_buffers_come_all_or_not_at_all(tmp_path):
    run_cpp(tmp_path, r"""
#include <cstdint>
#include <cstdlib>
#include "lbm_monbuf.h"
using lbm::kMonQ;
using lbm::kMonSub;
int main() {
    for (size_t steps : {1, 64}) for (size_t items : {1, 7, 456}) for (size_t n : {1, 3}) {
        lbm::MultiMonitor m;
        int calls = 0;
        if (m.allocate(steps, items, n, [&](void**, size_t) { ++calls; return false; })) return 1;
        if (calls != 1 || m.slots || m.sub || m.count) return 2;
        size_t bytes = 0;
        void* base = nullptr;
        if (!m.allocate(steps, items, n, [&](void** p, size_t b) { bytes = b; base = *p = std::malloc(b); return true; })) return 3;
        const char *b0 = (char*)base, *s = (char*)m.slots, *u = (char*)m.sub, *c = (char*)m.count;
        const size_t ns = steps * items * kMonQ * 8, nu = steps * n * kMonSub * kMonQ * 8, nc = steps * n * (kMonSub + 1) * 4;
        if (s != b0 || u < s + ns || c < u + nu || c + nc > b0 + bytes) return 4;
        if ((uintptr_t)u % 8 || (uintptr_t)c % 4) return 5;
        // a second attempt that fails leaves nothing of the first
        std::free(base);
        if (m.allocate(steps, items, n, [](void**, size_t) { return false; }) || m.slots || m.sub || m.count) return 6;
    }
    return 0;
}
""")
